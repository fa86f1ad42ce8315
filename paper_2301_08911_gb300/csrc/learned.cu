// Learned warm start: a periodic 3x3x3 convolution network that maps the filtered
// density of a cell to the 18 displacement planes of its 6 load cases (not part of the
// paper's method, which warm-starts from the previous iterate, Sec. 3.3).
//
// The layers' forward and backward-data convolutions run on the tcgen05 tensor cores
// (conv_tc.cu). This file holds the rest of the network's arithmetic: the weight gradient,
// which contracts over voxels (BF16 mma.sync, FP32 accumulation, all 27 taps of a chunk of
// voxels in one cluster; a second kernel sums the chunks in a fixed order, so it is
// deterministic), the input
// features, pooling, the MSE loss and its gradient, Adam, and the BF16 weight packing.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <string>
#include <vector>

#include "dev_common.cuh"

namespace homo {
namespace {

constexpr int kC = HOMO_NN_CHANNELS;    // output channels of every layer (32)
constexpr int kTaps = 27;


__device__ __forceinline__ uint32_t pack2(float a, float b) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);   // a -> low half
  uint32_t u;
  memcpy(&u, &h, 4);
  return u;
}

// D = A B + D, A 16x16 row-major, B 16x8 column-major, BF16 in, FP32 accumulate.
__device__ __forceinline__ void mma16816(float* d, const uint32_t* a, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ int wrapc(int a, int n) {
  a %= n;
  return a < 0 ? a + n : a;
}

// ---- weight gradient: dw[t][o][i] = sum_v dy[v, o] x[wrap(v + d_t), i], a contraction over voxels
// with M = N = 32 per tap, too small for a 128-row tcgen05 tile: mma.sync m16n8k16 on 16
// consecutive voxels per step. Training follows the last bits of the gradients (Adam divides
// by their size and the weights are rounded to BF16), so the sums keep one fixed order: a
// chunk's tiles of 128 voxels in order, the four 32-voxel quarters of the tiles as four FP32
// chains, ((q0 + q1) + q2) + q3, then the chunks.
// A cluster of four CTAs takes a chunk, CTA q its quarters, all 27 taps at once: MMA warp w < 14
// owns taps 2 w and 2 w + 1 in 64 accumulators (so that 16 warps of 128 registers fill an SM),
// one pair of dy fragments feeding 16 MMAs. Two warps stage a quarter's dy and, per (dy, dz), its
// 32 shifted voxels plus the at most 4 row neighbours outside the run by 16-byte asynchronous
// copies, kWgStages quarters deep, voxel-major as they lie in memory; ldmatrix.trans turns 8 x 8
// blocks on the way to the registers, its per-lane row addresses resolving the periodic x
// neighbours. 16-byte chunk c of slot v sits at chunk c ^ (v / 2 % 4) of its row, so that
// 8 consecutive slots' chunks fall on distinct banks. The quarters' chains meet through
// distributed shared memory. Extra clusters in front sum dy for the bias, a chunk per warp,
// voxel by voxel.
// 64^3, 32 channels: 124 us (a CTA per tap and chunk staged dy and x again for every tap,
// transposing through 2-byte shared-memory stores: 225 us, LSU 86 % busy; nine MMA warps
// of three taps that also copied: 171 us, most of it copy instructions and their latency).
constexpr int kWgTile = 128, kWgRun = 32, kWgCtas = 4;     // voxels of a tile, of a quarter; quarters
constexpr int kWgSlots = kWgRun + 4;
constexpr int kWgMma = 14, kWgWarps = 16, kWgThreads = 32 * kWgWarps, kWgCopy = kWgThreads - 32 * kWgMma;
constexpr int kWgBias = kWgCtas * kWgWarps;                // chunks of a bias cluster
constexpr int kWgStages = 4;

template <int CIN>
struct WgSmem {
  static constexpr int kDy = kWgRun * kC * 2, kX = 9 * kWgSlots * CIN * 2;
  static constexpr int kStage = kDy + kX;
  static constexpr int kSum = kTaps * kC * CIN * 4;        // the chain sums, in place of the stages
  static constexpr int kBytes = kWgStages * kStage > kSum ? kWgStages * kStage : kSum;
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// 16 bytes, or zeros where live is false (src is then any valid address)
__device__ __forceinline__ void cp_async16z(uint32_t dst, const void* src, bool live) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(live ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int kLeft>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(kLeft) : "memory");
}

__device__ __forceinline__ void ldmatrix_x4_t(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}

// Byte offset of 16-byte chunk c of slot v (kCh chunks per slot: 4, or 2 for 16 channels, where
// the swizzle period doubles).
template <int kCh>
__device__ __forceinline__ uint32_t wg_at(int v, int c) {
  return static_cast<uint32_t>((v * kCh + (c ^ (kCh == 4 ? (v >> 1) & 3 : (v >> 2) & 1))) * 16);
}

// Stage the run of voxels u0 .. u0 + 31 (those below N): dy, and for each (dy, dz) the shifted
// voxels in slots 0..31 and the x neighbours that lie in a partly covered row: slot 32 left of
// the first voxel, 33 x = 0 of its row, 34 x = n - 1 of the last voxel's row, 35 right of it.
template <int CIN>
__device__ __forceinline__ void wg_stage(size_t u0, size_t N, int n, const __nv_bfloat16* __restrict__ x,
                                         const __nv_bfloat16* __restrict__ dy, uint32_t s_dy, uint32_t s_x) {
  constexpr int kCh = CIN / 8, kPerPass = kWgCopy / kCh;     // slots per pass of the copy warps
  const int t = threadIdx.x - 32 * kWgMma;
  const int count = u0 >= N ? 0 : static_cast<int>(N - u0 < kWgRun ? N - u0 : kWgRun);
  if (count > 0) {
#pragma unroll
    for (int k = 0; k < kWgRun * (kC / 8) / kWgCopy; ++k) {
      const int c = t % (kC / 8), i = t / (kC / 8) + k * (kWgCopy / (kC / 8));
      cp_async16z(s_dy + wg_at<kC / 8>(i, c), dy + (u0 + (i < count ? i : 0)) * kC + c * 8, i < count);
    }
#pragma unroll 1
    for (int slot = t / kCh; slot < kWgSlots; slot += kPerPass) {
      const int c = t % kCh;
      const int i = slot < kWgRun ? slot : (slot < kWgRun + 2 ? 0 : count - 1);   // the voxel whose row it is in
      const bool live = i < count;
      int gx, gy, gz;
      decode3(static_cast<unsigned>(u0) + (live ? i : 0), static_cast<unsigned>(n), gx, gy, gz);
      if (slot == kWgRun) gx = gx == 0 ? n - 1 : gx - 1;
      if (slot == kWgRun + 1) gx = 0;
      if (slot == kWgRun + 2) gx = n - 1;
      if (slot == kWgRun + 3) gx = gx == n - 1 ? 0 : gx + 1;
      const Nb nb = make_nb(gx, gy, gz, n);   // the nine (dy, dz) rows share the slot's x
      const uint32_t dst = s_x + wg_at<kCh>(slot, c);
      const __nv_bfloat16* src = x + static_cast<size_t>(gx) * CIN + c * 8;
#pragma unroll
      for (int combo = 0; combo < 9; ++combo)
        cp_async16z(dst + combo * (kWgSlots * CIN * 2),
                    src + static_cast<size_t>(nb.Y[combo % 3] + nb.Z[combo / 3]) * CIN, live);
    }
  }
  cp_async_commit();
}

// Slot of the x neighbour (dx = -1, 0, 1) of voxel i of a run whose x coordinate is xi.
__device__ __forceinline__ int wg_slot(int i, int xi, int dx, int n) {
  if (dx < 0) {
    if (xi > 0) return i > 0 ? i - 1 : kWgRun;
    return i + n - 1 < kWgRun ? i + n - 1 : kWgRun + 2;
  }
  if (dx > 0) {
    if (xi < n - 1) return i < kWgRun - 1 ? i + 1 : kWgRun + 3;
    return i >= n - 1 ? i - (n - 1) : kWgRun + 1;
  }
  return i;
}

__device__ __forceinline__ float ld_cluster_f32(uint32_t addr) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
  return v;
}

// Partial gradients: part[(chunk * 27 + tap)][o][i], partb[chunk][o]. Clusters 0 .. bias - 1 take the
// bias, the others one chunk each.
template <int CIN>
__global__ void __launch_bounds__(kWgThreads, 1)
    k_wgrad(int n, int ntiles, int tiles_per_chunk, int chunks, int bias, const __nv_bfloat16* __restrict__ x,
            const __nv_bfloat16* __restrict__ dy, float* __restrict__ part, float* __restrict__ partb) {
  using S = WgSmem<CIN>;
  constexpr int kCh = CIN / 8, NT = CIN / 8;
  extern __shared__ __align__(128) unsigned char wsm[];
  const uint32_t base = smem_u32(wsm);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int q = blockIdx.x % kWgCtas, cluster = blockIdx.x / kWgCtas;
  const size_t N = static_cast<size_t>(n) * n * n;

  if (cluster < bias) {
    // lane = output channel, every voxel of the chunk in order, 32 loads ahead of the sum
    const int chunk = cluster * kWgBias + q * kWgWarps + warp;
    if (chunk >= chunks) return;
    const size_t v0 = static_cast<size_t>(chunk) * tiles_per_chunk * kWgTile;
    const size_t v1 = min(N, v0 + static_cast<size_t>(tiles_per_chunk) * kWgTile);
    const __nv_bfloat16* d = dy + lane;
    float cur[32], nxt[32], bsum = 0.f;
#pragma unroll
    for (int j = 0; j < 32; ++j) cur[j] = v0 + j < v1 ? __bfloat162float(d[(v0 + j) * kC]) : 0.f;
    for (size_t v = v0; v < v1; v += 32) {
#pragma unroll
      for (int j = 0; j < 32; ++j) nxt[j] = v + 32 + j < v1 ? __bfloat162float(d[(v + 32 + j) * kC]) : 0.f;
#pragma unroll
      for (int j = 0; j < 32; ++j) {
        bsum += cur[j];
        cur[j] = nxt[j];
      }
    }
    partb[static_cast<size_t>(chunk) * kC + lane] = bsum;
    return;
  }
  const int chunk = cluster - bias;
  const int t0 = chunk * tiles_per_chunk, t1 = min(ntiles, t0 + tiles_per_chunk);
  auto run_of = [&](int tile) { return static_cast<size_t>(tile) * kWgTile + kWgRun * q; };
  auto stage_at = [&](int k) { return base + static_cast<uint32_t>(k % kWgStages) * S::kStage; };

  if (warp >= kWgMma) {
    // ---- copies: stage k is in flight while stages before it are consumed
#pragma unroll 1
    for (int k = 0; k < kWgStages - 1; ++k) {
      if (t0 + k < t1) wg_stage<CIN>(run_of(t0 + k), N, n, x, dy, stage_at(k), stage_at(k) + S::kDy);
      else cp_async_commit();
    }
    for (int tile = t0; tile < t1; ++tile) {
      const int k = tile - t0 + kWgStages - 1;
      cp_async_wait<kWgStages - 2>();
      __syncthreads();   // this stage is complete, the one before it consumed
      if (t0 + k < t1) wg_stage<CIN>(run_of(t0 + k), N, n, x, dy, stage_at(k), stage_at(k) + S::kDy);
      else cp_async_commit();
    }
    cp_async_wait<0>();
    __syncthreads();
  } else {
    // ldmatrix lanes: lanes 0-7, 8-15, 16-23, 24-31 give the row addresses of matrices 0..3.
    // A (dy^T): matrices (v 0-7, o chunk 0), (v 0-7, chunk 1), (v 8-15, chunk 0), (v 8-15, chunk 1)
    const int av = (lane & 7) + ((lane >> 4) << 3), ac = (lane >> 3) & 1;
    // B (x): (v 0-7, i chunk 0), (v 8-15, chunk 0), (v 0-7, chunk 1), (v 8-15, chunk 1)
    const int bv = (lane & 7) + (((lane >> 3) & 1) << 3), bc = lane >> 4;
    float acc[2][2][NT][4];
#pragma unroll
    for (int t = 0; t < 2; ++t)
#pragma unroll
      for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
          for (int e = 0; e < 4; ++e) acc[t][mt][nt][e] = 0.f;
    for (int tile = t0; tile < t1; ++tile) {
      __syncthreads();
      const size_t u0 = run_of(tile);
      const uint32_t s_dy = stage_at(tile - t0), s_x = s_dy + S::kDy;
#pragma unroll
      for (int ks = 0; ks < 2; ++ks) {
        if (u0 + 16 * ks >= N) continue;   // past the grid: the products are zero
        uint32_t a[2][4];
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) ldmatrix_x4_t(a[mt], s_dy + wg_at<kC / 8>(16 * ks + av, 2 * mt + ac));
        const int i = 16 * ks + bv;
        const int xi = static_cast<int>((static_cast<unsigned>(u0) + i) % static_cast<unsigned>(n));
#pragma unroll
        for (int t = 0; t < 2; ++t) {
          const int tap = 2 * warp + t;
          if (tap >= kTaps) break;
          const int slot = u0 + i < N ? wg_slot(i, xi, tap % 3 - 1, n) : i;
          const uint32_t s_row = s_x + (tap / 3) * (kWgSlots * CIN * 2);
#pragma unroll
          for (int h = 0; h < NT / 2; ++h) {
            uint32_t b[4];
            ldmatrix_x4_t(b, s_row + wg_at<kCh>(slot, 2 * h + bc));
#pragma unroll
            for (int mt = 0; mt < 2; ++mt) {
              mma16816(acc[t][mt][2 * h], a[mt], b[0], b[1]);
              mma16816(acc[t][mt][2 * h + 1], a[mt], b[2], b[3]);
            }
          }
        }
      }
    }
    __syncthreads();   // the stages give way to the chain sums
    float* sum = reinterpret_cast<float*>(wsm);
    const int g = lane >> 2, t4 = lane & 3;
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      if (2 * warp + t >= kTaps) break;
#pragma unroll
      for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
          float* d = sum + (2 * warp + t) * (kC * CIN) + (16 * mt + g) * CIN + 8 * nt + 2 * t4;
          d[0] = acc[t][mt][nt][0];
          d[1] = acc[t][mt][nt][1];
          d[8 * CIN] = acc[t][mt][nt][2];
          d[8 * CIN + 1] = acc[t][mt][nt][3];
        }
    }
  }
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
  // each CTA adds a quarter of the values over the four chains
  constexpr int kPer = kTaps * kC * CIN / kWgCtas;
  uint32_t peer[kWgCtas];
#pragma unroll
  for (int r = 0; r < kWgCtas; ++r)
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(peer[r]) : "r"(base), "r"(r));
  float* dst = part + static_cast<size_t>(chunk) * kTaps * kC * CIN;
#pragma unroll 4
  for (int e = q * kPer + threadIdx.x; e < (q + 1) * kPer; e += kWgThreads) {
    float v[kWgCtas];
#pragma unroll
    for (int r = 0; r < kWgCtas; ++r) v[r] = ld_cluster_f32(peer[r] + 4u * e);
    dst[e] = __fadd_rn(__fadd_rn(__fadd_rn(v[0], v[1]), v[2]), v[3]);
  }
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");   // peers read this CTA's sums
}

// dw[t][o][i] = sum over chunks of the partials, db[o] likewise: four threads per value sum a
// quarter each in order as FP32 pairs (TwoSum), then the quarters. What is left of the error is the
// rounding of the low parts' own FP32 sum, far below half a unit of the FP32 result. (A one-thread
// FP64 sum kept the FP64 pipe 71 % busy: 38 -> 12 us for 27,680 values.) A pair has the range of
// FP32: where a sum is not finite, by an infinite partial or because its high part left that range
// on the way, the value is summed again in FP64.
__global__ void __launch_bounds__(256) k_wgrad_reduce(int chunks, int per, const float* __restrict__ part,
                                                      const float* __restrict__ partb, float* __restrict__ dw,
                                                      float* __restrict__ db) {
  __shared__ float sh[4][64], sl[4][64];
  const int q = threadIdx.x >> 6, k = threadIdx.x & 63;
  const int e = blockIdx.x * 64 + k;
  const int nw = kTaps * per;
  const int c0 = chunks * q / 4, c1 = chunks * (q + 1) / 4;
  float hi = 0.f, lo = 0.f;
  auto add = [&](float v) {
    const float s = __fadd_rn(hi, v), bb = __fadd_rn(s, -hi);
    lo = __fadd_rn(lo, __fadd_rn(__fadd_rn(hi, -__fadd_rn(s, -bb)), __fadd_rn(v, -bb)));
    hi = s;
  };
  if (e < nw + kC) {
    const float* src = e < nw ? part + e : partb + (e - nw);
    const size_t step = e < nw ? nw : kC;
#pragma unroll 8
    for (int c = c0; c < c1; ++c) add(__ldg(src + c * step));
  }
  sh[q][k] = hi;
  sl[q][k] = lo;
  __syncthreads();
  if (q != 0 || e >= nw + kC) return;
  for (int t = 1; t < 4; ++t) {
    add(sh[t][k]);
    lo = __fadd_rn(lo, sl[t][k]);
  }
  const float sum = __fadd_rn(hi, lo);
  (e < nw ? dw[e] : db[e - nw]) = sum;
  if (isfinite(sum)) return;
  // after the store and with its own addresses: written as a choice before the store it shared
  // the main loop's, which then ran 8 us longer
  double d = 0.0;
#pragma unroll 1
  for (int c = 0; c < chunks; ++c)
    d += e < nw ? part[static_cast<size_t>(c) * nw + e] : partb[static_cast<size_t>(c) * kC + e - nw];
  (e < nw ? dw[e] : db[e - nw]) = static_cast<float>(d);
}

// x[v] = (rho, rho^2, rho^3, 0 ... 0) in BF16, 16 channels.
__global__ void k_features(size_t N, const float* __restrict__ rho, __nv_bfloat16* __restrict__ x) {
  for (size_t v = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; v < N;
       v += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const float r = rho[v];
    uint4 lo, hi;
    lo.x = pack2(r, r * r);
    lo.y = pack2(r * r * r, 0.f);
    lo.z = lo.w = 0u;
    hi.x = hi.y = hi.z = hi.w = 0u;
    uint4* d = reinterpret_cast<uint4*>(x + v * HOMO_NN_FEATURES);
    d[0] = lo;
    d[1] = hi;
  }
}

// Loss sum_{v,p<18} (y[p][v] - u[p][v] inv[p/3])^2 / (18 N) per block (FP64) and the
// BF16 gradient dy[v][p] = 2 (y - u inv) / (18 N), zero in channels 18..31.
struct CaseInv {
  double inv[6];
};

__global__ void __launch_bounds__(256) k_mse(size_t N, const float* __restrict__ y, const float* __restrict__ u,
                                             CaseInv ci, __nv_bfloat16* __restrict__ dy, double* __restrict__ part) {
  __shared__ double sh[256];
  const double w = 2.0 / (18.0 * static_cast<double>(N));
  double s = 0.0;
  for (size_t v = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; v < N;
       v += static_cast<size_t>(gridDim.x) * blockDim.x) {
    uint32_t pk[16];
#pragma unroll
    for (int p = 0; p < 18; p += 2) {
      const double e0 = static_cast<double>(y[p * N + v]) - static_cast<double>(u[p * N + v]) * ci.inv[p / 3];
      const double e1 =
          static_cast<double>(y[(p + 1) * N + v]) - static_cast<double>(u[(p + 1) * N + v]) * ci.inv[(p + 1) / 3];
      s += e0 * e0 + e1 * e1;
      pk[p / 2] = pack2(static_cast<float>(w * e0), static_cast<float>(w * e1));
    }
#pragma unroll
    for (int q = 9; q < 16; ++q) pk[q] = 0u;
    uint4* d = reinterpret_cast<uint4*>(dy + v * kC);
#pragma unroll
    for (int q = 0; q < 4; ++q) d[q] = make_uint4(pk[4 * q], pk[4 * q + 1], pk[4 * q + 2], pk[4 * q + 3]);
  }
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = sh[0] / (18.0 * static_cast<double>(N));
}

// out[c] = mean of rho over the f^3 fine voxels of coarse voxel c (grid n -> n / f).
__global__ void k_pool(int n, int f, const float* __restrict__ rho, float* __restrict__ out) {
  const int nc = n / f;
  const size_t Nc = static_cast<size_t>(nc) * nc * nc;
  for (size_t c = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; c < Nc;
       c += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const int i = static_cast<int>(c % nc), j = static_cast<int>((c / nc) % nc),
              k = static_cast<int>(c / (static_cast<size_t>(nc) * nc));
    double s = 0.0;
    for (int dz = 0; dz < f; ++dz)
      for (int dy = 0; dy < f; ++dy) {
        const float* row = rho + static_cast<size_t>(i) * f +
                           static_cast<size_t>(n) * (static_cast<size_t>(j) * f + dy + static_cast<size_t>(n) * (static_cast<size_t>(k) * f + dz));
        for (int dx = 0; dx < f; ++dx) s += row[dx];
      }
    out[c] = static_cast<float>(s / (static_cast<double>(f) * f * f));
  }
}

__global__ void k_adam(size_t count, float* __restrict__ w, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, float lr, float b1, float b2, float c1, float c2, float eps) {
  for (size_t i = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; i < count;
       i += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    w[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

// wf[t][o][i] = bf16(w[t][o][i]); wb[t][i][o] = bf16(w[26 - t][o][i]) (weights of the
// transposed convolution that propagates gradients back, when c_in = 32).
__global__ void k_pack(int cin, const float* __restrict__ w, __nv_bfloat16* __restrict__ wf,
                       __nv_bfloat16* __restrict__ wb) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= kTaps * kC * cin) return;
  const int t = e / (kC * cin), r = e - t * kC * cin, o = r / cin, i = r - o * cin;
  const __nv_bfloat16 h = __float2bfloat16_rn(w[e]);
  wf[e] = h;
  if (wb) wb[(static_cast<size_t>(kTaps - 1 - t) * cin + i) * kC + o] = h;
}

int g_num_sms = 0;

int num_sms() {
  if (g_num_sms == 0) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&g_num_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || g_num_sms < 1)
      g_num_sms = 152;
  }
  return g_num_sms;
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

struct WgradPlan {
  int ntiles, tiles_per_chunk, chunks;
};

WgradPlan wgrad_plan(int n) {
  const size_t N = static_cast<size_t>(n) * n * n;
  WgradPlan p;
  p.ntiles = static_cast<int>((N + kWgTile - 1) / kWgTile);
  const int want = std::max(1, std::min(p.ntiles, 4 * num_sms() / 3));
  p.tiles_per_chunk = (p.ntiles + want - 1) / want;
  p.chunks = (p.ntiles + p.tiles_per_chunk - 1) / p.tiles_per_chunk;
  return p;
}

size_t wgrad_scratch_floats(int n, int cin) {
  const WgradPlan p = wgrad_plan(n);
  return static_cast<size_t>(p.chunks) * (static_cast<size_t>(kTaps) * kC * cin + kC);
}

}  // namespace

// ---- launchers --------------------------------------------------------------------------
cudaError_t nn_conv3d(int n, int cin, const void* x, const void* w, const float* bias, const void* res,
                      const void* mask, int epi, void* out, float* outf, const double* scale, cudaStream_t s) {
  return conv3d_tc(n, cin, epi, x, w, bias, res, mask, out, outf, scale, s);
}

namespace {
template <int CIN>
cudaError_t wgrad_launch(const WgradPlan& p, int n, const void* x, const void* dy, float* part, float* partb,
                         cudaStream_t s) {
  constexpr int shm = WgSmem<CIN>::kBytes;
  const cudaError_t e = cudaFuncSetAttribute(k_wgrad<CIN>, cudaFuncAttributeMaxDynamicSharedMemorySize, shm);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  const int bias = (p.chunks + kWgBias - 1) / kWgBias;
  cfg.gridDim = dim3((bias + p.chunks) * kWgCtas);
  cfg.blockDim = dim3(kWgThreads);
  cfg.dynamicSmemBytes = shm;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kWgCtas;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_wgrad<CIN>, n, p.ntiles, p.tiles_per_chunk, p.chunks, bias,
                            static_cast<const __nv_bfloat16*>(x),
                            static_cast<const __nv_bfloat16*>(dy), part, partb);
}
}  // namespace

cudaError_t nn_wgrad(int n, int cin, const void* x, const void* dy, float* dw, float* db, float* scratch,
                     cudaStream_t s) {
  const WgradPlan p = wgrad_plan(n);
  float* part = scratch;
  float* partb = scratch + static_cast<size_t>(p.chunks) * kTaps * kC * cin;
  if (cin != 16 && cin != 32) return cudaErrorInvalidValue;
  const cudaError_t e = cin == 16 ? wgrad_launch<16>(p, n, x, dy, part, partb, s)
                                  : wgrad_launch<32>(p, n, x, dy, part, partb, s);
  if (e != cudaSuccess) return e;
  const int total = kTaps * kC * cin + kC;
  k_wgrad_reduce<<<(total + 63) / 64, 256, 0, s>>>(p.chunks, kC * cin, part, partb, dw, db);
  return cudaGetLastError();
}

cudaError_t nn_features(int n, const float* rho, void* x, cudaStream_t s) {
  const size_t N = static_cast<size_t>(n) * n * n;
  k_features<<<grid_for(N, 256), 256, 0, s>>>(N, rho, static_cast<__nv_bfloat16*>(x));
  return cudaGetLastError();
}

cudaError_t nn_mse(int n, const float* y, const float* u, const double* scale, void* dy, double* part, int* nblk,
                   cudaStream_t s) {
  CaseInv ci;
  for (int k = 0; k < 6; ++k) ci.inv[k] = 1.0 / scale[k];
  const size_t N = static_cast<size_t>(n) * n * n;
  const int g = std::min(grid_for(N, 256), HOMO_NN_MSE_SCRATCH - 1);
  *nblk = g;
  k_mse<<<g, 256, 0, s>>>(N, y, u, ci, static_cast<__nv_bfloat16*>(dy), part);
  return cudaGetLastError();
}

cudaError_t nn_pool(int n, int f, const float* rho, float* out, cudaStream_t s) {
  const int nc = n / f;
  k_pool<<<grid_for(static_cast<size_t>(nc) * nc * nc, 256), 256, 0, s>>>(n, f, rho, out);
  return cudaGetLastError();
}

cudaError_t nn_adam(size_t count, float* w, const float* g, float* m, float* v, int step, double lr, double b1,
                    double b2, double eps, cudaStream_t s) {
  const double c1 = 1.0 - std::pow(b1, step), c2 = 1.0 - std::pow(b2, step);
  k_adam<<<grid_for(count, 256), 256, 0, s>>>(count, w, g, m, v, static_cast<float>(lr), static_cast<float>(b1),
                                              static_cast<float>(b2), static_cast<float>(c1), static_cast<float>(c2),
                                              static_cast<float>(eps));
  return cudaGetLastError();
}

cudaError_t nn_pack(int cin, const float* w, void* wf, void* wb, cudaStream_t s) {
  const int total = kTaps * kC * cin;
  k_pack<<<(total + 255) / 256, 256, 0, s>>>(cin, w, static_cast<__nv_bfloat16*>(wf),
                                             static_cast<__nv_bfloat16*>(wb));
  return cudaGetLastError();
}

}  // namespace homo

// ---- C ABI ------------------------------------------------------------------------------
using namespace homo;

namespace {

int cuda_status(cudaError_t e) { return e == cudaSuccess ? HOMO_OK : HOMO_ECUDA; }

bool conv_args_ok(int n, int c_in, const void* x, const void* w, const void* res, const void* mask, int epi,
                  const void* out, const float* outf) {
  if (n < 1 || n > 1024 || !x || !w || !aligned16(x) || !aligned16(w)) return false;
  if (res && (reinterpret_cast<uintptr_t>(res) & 3u)) return false;
  switch (epi) {
    case HOMO_NN_RELU:
      return (c_in == 16 || c_in == 32) && out && !mask && !outf && !(reinterpret_cast<uintptr_t>(out) & 3u);
    case HOMO_NN_MASK:
      return c_in == 32 && out && mask && !outf && !(reinterpret_cast<uintptr_t>(out) & 3u) &&
             !(reinterpret_cast<uintptr_t>(mask) & 3u);
    case HOMO_NN_PLANES:
    case HOMO_NN_PLANES_ADD:
      return c_in == 32 && outf && !out && !res && !mask;
    default:
      return false;
  }
}

}  // namespace

extern "C" {

int homo_nn_tc_timeouts(void) { return conv3d_tc_take_timeouts(); }

int homo_nn_tc_wait_probe(int blocks) {
  if (blocks < 1 || blocks > 1024) return HOMO_EINVAL;
  return cuda_status(conv3d_tc_wait_probe(blocks));
}

int homo_nn_conv3d(int n, int c_in, const void* x, const void* w, const float* bias, const void* res,
                   const void* mask, int epilogue, void* out, float* out_planes, const double* scale,
                   void* stream) {
  if (!conv_args_ok(n, c_in, x, w, res, mask, epilogue, out, out_planes)) return HOMO_EINVAL;
  return cuda_status(nn_conv3d(n, c_in, x, w, bias, res, mask, epilogue, out, out_planes, scale,
                               static_cast<cudaStream_t>(stream)));
}

size_t homo_nn_wgrad_scratch(int n, int c_in) {
  if (n < 1 || n > 1024 || (c_in != 16 && c_in != 32)) return 0;
  return wgrad_scratch_floats(n, c_in);
}

int homo_nn_wgrad(int n, int c_in, const void* x, const void* dy, float* dw, float* db, float* scratch,
                  size_t scratch_floats, void* stream) {
  if (n < 1 || n > 1024 || (c_in != 16 && c_in != 32) || !x || !dy || !dw || !db || !scratch) return HOMO_EINVAL;
  if (!aligned16(x) || !aligned16(dy) || scratch_floats < wgrad_scratch_floats(n, c_in)) return HOMO_EINVAL;
  return cuda_status(nn_wgrad(n, c_in, x, dy, dw, db, scratch, static_cast<cudaStream_t>(stream)));
}

int homo_nn_features(int n, const float* rho, void* x, void* stream) {
  if (n < 1 || n > 1024 || !rho || !x || !aligned16(x)) return HOMO_EINVAL;
  return cuda_status(nn_features(n, rho, x, static_cast<cudaStream_t>(stream)));
}

int homo_nn_pool(int n, int factor, const float* rho, float* out, void* stream) {
  if (n < 1 || n > 1024 || factor < 1 || n % factor != 0 || !rho || !out) return HOMO_EINVAL;
  return cuda_status(nn_pool(n, factor, rho, out, static_cast<cudaStream_t>(stream)));
}

static bool scales_ok(const double* scale) {
  if (!scale) return false;
  for (int k = 0; k < 6; ++k)
    if (!(scale[k] > 0.0) || !std::isfinite(scale[k])) return false;
  return true;
}

int homo_nn_mse(int n, const float* y, const float* u, const double* scale, void* dy, double* loss, void* stream) {
  if (n < 1 || n > 1024 || !y || !u || !dy || !loss || !aligned16(dy) || !scales_ok(scale)) return HOMO_EINVAL;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int nblk = 0;
  cudaError_t e = nn_mse(n, y, u, scale, dy, loss + 1, &nblk, s);
  if (e == cudaSuccess) e = launch_sum_partials(loss + 1, nblk, 1, loss, s);
  return cuda_status(e);
}

int homo_nn_adam(size_t count, float* w, const float* g, float* m, float* v, int step, double lr, double beta1,
                 double beta2, double eps, void* stream) {
  if (!w || !g || !m || !v || step < 1 || !(lr >= 0.0) || !(beta1 >= 0.0 && beta1 < 1.0) ||
      !(beta2 >= 0.0 && beta2 < 1.0) || !(eps > 0.0))
    return HOMO_EINVAL;
  if (count == 0) return HOMO_OK;
  return cuda_status(nn_adam(count, w, g, m, v, step, lr, beta1, beta2, eps, static_cast<cudaStream_t>(stream)));
}

int homo_nn_pack(int c_in, const float* w, void* w_fwd, void* w_bwd, void* stream) {
  if ((c_in != 16 && c_in != 32) || !w || !w_fwd || (w_bwd && c_in != 32)) return HOMO_EINVAL;
  return cuda_status(nn_pack(c_in, w, w_fwd, w_bwd, static_cast<cudaStream_t>(stream)));
}

}  // extern "C"
