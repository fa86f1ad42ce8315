// Periodic 3x3x3 convolution of the warm-start network on the 5th-generation tensor cores
// (tcgen05.mma, accumulators in tensor memory). Implicit GEMM: M = 128 voxels, N = 32
// output channels, K = 27 taps x c_in, BF16 operands, FP32 accumulation.
//
// A persistent CTA keeps the layer's weights in shared memory and walks tiles of TX x TY x TZ
// output voxels. Each tile's periodic halo box ((TX + 2) x (TY + 2) x (TZ + 2) voxels, all input
// channels) is staged with 16-byte asynchronous copies into a K-major, non-swizzled operand
// layout whose rows are 16 bytes apart along the box's (z, y, x) order: channel chunk c (8
// channels) of box row r sits at plane c, row r. The outputs of a z-plane are then consecutive
// box rows but for the two halo rows between lines, so blocks of 128 rows from the first
// output on are the M of an MMA, and for a tap the A operand is the same staged box seen
// through a descriptor shifted by the tap's constant row offset: no per-tap copy. Rows on
// halo positions are computed and discarded.
// Thirteen warps in three roles, handing tiles on through mbarriers, so that the copies of the
// next tiles, the MMAs of one and the epilogue of the one before run at the same time:
//   warps 8..11 copy boxes into a ring of buffers;
//   warp 12     issues (one elected lane) the 27 x c_in/16 MMAs of each of the tile's row blocks
//               into one of two sets of 32-column TMEM accumulators and commits them to the
//               barriers that free the box and publish the accumulators;
//   warps 0..7  (four per row block) read their 32 TMEM lanes (one voxel per thread, 32
//               channels), free the accumulators and apply the epilogue: bias, residual, ReLU or a backward ReLU
//               mask, BF16 voxel-major output or scaled FP32 displacement planes.
// Every wait is bounded. Bound: an MMA of 128 x 32 x 16 reads 5 KB of operands for 16 cycles
// of math; measured 68 cycles each, back to back (two thirds of the time on operands at 64 B a
// clock), so what counts is the share of rows that are outputs. 64^3, 32 -> 32 channels:
// 70 -> 39 us with 30 x 4 x 2 tiles (four warps did all three in turn before, two CTAs per
// SM: tensor pipe 14 % busy), 37 us with 32 x 11 x 1.
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdint>
#include <cstring>

#include "dev_common.cuh"

namespace homo {
namespace {

constexpr int kC = HOMO_NN_CHANNELS;     // 32 output channels
constexpr int kTaps = 27;
constexpr int kThreads = 13 * 32;                          // 8 epilogue, 4 copy and one MMA warp
constexpr int kEpi = 256, kRole = 128;                     // threads of the epilogue and of the copy role
constexpr long long kWaitLimit = 1LL << 18;                // bounded mbarrier polls (~1 s on a GB300)

// A tile shape and its box, row blocks and shared memory for CIN input channels.
template <int X, int Y, int Z, int kStagesOf>
struct TcTile {
  static constexpr int TX = X, TY = Y, TZ = Z, kStages = kStagesOf;   // kStages: boxes in flight
  static constexpr int BX = TX + 2, BY = TY + 2, BZ = TZ + 2;
  static constexpr int kBoxRows = BX * BY * BZ;
  static constexpr int kBlocks = (TY * BX - 2 + 127) / 128;   // row blocks per z-plane (y rows are BX apart)
  static constexpr int kUnits = TZ * kBlocks;                 // accumulators of a tile
  // rows the last block of the last plane reads for tap (1, 1, 1), a multiple of 8
  static constexpr int kLast = ((TZ + 1) * BY + 2) * BX + 2 + 128 * kBlocks;
  static constexpr int kRows = ((kLast > kBoxRows ? kLast : kBoxRows) + 7) / 8 * 8;
  static constexpr int kPlaneBytes = kRows * 16;              // one 8-channel chunk of every row
  static constexpr int kTmemUse = 2 * kUnits * kC;
  static constexpr int kTmemCols = kTmemUse <= 128 ? 128 : 256;
  static constexpr int kBarriers = 2 * kStages + 4;
  static_assert(kTmemUse <= kTmemCols, "two sets of accumulators");
};
typedef TcTile<30, 4, 2, 3> TileA;     // a line of 32 rows, 126 of 128 rows per block, 3 of 4 lines' halo
typedef TcTile<32, 11, 1, 2> TileB;    // 352 outputs of 3 x 128 rows

template <int CIN, typename TL>
struct TcShape {
  static constexpr int kChunks = CIN / 8;
  static constexpr int kBoxBytes = kChunks * TL::kPlaneBytes;
  static constexpr int kWBytes = kTaps * kChunks * kC * 16;
  static constexpr int kBytes = TL::kStages * kBoxBytes + kWBytes + 8 * TL::kBarriers + 16;   // + mbarriers, TMEM address
  static_assert(kBytes <= 227 * 1024, "shared memory of a CTA");
};

struct TcScale {
  float s[6];
};

__device__ int g_conv_tc_timeouts = 0;   // CTAs in which a wait ran out

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src) : "memory");
}

__device__ __forceinline__ int wrapc(int a, int n) {
  a %= n;
  return a < 0 ? a + n : a;
}

// the same for -n <= a < 2 n
__device__ __forceinline__ int wrap1(int a, int n) { return a < 0 ? a + n : (a >= n ? a - n : a); }

// Shared-memory matrix descriptor of a K-major, non-swizzled operand: core matrices of
// 8 rows x 16 bytes with rows 16 bytes apart, 8-row groups SBO bytes apart along M/N and
// 16-byte K chunks LBO bytes apart; descriptor version 1 (bits 46-47), no base offset.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((addr & 0x3FFFFu) >> 4);
  d |= static_cast<uint64_t>((lbo >> 4) & 0x3FFFu) << 16;
  d |= static_cast<uint64_t>((sbo >> 4) & 0x3FFFu) << 32;
  d |= static_cast<uint64_t>(1) << 46;
  return d;   // layout type 0 (no swizzle) in bits 61-63
}

// Instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both K-major,
// N = 32, M = 128.
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((kC >> 3) << 17) | ((128 >> 4) << 24);

// One MMA, issued by the lane whose leader flag is set. The whole warp runs the issue loop: a
// descriptor derived by one lane alone would have to be moved to the uniform registers the
// instruction reads it from, four moves an MMA.
__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t accumulate, uint32_t leader) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "setp.ne.b32 q, %5, 0;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem_d),
      "l"(a), "l"(b), "r"(kIdesc), "r"(accumulate), "r"(leader));
}

__device__ __forceinline__ void mma_commit(uint32_t mbar, uint32_t leader) {
  asm volatile(
      "{\n\t.reg .pred q;\n\t"
      "setp.ne.b32 q, %1, 0;\n\t"
      "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}\n" ::"r"(mbar), "r"(leader)
      : "memory");
}

// Poll the mbarrier for phase `parity` at most kWaitLimit times; true once it completed.
__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t parity) {
  for (long long i = 0; i < kWaitLimit; ++i) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(done)
        : "r"(mbar), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

// The CTA's closing barrier, which every thread reaches once its role is done: a wait that ran out
// in any role and warp (each decides for itself) counts, once per CTA.
__device__ __forceinline__ void close_cta(bool ok) {
  const int any = __syncthreads_or(ok ? 0 : 1);
  if (any && threadIdx.x == 0) atomicAdd(&g_conv_tc_timeouts, 1);
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]),
        "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]),
        "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ uint32_t bf2(float a, float b) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);   // a -> low half
  uint32_t u;
  memcpy(&u, &h, 4);
  return u;
}

__device__ __forceinline__ float2 unbf2(uint32_t u) {
  __nv_bfloat162 h;
  memcpy(&h, &u, 4);
  return __bfloat1622float2(h);
}

__device__ __forceinline__ void mbar_init(uint32_t mbar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(mbar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t mbar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(mbar) : "memory");
}

// The epilogue of one output voxel: acc[32] of the MMA.
template <int EPI>
__device__ __forceinline__ void conv_epilogue(const float (&acc)[32], const float (&bo)[32], const float (&so)[6],
                                              size_t v, size_t N, const uint4 (&rr)[4], const uint4 (&mm)[4], bool has_res,
                                              __nv_bfloat16* __restrict__ out, float* __restrict__ outf) {
  if (EPI == HOMO_NN_PLANES || EPI == HOMO_NN_PLANES_ADD) {
#pragma unroll
    for (int o = 0; o < 18; ++o) {
      float* d = outf + static_cast<size_t>(o) * N + v;
      const float val = so[o / 3] * (acc[o] + bo[o]);
      *d = EPI == HOMO_NN_PLANES_ADD ? *d + val : val;
    }
    return;
  }
  uint4* dst = reinterpret_cast<uint4*>(out + v * kC);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const uint32_t r4[4] = {rr[q].x, rr[q].y, rr[q].z, rr[q].w}, m4[4] = {mm[q].x, mm[q].y, mm[q].z, mm[q].w};
    uint32_t pk[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int o = 8 * q + 2 * j;
      float v0 = acc[o] + bo[o], v1 = acc[o + 1] + bo[o + 1];
      if (has_res) {
        const float2 r = unbf2(r4[j]);
        v0 += r.x;
        v1 += r.y;
      }
      if (EPI == HOMO_NN_RELU) {
        v0 = fmaxf(v0, 0.f);
        v1 = fmaxf(v1, 0.f);
      } else {
        const float2 m = unbf2(m4[j]);
        v0 = m.x > 0.f ? v0 : 0.f;
        v1 = m.y > 0.f ? v1 : 0.f;
      }
      pk[j] = bf2(v0, v1);
    }
    dst[q] = make_uint4(pk[0], pk[1], pk[2], pk[3]);
  }
}

template <int CIN, int EPI, typename TL>
__global__ void __launch_bounds__(kThreads, 1)
    k_conv3d_tc(int n, int tiles_x, int tiles_y, int ntiles, const __nv_bfloat16* __restrict__ x,
                const __nv_bfloat16* __restrict__ w, const float* __restrict__ bias,
                const __nv_bfloat16* __restrict__ res, const __nv_bfloat16* __restrict__ mask,
                __nv_bfloat16* __restrict__ out, float* __restrict__ outf, TcScale sc) {
  using S = TcShape<CIN, TL>;
  constexpr int kCh = S::kChunks, kStages = TL::kStages, kRows = TL::kRows, kBoxRows = TL::kBoxRows;
  constexpr int kPlaneBytes = TL::kPlaneBytes, BX = TL::BX, BY = TL::BY;
  extern __shared__ __align__(128) unsigned char smem[];
  unsigned char* wsm = smem + kStages * S::kBoxBytes;     // [tap][chunk][o][16 B]
  uint64_t* mbar = reinterpret_cast<uint64_t*>(wsm + S::kWBytes);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(mbar + TL::kBarriers);
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const size_t N = static_cast<size_t>(n) * n * n;
  const uint32_t box_s = smem_u32(smem), w_s = smem_u32(wsm), bar_s = smem_u32(mbar);
  // barriers: box filled / box free per stage, accumulators filled / free per pair
  auto full = [&](int s) { return bar_s + 8u * s; };
  auto empty = [&](int s) { return bar_s + 8u * (kStages + s); };
  auto tfull = [&](int t) { return bar_s + 8u * (2 * kStages + t); };
  auto tempty = [&](int t) { return bar_s + 8u * (2 * kStages + 2 + t); };

  // weights once per CTA; guard rows of every plane zeroed once (never loaded)
  for (int c = tid; c < kTaps * kC * kCh; c += kThreads) {
    const int ch = c % kCh, o = (c / kCh) % kC, tap = c / (kCh * kC);
    cp_async16(w_s + ((tap * kCh + ch) * kC + o) * 16, w + (static_cast<size_t>(tap) * kC + o) * CIN + ch * 8);
  }
  asm volatile("cp.async.commit_group;\n" ::: "memory");
  for (int c = tid; c < kStages * kCh * (kRows - kBoxRows); c += kThreads) {
    const int p = c / (kRows - kBoxRows), r = kBoxRows + c % (kRows - kBoxRows);   // plane p of all stages
    *reinterpret_cast<uint4*>(smem + p * kPlaneBytes + r * 16) = make_uint4(0u, 0u, 0u, 0u);
  }
  if (tid == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(full(s), kRole);
      mbar_init(empty(s), 1);
    }
    for (int t = 0; t < 2; ++t) {
      mbar_init(tfull(t), 1);
      mbar_init(tempty(t), kEpi);
    }
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tmem_slot)),
                 "r"(TL::kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  asm volatile("cp.async.wait_group 0;\n" ::: "memory");
  asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");   // weights and guard rows visible to the tensor core
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  const uint32_t tmem = *tmem_slot;
  bool ok = true;    // no wait of this thread's role ran out

  if (warp >= 8 && warp < 12) {
    // ---- copies: box rows t, t + 128, ... and all their chunks per thread
    const int t = tid - kEpi;
    int k = 0;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++k) {
      const int st = k % kStages;
      ok = mbar_wait(empty(st), ((k / kStages) & 1) ^ 1);   // a fresh barrier passes parity 1
      if (!ok) break;
      const int tx = tile % tiles_x, rest = tile / tiles_x;
      const int x0 = tx * TL::TX, y0 = (rest % tiles_y) * TL::TY, z0 = (rest / tiles_y) * TL::TZ;
      const uint32_t dst = box_s + st * S::kBoxBytes;
#pragma unroll 4
      for (int br = t; br < kBoxRows; br += kRole) {
        const int bx = br % BX, by = (br / BX) % BY, bz = br / (BX * BY);
        // a box starts at most one period in and spans at most BX: past it only on small grids
        const int gx = x0 - 1 + bx, gy = y0 - 1 + by, gz = z0 - 1 + bz;
        const size_t gv = n >= BX ? static_cast<size_t>(wrap1(gx, n)) +
                                        static_cast<size_t>(n) * (wrap1(gy, n) + static_cast<size_t>(n) * wrap1(gz, n))
                                  : static_cast<size_t>(wrapc(gx, n)) +
                                        static_cast<size_t>(n) * (wrapc(gy, n) + static_cast<size_t>(n) * wrapc(gz, n));
        const __nv_bfloat16* src = x + gv * CIN;
#pragma unroll
        for (int ch = 0; ch < kCh; ++ch) cp_async16(dst + ch * kPlaneBytes + br * 16, src + ch * 8);
      }
      asm volatile("cp.async.commit_group;\n" ::: "memory");
      asm volatile("cp.async.wait_group 0;\n" ::: "memory");
      asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
      mbar_arrive(full(st));
    }
  } else if (warp == 12) {
    // ---- MMAs: the warp runs the loop, one elected lane issues
    uint32_t leader;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}\n" : "=r"(leader));
    const uint64_t a0 = smem_desc(box_s, kPlaneBytes, 128), b0 = smem_desc(w_s, kC * 16, 128);
    int k = 0;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++k) {
      const int st = k % kStages, ac = k & 1;
      ok = mbar_wait(tempty(ac), ((k >> 1) & 1) ^ 1) && mbar_wait(full(st), (k / kStages) & 1);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
#pragma unroll 1
      for (int unit = 0; unit < TL::kUnits; ++unit) {
        const int zo = unit / TL::kBlocks, blk = unit - zo * TL::kBlocks;
        // box row of output (0, 0, zo), then the unit's block; descriptor addresses count 16-byte rows
        const uint64_t az = a0 + static_cast<uint32_t>(st * (S::kBoxBytes / 16) + ((zo + 1) * BY + 1) * BX + 1 + 128 * blk);
        const uint32_t d = tmem + (ac * TL::kUnits + unit) * kC;
#pragma unroll
        for (int tap = 0; tap < kTaps; ++tap) {
          const int row = ((tap / 9 - 1) * BY + (tap / 3) % 3 - 1) * BX + tap % 3 - 1;
#pragma unroll
          for (int ks = 0; ks < CIN / 16; ++ks)
            mma_bf16(d, az + static_cast<int64_t>(row + 2 * ks * kRows), b0 + (tap * kCh + 2 * ks) * kC,
                     (tap | ks) != 0 ? 1u : 0u, leader);
        }
      }
      mma_commit(empty(st), leader);
      mma_commit(tfull(ac), leader);
    }
    // the last commit covers every MMA issued: none runs when the CTA frees its TMEM and shared
    // memory, whoever gave up (bounded like the others; the epilogue waits for the same)
    if (k > 0) ok = mbar_wait(tfull((k - 1) & 1), ((k - 1) >> 1) & 1) && ok;
    __syncwarp();
  } else {
    // ---- epilogue: warps 0..3 take the even units, 4..7 the odd ones; warp w can read TMEM lanes
    // 32 (w % 4) .. + 31, the same rows of a unit's block
    const int set = warp >> 2, row0 = 32 * (warp & 3) + lane;
    const uint32_t tlane = tmem + (static_cast<uint32_t>(32 * (warp & 3)) << 16);
    float bo[kC], so[6];
#pragma unroll
    for (int o = 0; o < kC; ++o) bo[o] = (EPI != HOMO_NN_MASK && bias) ? bias[o] : 0.f;
#pragma unroll
    for (int o = 0; o < 6; ++o) so[o] = sc.s[o];
    const bool has_res = (EPI == HOMO_NN_RELU || EPI == HOMO_NN_MASK) && res != nullptr;
    int k = 0;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++k) {
      const int ac = k & 1;
      const int tx = tile % tiles_x, rest = tile / tiles_x;
      const int x0 = tx * TL::TX, y0 = (rest % tiles_y) * TL::TY, z0 = (rest / tiles_y) * TL::TZ;
#pragma unroll 1
      for (int unit = set; unit < TL::kUnits; unit += 2) {
        const int zo = unit / TL::kBlocks, row = (unit - zo * TL::kBlocks) * 128 + row0;
        const int ly = row / BX, lx = row - ly * BX;
        const int gx = x0 + lx, gy = y0 + ly, gz = z0 + zo;
        const bool live = lx < TL::TX && ly < TL::TY && gx < n && gy < n && gz < n;
        const size_t v = live ? static_cast<size_t>(gx) + static_cast<size_t>(n) * (gy + static_cast<size_t>(n) * gz) : 0;
        uint4 rr[4], mm[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {   // the residual and the mask do not wait for the MMAs
          rr[q] = has_res && live ? reinterpret_cast<const uint4*>(res + v * kC)[q] : make_uint4(0u, 0u, 0u, 0u);
          mm[q] = EPI == HOMO_NN_MASK && live ? reinterpret_cast<const uint4*>(mask + v * kC)[q] : make_uint4(0u, 0u, 0u, 0u);
        }
        if (unit == set) {
          ok = mbar_wait(tfull(ac), (k >> 1) & 1);
          ok = __all_sync(0xffffffffu, ok);   // a warp takes one decision (its TMEM loads are collective)
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        }
        float acc[32];
        tmem_ld32(tlane + (ac * TL::kUnits + unit) * kC, acc);
        if (unit + 2 >= TL::kUnits) {
          asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
          mbar_arrive(tempty(ac));
        }
        if (live) conv_epilogue<EPI>(acc, bo, so, v, N, rr, mm, has_res, out, outf);
        __syncwarp();
      }
      if (!ok) break;
    }
    // a warp that gives up leaves this tile and the rest unwritten; the other roles' waits then run
    // out too
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  close_cta(ok);
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(TL::kTmemCols) : "memory");
  }
}

// The bounded wait and the CTA's closing vote on their own: in CTA b one warp, b mod 13, waits on an
// mbarrier that no one arrives on and gives up after kWaitLimit polls, the others' waits complete
// at once; the CTA counts one timeout whichever warp it was (no MMA is issued here, so nothing is
// left in flight).
__global__ void __launch_bounds__(kThreads) k_wait_probe() {
  __shared__ __align__(8) uint64_t bar;
  const uint32_t b = smem_u32(&bar);
  if (threadIdx.x == 0) mbar_init(b, 1);
  __syncthreads();
  const bool stuck = threadIdx.x / 32 == blockIdx.x % (kThreads / 32);
  close_cta(mbar_wait(b, stuck ? 0 : 1));   // a fresh barrier passes parity 1
}

int g_sms = 0;

int sm_count() {
  if (g_sms == 0) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&g_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || g_sms < 1)
      g_sms = 152;
  }
  return g_sms;
}

template <int CIN, int EPI, typename TL>
cudaError_t tc_launch_tile(int n, const void* x, const void* w, const float* bias, const void* res, const void* mask,
                           void* out, float* outf, const TcScale& sc, cudaStream_t s) {
  using S = TcShape<CIN, TL>;
  auto kern = k_conv3d_tc<CIN, EPI, TL>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, S::kBytes);
  if (e != cudaSuccess) return e;
  const int tiles_x = (n + TL::TX - 1) / TL::TX, tiles_y = (n + TL::TY - 1) / TL::TY, tiles_z = (n + TL::TZ - 1) / TL::TZ;
  const long long ntiles = static_cast<long long>(tiles_x) * tiles_y * tiles_z;
  const int grid = static_cast<int>(std::min<long long>(ntiles, sm_count()));
  kern<<<grid, kThreads, S::kBytes, s>>>(n, tiles_x, tiles_y, static_cast<int>(ntiles),
                                         static_cast<const __nv_bfloat16*>(x), static_cast<const __nv_bfloat16*>(w),
                                         bias, static_cast<const __nv_bfloat16*>(res),
                                         static_cast<const __nv_bfloat16*>(mask), static_cast<__nv_bfloat16*>(out),
                                         outf, sc);
  return cudaGetLastError();
}

// Row blocks the busiest SM computes with a shape: what the kernel's time is proportional to.
template <typename TL>
long long tile_rounds(int n) {
  const long long tiles = static_cast<long long>((n + TL::TX - 1) / TL::TX) * ((n + TL::TY - 1) / TL::TY) *
                          ((n + TL::TZ - 1) / TL::TZ);
  return (tiles + sm_count() - 1) / sm_count() * TL::kUnits;
}

template <int CIN, int EPI>
cudaError_t tc_launch(int n, const void* x, const void* w, const float* bias, const void* res, const void* mask,
                      void* out, float* outf, const double* scale, cudaStream_t s) {
  TcScale sc;
  for (int k = 0; k < 6; ++k) sc.s[k] = scale ? static_cast<float>(scale[k]) : 1.f;
  return tile_rounds<TileB>(n) < tile_rounds<TileA>(n)
             ? tc_launch_tile<CIN, EPI, TileB>(n, x, w, bias, res, mask, out, outf, sc, s)
             : tc_launch_tile<CIN, EPI, TileA>(n, x, w, bias, res, mask, out, outf, sc, s);
}

}  // namespace

// tcgen05 convolution for c_in in {16, 32} and every epilogue (the contract of
// homo_nn_conv3d).
cudaError_t conv3d_tc(int n, int cin, int epi, const void* x, const void* w, const float* bias, const void* res,
                      const void* mask, void* out, float* outf, const double* scale, cudaStream_t s) {
#define HOMO_TC_CASE(CI, EP) \
  if (cin == CI && epi == EP) return tc_launch<CI, EP>(n, x, w, bias, res, mask, out, outf, scale, s);
  HOMO_TC_CASE(16, HOMO_NN_RELU)
  HOMO_TC_CASE(32, HOMO_NN_RELU)
  HOMO_TC_CASE(32, HOMO_NN_MASK)
  HOMO_TC_CASE(32, HOMO_NN_PLANES)
  HOMO_TC_CASE(32, HOMO_NN_PLANES_ADD)
#undef HOMO_TC_CASE
  return cudaErrorInvalidValue;
}

cudaError_t conv3d_tc_wait_probe(int blocks) {
  k_wait_probe<<<blocks, kThreads>>>();
  const cudaError_t e = cudaGetLastError();
  return e != cudaSuccess ? e : cudaDeviceSynchronize();
}

// Number of CTAs in which a wait ran out since the last call (and reset it).
int conv3d_tc_take_timeouts() {
  int h = 0;
  if (cudaMemcpyFromSymbol(&h, g_conv_tc_timeouts, sizeof(int)) != cudaSuccess) return -1;
  const int zero = 0;
  if (cudaMemcpyToSymbol(g_conv_tc_timeouts, &zero, sizeof(int)) != cudaSuccess) return -1;
  return h;
}

}  // namespace homo
