// Vector kernels of the CG driver, reductions, the periodic density filter and the OC
// update. All reductions are two-stage and deterministic: per-block partials in FP64,
// then one block sums them in a fixed order.
#include <algorithm>
#include <cmath>

#include "dev_common.cuh"

namespace homo {

namespace {

// W consecutive floats (W = 4: one 16-byte access; the caller guarantees alignment, i.e.
// N % 4 == 0 so that every plane starts on a 16-byte boundary).
template <int W>
struct Pk {
  float v[W];
};

template <int W>
__device__ __forceinline__ Pk<W> ldg_pk(const float* __restrict__ p) {
  Pk<W> r;
  if constexpr (W == 4) {
    const float4 t = __ldg(reinterpret_cast<const float4*>(p));
    r.v[0] = t.x; r.v[1] = t.y; r.v[2] = t.z; r.v[3] = t.w;
  } else {
    r.v[0] = __ldg(p);
  }
  return r;
}

template <int W>
__device__ __forceinline__ Pk<W> ld_pk(const float* p) {
  Pk<W> r;
  if constexpr (W == 4) {
    const float4 t = *reinterpret_cast<const float4*>(p);
    r.v[0] = t.x; r.v[1] = t.y; r.v[2] = t.z; r.v[3] = t.w;
  } else {
    r.v[0] = *p;
  }
  return r;
}

template <int W>
__device__ __forceinline__ void st_pk(float* p, const Pk<W>& x) {
  if constexpr (W == 4) *reinterpret_cast<float4*>(p) = make_float4(x.v[0], x.v[1], x.v[2], x.v[3]);
  else *p = x.v[0];
}

// hi + lo += d + dlo in double-float (TwoSum, then FastTwoSum renormalisation), with
// operations the compiler may not contract or reorder.
__device__ __forceinline__ void df_add(float& hi, float& lo, float d, float dlo) {
  const float sm = __fadd_rn(hi, d);
  const float bb = __fadd_rn(sm, -hi);
  const float er = __fadd_rn(__fadd_rn(hi, -__fadd_rn(sm, -bb)), __fadd_rn(d, -bb));
  const float l = __fadd_rn(__fadd_rn(lo, dlo), er);
  const float s2 = __fadd_rn(sm, l);
  lo = __fadd_rn(l, -__fadd_rn(s2, -sm));
  hi = s2;
}

// CG scalar steps (thread c < 6 of a block that has just written the sums they read; the FP32
// plane means by thread q < 18 of its second warp).
__device__ __forceinline__ float* f32_of(double* s) { return reinterpret_cast<float*>(s + S_F32); }

__device__ __forceinline__ void plane_mean(double* s, int sum_slot, int mean_slot, int q, double N) {
  f32_of(s)[mean_slot + q] = static_cast<float>(s[sum_slot + q] / N);
}

__device__ __forceinline__ void cg_alpha(double* s, int c) {
  const double pq = s[S_PQ + c];
  double a = 0.0;
  if (s[S_ACTIVE + c] != 0.0 && pq > 0.0 && isfinite(pq)) a = s[S_RZ + c] / pq;
  s[S_ALPHA + c] = a;
  f32_of(s)[F_ALPHA + c] = static_cast<float>(a);
}

// beta = rz_new / rz_old (0 on the first step or for finished cases); rz_old <- rz_new.
__device__ __forceinline__ void cg_beta(double* s, int c, int first) {
  const double rz = s[S_RZ + c], old = s[S_RZ_OLD + c];
  double b = 0.0;
  if (!first && s[S_ACTIVE + c] != 0.0 && old != 0.0 && isfinite(rz)) b = rz / old;
  s[S_BETA + c] = b;
  f32_of(s)[F_BETA + c] = static_cast<float>(b);
  s[S_RZ_OLD + c] = rz;
}

// The stored residual keeps the plane means it had when it was last recomputed (the
// rigid translations, outside the range of K); every consumer subtracts them. This
// step turns the raw sums into the centred norms ||r_c - mean||^2 = sum r^2 - sum^2/N
// and the plane means, and marks case c active while ||r_c||^2 > tol^2 ||f_c||^2.
__device__ __forceinline__ void cg_active(double* s, int c, double tol2, double N) {
  double rr = s[S_RR + c];
  for (int k = 0; k < 3; ++k) {
    const double sum = s[S_RSUM + 3 * c + k];
    rr -= sum * sum / N;
  }
  rr = fmax(rr, 0.0);
  s[S_RR + c] = rr;
  const double ff = s[S_FF + c];
  s[S_ACTIVE + c] = (ff > 0.0 && rr > tol2 * ff) ? 1.0 : 0.0;
}

// out[k] = sum over the nblk rows of part, then the CG step the sums are for (STEP: SumStep;
// scal: the slots, out one of them). One block: the step needs no launch of its own, which
// cost a small cell's iteration three of its launches. 16 loads of a thread in flight: with 4 the
// one block took 33 us over 2432 x 24 partials.
template <int STEP>
__global__ void __launch_bounds__(256) k_sum_partials(const double* __restrict__ part, int nblk,
                                                      int nv, double* out, double* scal, int first,
                                                      double tol2, double N) {
  // thread t owns value k = t % nv of rows r0, r0 + per, r0 + 2 per, ... (r0 = t / nv):
  // the block reads the row-major partials contiguously, with four independent sums
  __shared__ double sh[256];
  const int t = threadIdx.x;
  const int per = blockDim.x / nv;
  const int k = t % nv, r0 = t / nv;
  double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
  if (r0 < per) {
    const size_t stride = static_cast<size_t>(per) * nv;
    const size_t total = static_cast<size_t>(nblk) * nv;
    size_t i = static_cast<size_t>(r0) * nv + k;
#pragma unroll 4
    for (; i + 3 * stride < total; i += 4 * stride) {
      s0 += __ldg(part + i);
      s1 += __ldg(part + i + stride);
      s2 += __ldg(part + i + 2 * stride);
      s3 += __ldg(part + i + 3 * stride);
    }
    for (; i < total; i += stride) s0 += __ldg(part + i);
  }
  sh[t] = (s0 + s1) + (s2 + s3);
  __syncthreads();
  if (t < nv) {
    double acc = 0.0;
    for (int r = 0; r < per; ++r) acc += sh[r * nv + t];
    out[t] = acc;
  }
  if (STEP == kSumOnly) return;
  __syncthreads();
  if (t >= 32 && t < 32 + kPlanes)
    plane_mean(scal, STEP == kSumAlpha ? S_QSUM : STEP == kSumBeta ? S_ZSUM : S_RSUM,
               STEP == kSumAlpha ? F_QMEAN : STEP == kSumBeta ? F_ZMEAN : F_RMEAN, t - 32, N);
  if (t >= kCases) return;
  if (STEP == kSumAlpha) cg_alpha(scal, t);
  if (STEP == kSumBeta) cg_beta(scal, t, first);
  if (STEP == kSumActive) cg_active(scal, t, tol2, N);
}

// The CG vector kernels take one load case per blockIdx.y (3 planes a thread): six times the
// blocks of a thread for all 18 planes, whose loads a small cell waits for one plane after
// another (16^3: 12 to 17 us a kernel). A case's sums keep their order and their block: row
// blockIdx.x of the partials holds the 6 dots, then the 18 plane sums.
constexpr int kCgSums = kCases + kPlanes;

// Block sums of (dot, 3 plane sums) of case c into their slots of partial row blockIdx.x.
__device__ __forceinline__ void case_sums_store(const float (&v)[4], int c, double* part) {
  __shared__ float sh[32][4];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int nw = (blockDim.x + 31) >> 5;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    float s = v[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) sh[wid][k] = s;
  }
  __syncthreads();
  if (threadIdx.x < 4) {
    const int k = threadIdx.x;
    double s = 0.0;
    for (int w = 0; w < nw; ++w) s += static_cast<double>(sh[w][k]);
    part[static_cast<size_t>(blockIdx.x) * kCgSums + (k == 0 ? c : kCases + 3 * c + k - 1)] = s;
  }
}

// Per case c: sum over the 3 planes of case c of a*b. Each thread takes W consecutive
// vertices per step (W = 4: 16-byte accesses, four times the bytes in flight).
template <int W>
__global__ void __launch_bounds__(256) k_dot6(const float* __restrict__ a,
                                              const float* __restrict__ b, size_t N,
                                              double* __restrict__ part) {
  float red[kCases];
#pragma unroll
  for (int c = 0; c < kCases; ++c) red[c] = 0.f;
  for (size_t i = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < N / W;
       i += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const size_t v = i * W;
#pragma unroll
    for (int q = 0; q < kPlanes; ++q) {
      const Pk<W> x = ldg_pk<W>(a + q * N + v), y = ldg_pk<W>(b + q * N + v);
#pragma unroll
      for (int w = 0; w < W; ++w) red[q / 3] = fmaf(x.v[w], y.v[w], red[q / 3]);
    }
  }
  block_sum_store<kCases>(red, part);
}

// (r_c - mean r, z_c) for the 6 cases and the 18 plane sums of z (for removing its mean).
// rmean: 18 plane means of r, or null.
template <int W>
__global__ void __launch_bounds__(256) k_dot6_zsum(const float* __restrict__ r,
                                                   const float* __restrict__ z, size_t N,
                                                   const float* __restrict__ rmean,
                                                   double* __restrict__ part) {
  const int c = blockIdx.y;
  float red[4] = {0.f, 0.f, 0.f, 0.f}, rm[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) rm[k] = rmean ? __ldg(rmean + 3 * c + k) : 0.f;
  r += 3 * c * N;
  z += 3 * c * N;
  for (size_t i = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < N / W;
       i += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const size_t v = i * W;
    Pk<W> zz[3], rr[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      zz[k] = ldg_pk<W>(z + k * N + v);
      rr[k] = ldg_pk<W>(r + k * N + v);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int w = 0; w < W; ++w) {
        red[0] = fmaf(rr[k].v[w] - rm[k], zz[k].v[w], red[0]);
        red[1 + k] += zz[k].v[w];
      }
  }
  case_sums_store(red, c, part);
}

// e += alpha p, e kept in double-float (e + elo): the product is split exactly (its
// rounding error recovered with an FMA) and both parts are added with error-free
// transformations, so the correction carries no FP32 rounding noise; K applied to such
// noise would be amplified by the operator's spread of eigenvalues and leave the true
// residual far above the recursive one. r -= alpha (q - mean q) in FP32. Partial sums of
// ||r_c||^2 and of the 18 plane sums of r. s: the FP32 scalars (SlotF).
template <int W>
__global__ void __launch_bounds__(256) k_cg_update_er(float* __restrict__ e, float* __restrict__ elo,
                                                      float* __restrict__ r,
                                                      const float* __restrict__ p,
                                                      const float* __restrict__ q,
                                                      const float* __restrict__ s, size_t N,
                                                      double* __restrict__ part) {
  const int c = blockIdx.y;
  const float a = __ldg(s + F_ALPHA + c);
  float red[4] = {0.f, 0.f, 0.f, 0.f}, qm[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) qm[k] = __ldg(s + F_QMEAN + 3 * c + k);
  e += 3 * c * N;
  elo += 3 * c * N;
  r += 3 * c * N;
  p += 3 * c * N;
  q += 3 * c * N;
  for (size_t i = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < N / W;
       i += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const size_t v = i * W;
    Pk<W> rv[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) rv[k] = ld_pk<W>(r + k * N + v);
    if (a != 0.f) {
      Pk<W> pv[3], qv[3], hi[3], lo[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        pv[k] = ldg_pk<W>(p + k * N + v);
        qv[k] = ldg_pk<W>(q + k * N + v);
        hi[k] = ld_pk<W>(e + k * N + v);
        lo[k] = ld_pk<W>(elo + k * N + v);
      }
#pragma unroll
      for (int k = 0; k < 3; ++k) {
#pragma unroll
        for (int w = 0; w < W; ++w) {
          const float pr = __fmul_rn(a, pv[k].v[w]);        // TwoProd: pr + pe = a p exactly
          const float pe = fmaf(a, pv[k].v[w], -pr);
          df_add(hi[k].v[w], lo[k].v[w], pr, pe);
          rv[k].v[w] = fmaf(-a, qv[k].v[w] - qm[k], rv[k].v[w]);
        }
        st_pk<W>(e + k * N + v, hi[k]);
        st_pk<W>(elo + k * N + v, lo[k]);
        st_pk<W>(r + k * N + v, rv[k]);
      }
    }
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int w = 0; w < W; ++w) {
        red[0] = fmaf(rv[k].v[w], rv[k].v[w], red[0]);
        red[1 + k] += rv[k].v[w];
      }
  }
  case_sums_store(red, c, part);
}

// (u + ulo) += (e + elo) in double-float arithmetic (error-free transformations with
// non-contracted operations), then e = elo = 0. Closes a CG cycle. n % W == 0.
template <int W>
__global__ void __launch_bounds__(256) k_fold(float* __restrict__ u, float* __restrict__ ulo,
                                              float* __restrict__ e, float* __restrict__ elo,
                                              size_t n) {
  Pk<W> zero;
#pragma unroll
  for (int w = 0; w < W; ++w) zero.v[w] = 0.f;
  for (size_t i = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n / W;
       i += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const size_t o = i * W;
    const Pk<W> d = ld_pk<W>(e + o), dlo = ld_pk<W>(elo + o);
    Pk<W> hi = ld_pk<W>(u + o), lo = ld_pk<W>(ulo + o);
#pragma unroll
    for (int w = 0; w < W; ++w) df_add(hi.v[w], lo.v[w], d.v[w], dlo.v[w]);
    st_pk<W>(u + o, hi);
    st_pk<W>(ulo + o, lo);
    st_pk<W>(e + o, zero);
    st_pk<W>(elo + o, zero);
  }
}

// p = (z - mean(z)) + beta p per plane. s: the FP32 scalars (SlotF).
template <int W>
__global__ void __launch_bounds__(256) k_cg_update_p(float* __restrict__ p,
                                                     const float* __restrict__ z,
                                                     const float* __restrict__ s, size_t N) {
  const int c = blockIdx.y;
  const float b = __ldg(s + F_BETA + c);
  float mz[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) mz[k] = __ldg(s + F_ZMEAN + 3 * c + k);
  p += 3 * c * N;
  z += 3 * c * N;
  for (size_t i = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < N / W;
       i += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const size_t v = i * W;
    Pk<W> zz[3], pp[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      zz[k] = ldg_pk<W>(z + k * N + v);
      if (b != 0.f) pp[k] = ld_pk<W>(p + k * N + v);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
#pragma unroll
      for (int w = 0; w < W; ++w)
        pp[k].v[w] = b != 0.f ? fmaf(b, pp[k].v[w], zz[k].v[w] - mz[k]) : zz[k].v[w] - mz[k];
      st_pk<W>(p + k * N + v, pp[k]);
    }
  }
}

__global__ void k_split_set(float* __restrict__ hi, float* __restrict__ lo,
                            const float* __restrict__ src, size_t n) {
  for (size_t i = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
       i += static_cast<size_t>(gridDim.x) * blockDim.x) {
    hi[i] = src[i];
    lo[i] = 0.f;
  }
}

__global__ void k_split_get(const float* __restrict__ hi, const float* __restrict__ lo,
                            float* __restrict__ dst, size_t n) {
  for (size_t i = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
       i += static_cast<size_t>(gridDim.x) * blockDim.x)
    dst[i] = hi[i] + lo[i];
}

// Periodic linear-cone filter: out_e = inv_wsum * sum_k w_k in_(e + off_k).
// kSens = false: out_e = sum_d w(d) in_(e+d) / sum_d w(d) (density filter, its own
// adjoint). kSens = true: the density-weighted sensitivity filter of the unfiltered variant
// (Sec. 5.3), out_e = sum_d w(d) rho_(e+d) in_(e+d) / (max(gamma, rho_e) sum_d w(d)).
template <bool kSens>
__global__ void __launch_bounds__(256) k_filter(const __grid_constant__ FilterParam F, int n,
                                                const float* __restrict__ in,
                                                const float* __restrict__ rho, float gamma,
                                                float* __restrict__ out) {
  const size_t N = static_cast<size_t>(n) * n * n;
  for (size_t e = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; e < N;
       e += static_cast<size_t>(gridDim.x) * blockDim.x) {
    int x, y, z;
    decode3(static_cast<unsigned>(e), static_cast<unsigned>(n), x, y, z);
    float s = 0.f;
    for (int k = 0; k < F.count; ++k) {
      int xx = x + F.off[k][0], yy = y + F.off[k][1], zz = z + F.off[k][2];
      xx += xx < 0 ? n : (xx >= n ? -n : 0);
      yy += yy < 0 ? n : (yy >= n ? -n : 0);
      zz += zz < 0 ? n : (zz >= n ? -n : 0);
      const size_t f = xx + static_cast<size_t>(n) * (yy + static_cast<size_t>(n) * zz);
      const float v = kSens ? __ldg(in + f) * __ldg(rho + f) : __ldg(in + f);
      s = fmaf(F.w[k], v, s);
    }
    out[e] = kSens ? s * F.inv_wsum / fmaxf(gamma, __ldg(rho + e)) : s * F.inv_wsum;
  }
}

// The same for a radius in (sqrt 3, 2]: exactly the 27 offsets of the unit cube, in k_filter's
// order with its weights (w[k]: k nonzero components), so the result is bitwise k_filter's.
// The general loop spends about 20 integer instructions per offset on wrapping and on
// indexing its offset table; with the neighbour indices taken once per element the pass
// is bound by its 27 loads through L1 (192^3: 265 -> 58 us).
struct Filter27 {
  float w[4];
  float inv_wsum;
};

template <bool kSens>
__global__ void __launch_bounds__(256) k_filter27(Filter27 F, int n, const float* __restrict__ in,
                                                  const float* __restrict__ rho, float gamma,
                                                  float* __restrict__ out) {
  const unsigned N = static_cast<unsigned>(n) * n * n;
  for (unsigned e = blockIdx.x * blockDim.x + threadIdx.x; e < N; e += gridDim.x * blockDim.x) {
    int x, y, z;
    decode3(e, static_cast<unsigned>(n), x, y, z);
    const Nb nb = make_nb(x, y, z, n);
    float s = 0.f;
#pragma unroll
    for (int k = 0; k < 27; ++k) {
      const int a = k % 3, b = (k / 3) % 3, c = k / 9;
      const unsigned f = static_cast<unsigned>(nb.X[a] + nb.Y[b] + nb.Z[c]);
      const float v = kSens ? __ldg(in + f) * __ldg(rho + f) : __ldg(in + f);
      s = fmaf(F.w[(a != 1) + (b != 1) + (c != 1)], v, s);
    }
    out[e] = kSens ? s * F.inv_wsum / fmaxf(gamma, __ldg(rho + e)) : s * F.inv_wsum;
  }
}

// ---------------------------------------------------------------- OC update
// rho_new(s) = clamp(base_e * s, lo_e, hi_e), base_e = rho_e max(-dc_e, 0)^eta,
// s = lambda^(-eta); mean(rho_new) increases with s. OC scratch (doubles at S_OC):
constexpr int kOcCand = 15;      // candidate multipliers per pass
// kOcPasses passes (homo_internal.cuh): the bracket shrinks 16x per pass in log scale
enum { OC_SLO = 0, OC_SHI = 1, OC_MODE = 2, OC_CAND = 8, OC_CHANGE = 32, OC_TICKET = 56 };

// One launch per pass: the block that finishes last (a ticket counter, taken after its partials
// are fenced; no block waits) sums the partials in a fixed order and takes the pass's host-free
// decision. Sums: an FP32 pair per thread and through the warp (TwoSum), FP64 across warps:
// an FP64 warp reduction of 15 values by every thread cost 80 of the 90 us of a 192^3
// pass (2 FP64 operations per clock and SM). What is summed are the FP32 sums of the up to 8
// terms e, e + stride, ... e + 7 stride of a run (stride: the grid of one thread per element, at most 16 blocks per SM), which decide the last
// bits of the multiplier and with it the density: they keep their grouping whatever the grid.
// 192^3 update: 2600 -> 440 us in 10 launches instead of 28.
constexpr int kOcBlock = 256;
constexpr int kOcGrid = 152 * 4;

__device__ __forceinline__ float oc_lo(float r, float move, float rmin) { return fmaxf(rmin, r - move); }
__device__ __forceinline__ float oc_hi(float r, float move) { return fminf(1.f, r + move); }

// hi + lo += v with TwoSum, lo collecting the rounding errors
__device__ __forceinline__ void pair_add(float& hi, float& lo, float v) {
  const float s = __fadd_rn(hi, v);
  const float bb = __fadd_rn(s, -hi);
  lo = __fadd_rn(lo, __fadd_rn(__fadd_rn(hi, -__fadd_rn(s, -bb)), __fadd_rn(v, -bb)));
  hi = s;
}

// Block sums of NV FP32 pairs into part[blockIdx.x * NV + k] (FP64 across the warps). A high part
// that is infinite stays so (it is the plain FP32 sum), but TwoSum then leaves inf - inf in the low
// part, which does not count: the sum of a density with an infinite value is infinite, not NaN.
template <int NV>
__device__ __forceinline__ void pair_block_sum(float (&hi)[NV], float (&lo)[NV], double* part) {
  __shared__ float sh[kOcBlock / 32][NV], sl[kOcBlock / 32][NV];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < NV; ++k) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float h = __shfl_down_sync(0xffffffffu, hi[k], o), l = __shfl_down_sync(0xffffffffu, lo[k], o);
      pair_add(hi[k], lo[k], h);
      lo[k] = __fadd_rn(lo[k], l);
    }
    if (lane == 0) {
      sh[wid][k] = hi[k];
      sl[wid][k] = lo[k];
    }
  }
  __syncthreads();
  if (threadIdx.x < NV) {
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < kOcBlock / 32; ++w)
      s += static_cast<double>(sh[w][threadIdx.x]) +
           (isinf(sh[w][threadIdx.x]) ? 0.0 : static_cast<double>(sl[w][threadIdx.x]));
    part[static_cast<size_t>(blockIdx.x) * NV + threadIdx.x] = s;
  }
}

// True in every thread of the block that arrives last; its view of part is then complete.
__device__ __forceinline__ bool oc_last_block(double* oc) {
  __shared__ bool last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned* ticket = reinterpret_cast<unsigned*>(oc + OC_TICKET);
    last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    if (last) *ticket = 0u;
  }
  __syncthreads();
  if (last) __threadfence();
  return last;
}

// Sums over blocks of the NV partials (thread t: value t % NV, rows t / NV + i * per; then the
// rows' sums in order), valid in thread k < NV.
template <int NV>
__device__ __forceinline__ double oc_total(const double* part, int nblk) {
  __shared__ double sh[kOcBlock];
  constexpr int per = kOcBlock / NV;
  const int k = threadIdx.x % NV, r0 = threadIdx.x / NV;
  double s = 0.0;
  if (r0 < per)
#pragma unroll 8
    for (int r = r0; r < nblk; r += per) s += __ldcg(part + static_cast<size_t>(r) * NV + k);
  sh[threadIdx.x] = s;
  __syncthreads();
  double acc = 0.0;
  if (threadIdx.x < NV)
    for (int r = 0; r < per; ++r) acc += sh[r * NV + threadIdx.x];
  return acc;
}

// Thread k < kOcCand: candidate k of the bracket (log-uniform).
__device__ __forceinline__ void oc_make_candidates(double* oc, double lo, double hi) {
  if (threadIdx.x < kOcCand) {
    const double lr = log(hi / lo);
    oc[OC_CAND + threadIdx.x] = lo * exp(lr * (threadIdx.x + 1) / (kOcCand + 1));
  }
}

// W consecutive elements per step (4: 16-byte accesses; the launcher checks the alignment).
// base -> tmp; min lo/base, max hi/base over base > 0, sum lo, sum hi: the bracket of s.
template <int W>
__global__ void __launch_bounds__(kOcBlock) k_oc_setup(const float* __restrict__ rho,
                                                       const float* __restrict__ dc,
                                                       float* __restrict__ base, size_t N, float eta,
                                                       float move, float rmin, double V,
                                                       double* __restrict__ part, double* __restrict__ oc) {
  float mn = INFINITY, mx = 0.f;
  float hi2[2] = {0.f, 0.f}, lo2[2] = {0.f, 0.f};
  for (size_t i = static_cast<size_t>(blockIdx.x) * kOcBlock + threadIdx.x; i < N / W;
       i += static_cast<size_t>(gridDim.x) * kOcBlock) {
    const Pk<W> r = ldg_pk<W>(rho + i * W), d = ldg_pk<W>(dc + i * W);
    Pk<W> bs;
#pragma unroll
    for (int w = 0; w < W; ++w) {
      const float D = fmaxf(-d.v[w], 0.f);
      bs.v[w] = D > 0.f ? r.v[w] * powf(D, eta) : 0.f;
      const float lo = oc_lo(r.v[w], move, rmin), hi = oc_hi(r.v[w], move);
      pair_add(hi2[0], lo2[0], lo);
      pair_add(hi2[1], lo2[1], hi);
      if (bs.v[w] > 0.f) {
        mn = fminf(mn, lo / bs.v[w]);
        mx = fmaxf(mx, hi / bs.v[w]);
      }
    }
    st_pk<W>(base + i * W, bs);
  }
  __shared__ float smn[kOcBlock / 32], smx[kOcBlock / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    mn = fminf(mn, __shfl_down_sync(0xffffffffu, mn, o));
    mx = fmaxf(mx, __shfl_down_sync(0xffffffffu, mx, o));
  }
  if ((threadIdx.x & 31) == 0) {
    smn[threadIdx.x >> 5] = mn;
    smx[threadIdx.x >> 5] = mx;
  }
  pair_block_sum<2>(hi2, lo2, part);   // its barrier also publishes smn and smx
  double* ext = part + 2 * static_cast<size_t>(gridDim.x);
  if (threadIdx.x == 0) {
    for (int w = 1; w < kOcBlock / 32; ++w) {
      smn[0] = fminf(smn[0], smn[w]);
      smx[0] = fmaxf(smx[0], smx[w]);
    }
    ext[2 * blockIdx.x] = smn[0];
    ext[2 * blockIdx.x + 1] = smx[0];
  }
  if (!oc_last_block(oc)) return;
  __shared__ double tot[4];
  const double t = oc_total<2>(part, gridDim.x);
  if (threadIdx.x < 2) tot[threadIdx.x] = t;
  if (threadIdx.x >= 32 && threadIdx.x < 64) {
    double a = INFINITY, b = 0.0;
    for (int i = threadIdx.x - 32; i < static_cast<int>(gridDim.x); i += 32) {
      a = fmin(a, __ldcg(ext + 2 * i));
      b = fmax(b, __ldcg(ext + 2 * i + 1));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      a = fmin(a, __shfl_down_sync(0xffffffffu, a, o));
      b = fmax(b, __shfl_down_sync(0xffffffffu, b, o));
    }
    if (threadIdx.x == 32) {
      tot[2] = a;
      tot[3] = b;
    }
  }
  __syncthreads();
  const double lo = tot[2], hi = tot[3];
  const double vlo = tot[0] / static_cast<double>(N), vhi = tot[1] / static_cast<double>(N);
  int mode = 0;
  if (!(hi > 0.0) || !isfinite(lo) || vlo >= V) mode = 2;     // everything at its lower bound
  else if (vhi <= V) mode = 1;                                // everything at its upper bound
  if (threadIdx.x == 0) {
    oc[OC_SLO] = lo;
    oc[OC_SHI] = hi;
    oc[OC_MODE] = mode;
  }
  if (mode == 0) oc_make_candidates(oc, lo, hi);
}

// Volumes of the 15 candidates; the last block narrows the bracket to the two they straddle V
// with and makes the next candidates. stride: distance of a run's terms (a run: 8 of the
// elements v, v + stride, v + 2 stride, ... of one v < stride).
__global__ void __launch_bounds__(kOcBlock) k_oc_pass(const float* __restrict__ rho,
                                                      const float* __restrict__ base, size_t N,
                                                      size_t stride, float move, float rmin, double V,
                                                      double* oc, double* __restrict__ part) {
  if (oc[OC_MODE] != 0) return;
  __shared__ float cand_s[kOcCand];   // rounded to FP32 by one warp (a conversion is FP64-pipe work)
  if (threadIdx.x < kOcCand) cand_s[threadIdx.x] = static_cast<float>(oc[OC_CAND + threadIdx.x]);
  __syncthreads();
  float cand[kOcCand], hi[kOcCand], lo[kOcCand];
#pragma unroll
  for (int k = 0; k < kOcCand; ++k) {
    cand[k] = cand_s[k];
    hi[k] = lo[k] = 0.f;
  }
  const size_t runs = (N + 8 * stride - 1) / (8 * stride);
  for (size_t run = 0; run < runs; ++run)
    for (size_t v = static_cast<size_t>(blockIdx.x) * kOcBlock + threadIdx.x; v < stride;
         v += static_cast<size_t>(gridDim.x) * kOcBlock) {
      const size_t e0 = v + 8 * stride * run;
      if (e0 >= N) continue;
      float r[8], bs[8];
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        const size_t e = e0 + t * stride;
        r[t] = e < N ? __ldg(rho + e) : -1.f;
        bs[t] = e < N ? __ldg(base + e) : 0.f;
      }
      float acc[kOcCand];
#pragma unroll
      for (int k = 0; k < kOcCand; ++k) acc[k] = 0.f;
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        if (e0 + t * stride >= N) break;
        const float l = oc_lo(r[t], move, rmin), h = oc_hi(r[t], move);
#pragma unroll
        for (int k = 0; k < kOcCand; ++k) acc[k] += fminf(fmaxf(bs[t] * cand[k], l), h);
      }
#pragma unroll
      for (int k = 0; k < kOcCand; ++k) pair_add(hi[k], lo[k], acc[k]);
    }
  pair_block_sum<kOcCand>(hi, lo, part);
  if (!oc_last_block(oc)) return;
  __shared__ double vol[kOcCand], br[2];
  const double t = oc_total<kOcCand>(part, gridDim.x);
  if (threadIdx.x < kOcCand) vol[threadIdx.x] = t / static_cast<double>(N);
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = oc[OC_SLO], b = oc[OC_SHI];
    for (int k = 0; k < kOcCand; ++k) {
      if (vol[k] <= V) {
        a = oc[OC_CAND + k];
      } else {
        b = oc[OC_CAND + k];
        break;
      }
    }
    oc[OC_SLO] = br[0] = a;
    oc[OC_SHI] = br[1] = b;
  }
  __syncthreads();
  oc_make_candidates(oc, br[0], br[1]);
}

template <int W>
__global__ void __launch_bounds__(kOcBlock) k_oc_apply(float* __restrict__ rho,
                                                       const float* __restrict__ base, size_t N,
                                                       float move, float rmin, double* __restrict__ oc,
                                                       double* __restrict__ part) {
  const int mode = static_cast<int>(oc[OC_MODE]);
  const float s = mode == 2 ? 0.f : static_cast<float>(mode == 1 ? oc[OC_SHI] : oc[OC_SLO]);
  float ch = 0.f;
  for (size_t i = static_cast<size_t>(blockIdx.x) * kOcBlock + threadIdx.x; i < N / W;
       i += static_cast<size_t>(gridDim.x) * kOcBlock) {
    const Pk<W> r = ld_pk<W>(rho + i * W), bs = ldg_pk<W>(base + i * W);
    Pk<W> nr;
#pragma unroll
    for (int w = 0; w < W; ++w) {
      nr.v[w] = fminf(fmaxf(bs.v[w] * s, oc_lo(r.v[w], move, rmin)), oc_hi(r.v[w], move));
      ch = fmaxf(ch, fabsf(nr.v[w] - r.v[w]));
    }
    st_pk<W>(rho + i * W, nr);
  }
  __shared__ float sm[kOcBlock / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) ch = fmaxf(ch, __shfl_down_sync(0xffffffffu, ch, o));
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = ch;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kOcBlock / 32; ++w) ch = fmaxf(ch, sm[w]);
    part[blockIdx.x] = ch;
  }
  if (!oc_last_block(oc)) return;
  if (threadIdx.x < 32) {
    double m = 0.0;
    for (int i = threadIdx.x; i < static_cast<int>(gridDim.x); i += 32) m = fmax(m, __ldcg(part + i));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_down_sync(0xffffffffu, m, o));
    if (threadIdx.x == 0) oc[OC_CHANGE] = m;
  }
}

// Orbit averages under a cube symmetry group (Sec. 6.1). Thread per element: it forms
// the indices of the element's images (index arithmetic only) and continues only if its
// own index is the smallest, i.e. once per orbit; that thread sums the orbit's values in
// FP64 and writes the average to every member. For values within a factor 2^29 of each
// other (densities in [1e-3, 1], say) the FP64 sum of at most 48 FP32 values is exact, so
// the result does not depend on the order and every member gets the same FP32 value.
// Orbits are disjoint, so the kernel may run in place.
__device__ __forceinline__ unsigned sym_image(const SymParam& S, int g, int x, int y, int z, int n) {
  const int c[3] = {x, y, z};
  int j[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int p = S.perm[g][k];
    const int v = p == 0 ? c[0] : (p == 1 ? c[1] : c[2]);
    j[k] = ((S.flip[g] >> k) & 1) ? n - 1 - v : v;
  }
  return static_cast<unsigned>(j[0]) + static_cast<unsigned>(n) * (j[1] + static_cast<unsigned>(n) * j[2]);
}

__global__ void __launch_bounds__(256) k_symmetrize(const __grid_constant__ SymParam S, const float* in,
                                                    float* out, int n) {
  const unsigned N = static_cast<unsigned>(n) * n * n;
  for (unsigned e = blockIdx.x * blockDim.x + threadIdx.x; e < N; e += gridDim.x * blockDim.x) {
    int x, y, z;
    decode3(e, static_cast<unsigned>(n), x, y, z);
    bool canonical = true;
    for (int g = 0; g < S.count && canonical; ++g) canonical = sym_image(S, g, x, y, z, n) >= e;
    if (!canonical) continue;
    double acc = 0.0;
    for (int g = 0; g < S.count; ++g) acc += static_cast<double>(in[sym_image(S, g, x, y, z, n)]);
    const float avg = static_cast<float>(acc / S.count);
    for (int g = 0; g < S.count; ++g) out[sym_image(S, g, x, y, z, n)] = avg;
  }
}

// Trigonometric initialisation (Sec. 6.2), FP64 throughout (a one-time setup step).
// Basis order: T index 2 (3 (k - 1) + i) + {0: cos, 1: sin} of 2 pi k xb_i, then the
// products T_a T_b, a <= b, row by row; xb = R (centre - 1/2).
__global__ void __launch_bounds__(256) k_trig_basis(const __grid_constant__ TrigParam P, int n, double* y) {
  const unsigned N = static_cast<unsigned>(n) * n * n;
  const int nt = 6 * P.nb;
  for (unsigned e = blockIdx.x * blockDim.x + threadIdx.x; e < N; e += gridDim.x * blockDim.x) {
    int x, yy, z;
    decode3(e, static_cast<unsigned>(n), x, yy, z);
    const double c[3] = {(x + 0.5) / n - 0.5, (yy + 0.5) / n - 0.5, (z + 0.5) / n - 0.5};
    double xb[3];
    for (int r = 0; r < 3; ++r) xb[r] = P.R[3 * r] * c[0] + P.R[3 * r + 1] * c[1] + P.R[3 * r + 2] * c[2];
    double T[kTrigMaxT];
    for (int k = 1; k <= P.nb; ++k)
      for (int i = 0; i < 3; ++i) {
        double sv, cv;
        sincospi(2.0 * k * xb[i], &sv, &cv);
        T[2 * (3 * (k - 1) + i)] = cv;
        T[2 * (3 * (k - 1) + i) + 1] = sv;
      }
    double acc = 0.0;
    int idx = 0;
    for (int a = 0; a < nt; ++a) acc = fma(P.w[idx++], T[a], acc);
    for (int a = 0; a < nt; ++a)
      for (int b = a; b < nt; ++b) acc = fma(P.w[idx++], T[a] * T[b], acc);
    y[e] = acc;
  }
}

__device__ __forceinline__ double trig_sigmoid(double y, double mu, double k, double Vh, double rho_min) {
  const double r = rho_min + Vh / (1.0 + exp(-k * (y - mu)));
  return fmin(fmax(r, rho_min), 1.0);
}

__global__ void __launch_bounds__(256) k_trig_volume(const double* __restrict__ y, size_t N, double mu0,
                                                     double dmu, double k, double Vh, double rho_min,
                                                     double* __restrict__ part) {
  double acc[kTrigCand];
#pragma unroll
  for (int c = 0; c < kTrigCand; ++c) acc[c] = 0.0;
  for (size_t e = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; e < N;
       e += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const double v = y[e];
#pragma unroll
    for (int c = 0; c < kTrigCand; ++c) acc[c] += trig_sigmoid(v, mu0 + c * dmu, k, Vh, rho_min);
  }
  block_sum_store_d<kTrigCand>(acc, part);
}

__global__ void __launch_bounds__(256) k_trig_project(const double* __restrict__ y, size_t N, double mu,
                                                      double k, double Vh, double rho_min, float* rho) {
  for (size_t e = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; e < N;
       e += static_cast<size_t>(gridDim.x) * blockDim.x)
    rho[e] = static_cast<float>(trig_sigmoid(y[e], mu, k, Vh, rho_min));
}

}  // namespace

int reduce_grid(size_t n_items) { return grid_for(n_items, 256); }

cudaError_t launch_sum_partials(const double* part, int nblk, int nv, double* out,
                                cudaStream_t s) {
  if (nv < 1 || nv > 256) return cudaErrorInvalidValue;
  k_sum_partials<kSumOnly><<<1, 256, 0, s>>>(part, nblk, nv, out, nullptr, 0, 0.0, 0.0);
  return cudaGetLastError();
}

cudaError_t launch_sum_step(int step, const double* part, int nblk, double* scal, int first, double tol, size_t N,
                            cudaStream_t s) {
  const int nv = kCases + kPlanes;
  if (step == kSumAlpha)
    k_sum_partials<kSumAlpha><<<1, 256, 0, s>>>(part, nblk, nv, scal + S_PQ, scal, 0, 0.0, static_cast<double>(N));
  else if (step == kSumBeta)
    k_sum_partials<kSumBeta><<<1, 256, 0, s>>>(part, nblk, nv, scal + S_RZ, scal, first, 0.0, static_cast<double>(N));
  else if (step == kSumActive)
    k_sum_partials<kSumActive><<<1, 256, 0, s>>>(part, nblk, nv, scal + S_RR, scal, 0, tol * tol, static_cast<double>(N));
  else
    return cudaErrorInvalidValue;
  return cudaGetLastError();
}

cudaError_t launch_dot6(const float* a, const float* b, size_t N, double* part, int* grid_out,
                        cudaStream_t s) {
  const int g = grid_for(N % 4 == 0 ? N / 4 : N, 256);
  *grid_out = g;
  if (N % 4 == 0) k_dot6<4><<<g, 256, 0, s>>>(a, b, N, part);
  else k_dot6<1><<<g, 256, 0, s>>>(a, b, N, part);
  return cudaGetLastError();
}

cudaError_t launch_dot6_zsum(const float* r, const float* z, size_t N, const float* rmean,
                             double* part, int* grid_out, cudaStream_t s) {
  const int g = grid_for(N % 4 == 0 ? N / 4 : N, 256);
  *grid_out = g;
  if (N % 4 == 0) k_dot6_zsum<4><<<dim3(g, kCases), 256, 0, s>>>(r, z, N, rmean, part);
  else k_dot6_zsum<1><<<dim3(g, kCases), 256, 0, s>>>(r, z, N, rmean, part);
  return cudaGetLastError();
}

cudaError_t launch_cg_update_er(float* e, float* elo, float* r, const float* p, const float* q,
                                const double* scal, size_t N, double* part, int* grid_out,
                                cudaStream_t s) {
  const int g = grid_for(N % 4 == 0 ? N / 4 : N, 256);
  *grid_out = g;
  const float* fs = reinterpret_cast<const float*>(scal + S_F32);
  if (N % 4 == 0) k_cg_update_er<4><<<dim3(g, kCases), 256, 0, s>>>(e, elo, r, p, q, fs, N, part);
  else k_cg_update_er<1><<<dim3(g, kCases), 256, 0, s>>>(e, elo, r, p, q, fs, N, part);
  return cudaGetLastError();
}

cudaError_t launch_fold(float* u, float* ulo, float* e, float* elo, size_t n, cudaStream_t s) {
  if (n % 4 == 0) k_fold<4><<<grid_for(n / 4, 256), 256, 0, s>>>(u, ulo, e, elo, n);
  else k_fold<1><<<grid_for(n, 256), 256, 0, s>>>(u, ulo, e, elo, n);
  return cudaGetLastError();
}

cudaError_t launch_cg_update_p(float* p, const float* z, const double* scal, size_t N,
                               cudaStream_t s) {
  if (N % 4 == 0) k_cg_update_p<4><<<dim3(grid_for(N / 4, 256), kCases), 256, 0, s>>>(p, z, reinterpret_cast<const float*>(scal + S_F32), N);
  else k_cg_update_p<1><<<dim3(grid_for(N, 256), kCases), 256, 0, s>>>(p, z, reinterpret_cast<const float*>(scal + S_F32), N);
  return cudaGetLastError();
}

cudaError_t launch_split_set(float* hi, float* lo, const float* src, size_t n, cudaStream_t s) {
  k_split_set<<<grid_for(n, 256), 256, 0, s>>>(hi, lo, src, n);
  return cudaGetLastError();
}

cudaError_t launch_split_get(const float* hi, const float* lo, float* dst, size_t n,
                             cudaStream_t s) {
  k_split_get<<<grid_for(n, 256), 256, 0, s>>>(hi, lo, dst, n);
  return cudaGetLastError();
}

int build_sym_param(int kind, SymParam& sp) {
  sp.count = 0;
  const int perms[6][3] = {{0, 1, 2}, {0, 2, 1}, {1, 0, 2}, {1, 2, 0}, {2, 0, 1}, {2, 1, 0}};
  const int parity[6] = {1, -1, -1, 1, 1, -1};
  if (kind != HOMO_SYM_REFLECT3 && kind != HOMO_SYM_ROTATE3 && kind != HOMO_SYM_REFLECT6) return HOMO_EINVAL;
  for (int p = 0; p < 6; ++p)
    for (int f = 0; f < 8; ++f) {
      const int det = parity[p] * (((f & 1) + ((f >> 1) & 1) + (f >> 2)) % 2 ? -1 : 1);
      if (kind == HOMO_SYM_REFLECT3 && p != 0) continue;
      if (kind == HOMO_SYM_ROTATE3 && det != 1) continue;
      for (int k = 0; k < 3; ++k) sp.perm[sp.count][k] = static_cast<unsigned char>(perms[p][k]);
      sp.flip[sp.count] = static_cast<unsigned char>(f);
      ++sp.count;
    }
  return HOMO_OK;
}

cudaError_t launch_trig_basis(const TrigParam& tp, int n, double* y, cudaStream_t s) {
  const size_t N = static_cast<size_t>(n) * n * n;
  k_trig_basis<<<grid_for(N, 256), 256, 0, s>>>(tp, n, y);
  return cudaGetLastError();
}

cudaError_t launch_trig_volume(const double* y, size_t N, double mu0, double dmu, double k, double Vh,
                               double rho_min, double* part, int* grid_out, cudaStream_t s) {
  const int g = grid_for(N, 256);
  *grid_out = g;
  k_trig_volume<<<g, 256, 0, s>>>(y, N, mu0, dmu, k, Vh, rho_min, part);
  return cudaGetLastError();
}

cudaError_t launch_trig_project(const double* y, size_t N, double mu, double k, double Vh, double rho_min,
                                float* rho, cudaStream_t s) {
  k_trig_project<<<grid_for(N, 256), 256, 0, s>>>(y, N, mu, k, Vh, rho_min, rho);
  return cudaGetLastError();
}

cudaError_t launch_symmetrize(const SymParam& sp, int n, const float* in, float* out, cudaStream_t s) {
  const size_t N = static_cast<size_t>(n) * n * n;
  k_symmetrize<<<grid_for(N, 256), 256, 0, s>>>(sp, in, out, n);
  return cudaGetLastError();
}

namespace {
// The 27-offset form's weights, or false when fp is another stencil (27 offsets are exactly the
// unit cube: the next ones, at distance 2, come six at a time with 33).
bool filter27(const FilterParam& fp, Filter27& F) {
  if (fp.count != 27) return false;
  F = {{fp.w[13], fp.w[14], fp.w[17], fp.w[26]}, fp.inv_wsum};   // centre, +x, +x+y, +x+y+z
  return true;
}
}  // namespace

cudaError_t launch_filter(const FilterParam& fp, int n, const float* in, float* out,
                          cudaStream_t s) {
  const size_t N = static_cast<size_t>(n) * n * n;
  Filter27 F;
  if (filter27(fp, F)) k_filter27<false><<<grid_for(N, 256), 256, 0, s>>>(F, n, in, nullptr, 0.f, out);
  else k_filter<false><<<grid_for(N, 256), 256, 0, s>>>(fp, n, in, nullptr, 0.f, out);
  return cudaGetLastError();
}

cudaError_t launch_sensitivity_filter(const FilterParam& fp, int n, const float* rho, const float* dc,
                                      float gamma, float* out, cudaStream_t s) {
  const size_t N = static_cast<size_t>(n) * n * n;
  Filter27 F;
  if (filter27(fp, F)) k_filter27<true><<<grid_for(N, 256), 256, 0, s>>>(F, n, dc, rho, gamma, out);
  else k_filter<true><<<grid_for(N, 256), 256, 0, s>>>(fp, n, dc, rho, gamma, out);
  return cudaGetLastError();
}

namespace {
template <int W>
cudaError_t oc_run(homo_ctx* c, const float* dc, float* rho, double volfrac, double move, double eta, double rho_min) {
  const size_t N = c->N;
  const int g = static_cast<int>(std::min<size_t>((N / W + kOcBlock - 1) / kOcBlock, kOcGrid));
  const size_t stride = static_cast<size_t>(grid_for(N, kOcBlock)) * kOcBlock;
  const int gp = std::min(grid_for(N, kOcBlock), kOcGrid);
  double* oc = c->scal + S_OC;
  cudaStream_t s = c->stream;
  const float mv = static_cast<float>(move), rm = static_cast<float>(rho_min);
  k_oc_setup<W><<<g, kOcBlock, 0, s>>>(rho, dc, c->tmp, N, static_cast<float>(eta), mv, rm, volfrac, c->part, oc);
  for (int it = 0; it < kOcPasses; ++it)
    k_oc_pass<<<gp, kOcBlock, 0, s>>>(rho, c->tmp, N, stride, mv, rm, volfrac, oc, c->part);
  k_oc_apply<W><<<g, kOcBlock, 0, s>>>(rho, c->tmp, N, mv, rm, oc, c->part);
  return cudaGetLastError();
}
}  // namespace

cudaError_t launch_oc(homo_ctx* c, const float* dc, float* rho, double volfrac, double move,
                      double eta, double rho_min, double* change) {
  double* oc = c->scal + S_OC;
  cudaStream_t s = c->stream;
  const bool vec = c->N % 4 == 0 && (reinterpret_cast<uintptr_t>(dc) | reinterpret_cast<uintptr_t>(rho)) % 16 == 0;
  cudaError_t e = vec ? oc_run<4>(c, dc, rho, volfrac, move, eta, rho_min)
                      : oc_run<1>(c, dc, rho, volfrac, move, eta, rho_min);
  if (e != cudaSuccess) return e;
  if (change) {
    e = cudaMemcpyAsync(c->hscal + S_OC + OC_CHANGE, oc + OC_CHANGE, sizeof(double),
                        cudaMemcpyDeviceToHost, s);
    if (e != cudaSuccess) return e;
    e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return e;
    *change = c->hscal[S_OC + OC_CHANGE];
  }
  return cudaSuccess;
}

}  // namespace homo
