// The finest-level 8-colour block Gauss-Seidel smoother (Eq. 15-16), two colours per launch.
#include "stencil.cuh"

namespace homo {

namespace {

// Colours 2q and 2q + 1 (the even- and odd-x vertices of the rows (y, z) of one parity) in
// one pass over memory. For every vertex v of a colour, S_v u_v = f_v - M_v with S_v = A_0
// and M_v = sum_(d != 0) A_d u_(v+d). The two colours couple only inside a row (x and x +- 1
// of the same y, z), so a block that owns whole rows updates the first colour, exchanges
// the new values through shared memory and updates the second: the values and the FMA
// order are those of two separate colour passes. reverse: the odd-x colour first.
//
// A thread owns an x pair (2i, 2i + 1). Per neighbour row it needs the pair itself (one
// 8-byte load, a warp's loads are whole lines) and one value beside it, so a sweep moves
// 4 x 112 B per vertex of u, f and E in whole sectors; a launch per colour read all of u
// eight times and touched half of every sector of f and of the written u (8 x 109 B measured).
// Of those 112 B, 9 are the first colour's old values, which are overwritten unread but share
// their sectors with the second colour's. A neighbour row's pair is loaded once per vertex of
// the pair, the second time from L1. The bound is instruction issue: about 4,260 per vertex and
// sweep, of which 1404 are the scalar FMAs, 350 per case group build the blocks A_d and about 1.7
// integer instructions go with each load; ncu at 160^3, full pass: issue active 74 %, shared/L1
// data pipe 52 %, FMA pipe 42 %, DRAM 36 %, 23 warps an SM (80 registers). One sweep, against a launch per colour: 24^3 82 -> 43 us,
// 64^3 98 -> 58 us, 256^3 3350 -> 2460 us. Measured and not adopted: plane pointers as kernel
// parameters (fewer integer instructions, 2570 us: the loads come later).
//
// first: first sweep from u = 0 in colour order 0..7: rows of a later colour pair still
// hold zero and are skipped, and so is the second colour of the own row (u need not be
// cleared beforehand).
// The load cases are split over blockIdx.y in groups of CASES (3: the blocks A_d are rebuilt
// per group, fewer registers and twice the warps; 6: built once). Every variant performs
// the same arithmetic per vertex and case in the same order, so all give bitwise the same
// result; homo_autotune picks the fastest for a grid size.

// Value(s) at a 32-bit byte offset from a plane: the plane pointer is uniform over the grid, so
// a load needs no 64-bit address arithmetic (a plane has at most 4 GB).
template <bool VEC>
__device__ __forceinline__ float2 ld_pair(const float* __restrict__ plane, unsigned off) {
  const char* p = reinterpret_cast<const char*>(plane) + off;
  if (VEC) return __ldg(reinterpret_cast<const float2*>(p));
  return make_float2(__ldg(reinterpret_cast<const float*>(p)), __ldg(reinterpret_cast<const float*>(p) + 1));
}

__device__ __forceinline__ float ld_one(const float* __restrict__ plane, unsigned off) {
  return __ldg(reinterpret_cast<const float*>(reinterpret_cast<const char*>(plane) + off));
}

// Row update of one vertex: rhs -= A_d u_(v+d) for the three d of neighbour row (dy, dz), in
// the order dx = -1, 0, 1. ODD: the vertex is the pair's odd one, so the pair is its dx = -1
// and 0 and the side value (x + 2) its dx = +1; even: side (x - 1), pair at 0 and +1.
template <int CASES, bool ODD, bool VEC>
__device__ __forceinline__ void gs_row(const KeParam& K, const float (&Et)[8], int dy, int dz,
                                       const float* __restrict__ u, size_t N, unsigned own, unsigned side,
                                       float (&rhs)[3 * CASES]) {
  float A[3][9];
#pragma unroll
  for (int dx = -1; dx <= 1; ++dx) nb_block(K, Et, dx, dy, dz, A[dx + 1]);
#pragma unroll
  for (int c = 0; c < CASES; ++c) {
    float2 o[3];
    float s[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float* uq = u + (3 * c + k) * N;
      o[k] = ld_pair<VEC>(uq, own);
      s[k] = ld_one(uq, side);
    }
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      float b = rhs[3 * c + r];
#pragma unroll
      for (int dx = 0; dx < 3; ++dx) {
        const float u0 = ODD ? (dx == 0 ? o[0].x : dx == 1 ? o[0].y : s[0]) : (dx == 0 ? s[0] : dx == 1 ? o[0].x : o[0].y);
        const float u1 = ODD ? (dx == 0 ? o[1].x : dx == 1 ? o[1].y : s[1]) : (dx == 0 ? s[1] : dx == 1 ? o[1].x : o[1].y);
        const float u2 = ODD ? (dx == 0 ? o[2].x : dx == 1 ? o[2].y : s[2]) : (dx == 0 ? s[2] : dx == 1 ? o[2].x : o[2].y);
        b = fmaf(-A[dx][3 * r + 2], u2, fmaf(-A[dx][3 * r + 1], u1, fmaf(-A[dx][3 * r], u0, b)));
      }
      rhs[3 * c + r] = b;
    }
  }
}

// The same for the vertex's own row, whose values lo (x - 1) and hi (x + 1) come from get(q, side).
template <int CASES, typename Get>
__device__ __forceinline__ void gs_own_row(const KeParam& K, const float (&Et)[8], float (&rhs)[3 * CASES], Get get) {
  float A[2][9];
  nb_block(K, Et, -1, 0, 0, A[0]);
  nb_block(K, Et, 1, 0, 0, A[1]);
#pragma unroll
  for (int c = 0; c < CASES; ++c)
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const float u0 = get(3 * c, e), u1 = get(3 * c + 1, e), u2 = get(3 * c + 2, e);
#pragma unroll
      for (int r = 0; r < 3; ++r)
        rhs[3 * c + r] =
            fmaf(-A[e][3 * r + 2], u2, fmaf(-A[e][3 * r + 1], u1, fmaf(-A[e][3 * r], u0, rhs[3 * c + r])));
    }
}

// One vertex of the pair. SECOND: the own row's neighbours were updated in this launch (read
// from shared memory: plane q of the pairs p0 and p1 at sh[q * T + p]); otherwise they are the
// other colour's old values in u. mask: bit (dy != 0) + 2 (dz != 0) set when such rows are read.
template <int CASES, bool ODD, bool SECOND, bool VEC>
__device__ __forceinline__ void gs_vertex(const KeParam& K, const float* __restrict__ E, const float* __restrict__ u,
                                          size_t N, int n, int x, int y, int z, int mask, bool skip_own,
                                          const float* sh, int T, int p0, int p1, float (&rhs)[3 * CASES]) {
  const Nb nb = make_nb(x, y, z, n);
  float Et[8];
  load_E8(E, nb, Et);
  const unsigned own = 4u * (ODD ? nb.X[0] : nb.X[1]);   // the pair's even vertex
  const unsigned side = 4u * (ODD ? nb.X[2] : nb.X[0]);
#pragma unroll
  for (int row = 0; row < 9; ++row) {
    const int dy = row % 3 - 1, dz = row / 3 - 1;
    if (row == 4) {
      if (skip_own) continue;
      if (SECOND) {
        gs_own_row<CASES>(K, Et, rhs, [&](int q, int e) { return sh[q * T + (e == 0 ? p0 : p1)]; });
      } else {
        const unsigned base = 4u * (nb.Y[1] + nb.Z[1]);
        gs_own_row<CASES>(K, Et, rhs, [&](int q, int e) { return ld_one(u + q * N, base + 4u * nb.X[2 * e]); });
      }
      continue;
    }
    if (!((mask >> ((dy != 0 ? 1 : 0) | (dz != 0 ? 2 : 0))) & 1)) continue;
    const unsigned base = 4u * (nb.Y[dy + 1] + nb.Z[dz + 1]);
    gs_row<CASES, ODD, VEC>(K, Et, dy, dz, u, N, base + own, base + side, rhs);
  }
  float S[9];
  nb_block(K, Et, 0, 0, 0, S);
  solve3xn<CASES>(S, rhs);
}

// A block holds `rows` whole rows of x pairs (thread = pair of a row). MAXT: threads at most.
// VEC: f and u are 8-byte aligned (n is even, so then every pair is); otherwise the pairs move
// as single values.
template <int CASES, int MAXT, bool REVERSE, bool VEC>
__global__ void __launch_bounds__(MAXT, MAXT == 256 ? (CASES == 3 ? 3 : 2) : 1)
    k_fine_gs(const __grid_constant__ KeParam K, const float* __restrict__ E, const float* __restrict__ f,
              float* __restrict__ u, int n, int pair, int first, const float* __restrict__ fmean, int rows) {
  extern __shared__ float sh[];                            // [3 CASES][blockDim.x], then the means
  const int T = static_cast<int>(blockDim.x), me = static_cast<int>(threadIdx.x);
  float* fm = sh + 3 * CASES * T;
  const size_t N = static_cast<size_t>(n) * n * n;
  const int h = n >> 1;
  const int cy = pair & 1, cz = pair >> 1;
  const size_t q0 = 3 * CASES * blockIdx.y;                // first plane of the case group
  f += q0 * N;
  u += q0 * N;
  if (me < 3 * CASES) fm[me] = fmean ? __ldg(fmean + q0 + me) : 0.f;
  __syncthreads();
  const int lrow = me / h, i = me - lrow * h;
  const int row = static_cast<int>(blockIdx.x) * rows + lrow;
  const bool live = lrow < rows && row < h * h;
  const int y = 2 * (row % h) + cy, z = 2 * (row / h) + cz, x = 2 * i;
  const unsigned at = 4u * (static_cast<unsigned>(x) + static_cast<unsigned>(n) * (y + static_cast<unsigned>(n) * z));
  // the first sweep from zero reads only the rows of an earlier colour pair
  int mask = 15;
  if (first) {
    mask = 0;
#pragma unroll
    for (int odd = 1; odd < 4; ++odd)
      if ((pair ^ odd) < pair) mask |= 1 << odd;
  }
  float a[3 * CASES];
  if (live) {
#pragma unroll
    for (int q = 0; q < 3 * CASES; ++q) a[q] = ld_one(f + q * N, at + (REVERSE ? 4u : 0u)) - fm[q];
    gs_vertex<CASES, REVERSE, false, VEC>(K, E, u, N, n, REVERSE ? x + 1 : x, y, z, mask, first != 0, nullptr, 0, 0, 0, a);
#pragma unroll
    for (int q = 0; q < 3 * CASES; ++q) sh[q * T + me] = a[q];
  }
  __syncthreads();
  if (!live) return;
#pragma unroll
  for (int q = 0; q < 3 * CASES; ++q) a[q] = ld_one(f + q * N, at + (REVERSE ? 0u : 4u)) - fm[q];
  // the odd vertex lies between its pair's even one and the next pair's, the even vertex
  // between the previous pair's odd one and its own
  const int p0 = REVERSE ? (i == 0 ? me + h - 1 : me - 1) : me;
  const int p1 = REVERSE ? me : (i == h - 1 ? me - (h - 1) : me + 1);
  gs_vertex<CASES, !REVERSE, true, VEC>(K, E, u, N, n, REVERSE ? x : x + 1, y, z, mask, false, sh, T, p0, p1, a);
#pragma unroll
  for (int q = 0; q < 3 * CASES; ++q) {
    const float o = sh[q * T + me];
    char* d = reinterpret_cast<char*>(u + q * N) + at;
    const float2 t = REVERSE ? make_float2(a[q], o) : make_float2(o, a[q]);
    if (VEC) {
      *reinterpret_cast<float2*>(d) = t;
    } else {
      reinterpret_cast<float*>(d)[0] = t.x;
      reinterpret_cast<float*>(d)[1] = t.y;
    }
  }
}

template <int CASES, int MAXT, bool VEC>
cudaError_t gs_launch(const homo_ctx* c, int block, int pair, int reverse, const float* f, float* u, int first,
                      const float* fmean) {
  const int h = c->n / 2;
  const int rows = h >= block ? 1 : block / h;
  const int threads = (rows * h + 31) / 32 * 32;
  const dim3 grid((h * h + rows - 1) / rows, kCases / CASES);
  const size_t shm = sizeof(float) * 3 * CASES * (threads + 1);
  if (reverse)
    k_fine_gs<CASES, MAXT, true, VEC><<<grid, threads, shm, c->stream>>>(c->ke, c->E, f, u, c->n, pair, 0, fmean, rows);
  else
    k_fine_gs<CASES, MAXT, false, VEC><<<grid, threads, shm, c->stream>>>(c->ke, c->E, f, u, c->n, pair, first, fmean, rows);
  return cudaGetLastError();
}

}  // namespace

bool gs_variant_ok(int cases, int block) { return (cases == 3 || cases == 6) && (block == 128 || block == 256); }

cudaError_t launch_fine_gs(const homo_ctx* c, int pair, int reverse, const float* f, float* u, int first,
                           const float* fmean) {
  const int b = c->gs_block;
  const bool wide = c->n > 512;   // a row of more than 256 pairs
  if ((reinterpret_cast<uintptr_t>(f) | reinterpret_cast<uintptr_t>(u)) % 8 != 0)
    return wide ? gs_launch<3, 512, false>(c, b, pair, reverse, f, u, first, fmean)
                : gs_launch<3, 256, false>(c, b, pair, reverse, f, u, first, fmean);
  if (c->gs_cases == 6)
    return wide ? gs_launch<6, 512, true>(c, b, pair, reverse, f, u, first, fmean)
                : gs_launch<6, 256, true>(c, b, pair, reverse, f, u, first, fmean);
  return wide ? gs_launch<3, 512, true>(c, b, pair, reverse, f, u, first, fmean)
              : gs_launch<3, 256, true>(c, b, pair, reverse, f, u, first, fmean);
}

}  // namespace homo
