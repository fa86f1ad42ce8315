// Coarse levels of the multigrid hierarchy (Sec. 3.3, Sec. 4.2): Galerkin stencils,
// stored-stencil relaxation and residual, trilinear transfers and the direct coarsest
// solve with the rigid-translation null space projected out.
#include "stencil.cuh"

#include <algorithm>
#include <iterator>
#include <mutex>

namespace homo {

namespace {

struct BfParam {
  float b[8 * 576];   // B_f = P_f^T K0 P_f for the 8 fine elements of a coarse element
};

// Level-1 stencil from the fine moduli (Eq. 17-18, grouped per coarse element): the
// coarse element with origin O has matrix sum_f E[2O + f] B_f; vertex V is local vertex
// 7 - t of its incident coarse element t, and local vertex J of that element is the
// neighbour V + bits(t) + bits(J) - 1. One thread per coarse vertex.
__global__ void __launch_bounds__(128) k_level1(const __grid_constant__ BfParam B,
                                                const float* __restrict__ E, int nf,
                                                float* __restrict__ st, int nc, bool cb) {
  const size_t Nc = static_cast<size_t>(nc) * nc * nc;
  for (size_t p = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; p < Nc;
       p += static_cast<size_t>(gridDim.x) * blockDim.x) {
    int X, Y, Z;
    vertex_of_pos(p, nc, cb, X, Y, Z);
    // fine elements of the 4x4x4 box with origin 2V - (2,2,2)
    float Eb[64];
    int ix[4], iy[4], iz[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      ix[a] = ((2 * X - 2 + a) % nf + nf) % nf;
      iy[a] = (((2 * Y - 2 + a) % nf + nf) % nf) * nf;
      iz[a] = (((2 * Z - 2 + a) % nf + nf) % nf) * nf * nf;
    }
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
      for (int b = 0; b < 4; ++b)
#pragma unroll
        for (int a = 0; a < 4; ++a) Eb[a + 4 * b + 16 * c] = __ldg(E + ix[a] + iy[b] + iz[c]);
#pragma unroll 1
    for (int d = 0; d < 27; ++d) {
      const int dx = d % 3 - 1, dy = (d / 3) % 3 - 1, dz = d / 9 - 1;
      float A[9];
#pragma unroll
      for (int q = 0; q < 9; ++q) A[q] = 0.f;
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        const int ta = t & 1, tb = (t >> 1) & 1, tc = t >> 2;
        const int Ja = dx + 1 - ta, Jb = dy + 1 - tb, Jc = dz + 1 - tc;
        if (Ja < 0 || Ja > 1 || Jb < 0 || Jb > 1 || Jc < 0 || Jc > 1) continue;
        const int J = Ja + 2 * Jb + 4 * Jc, row = 7 - t;
#pragma unroll
        for (int f = 0; f < 8; ++f) {
          const float Ef = Eb[(2 * ta + (f & 1)) + 4 * (2 * tb + ((f >> 1) & 1)) + 16 * (2 * tc + (f >> 2))];
#pragma unroll
          for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int c = 0; c < 3; ++c)
              A[3 * r + c] = fmaf(Ef, B.b[f * 576 + (3 * row + r) * 24 + 3 * J + c], A[3 * r + c]);
        }
      }
#pragma unroll
      for (int q = 0; q < 9; ++q) st[static_cast<size_t>(9 * d + q) * Nc + p] = A[q];
    }
  }
}

// One axis of the Galerkin product R K I (Eq. 17-18 on coarse levels). The trilinear
// transfers are tensor products of the 1-D linear interpolation, so R K I factors into
// three one-axis coarsenings, each a 27-point block stencil again. Coarsening axis `ax`
// of a stencil S on an (mx, my, mz) grid: for output vertex V and output offset d,
//   S'(V, d) = sum over a, e in {-1,0,1} with |2 d_ax + e - a| <= 1 of
//              w(a) w(e) S(V with x_ax -> 2 V_ax + a, d with d_ax -> 2 d_ax + e - a),
// w(t) = 1 - |t|/2: 7 pairs when d_ax = 0, 3 when d_ax = +-1. src_cb / dst_cb: the grid
// is cubic and its stencil planes are colour-blocked (a level's own layout); otherwise
// x-fastest. Thread per (d, output vertex).
template <int ax>
__global__ void __launch_bounds__(256) k_galerkin_axis(const float* __restrict__ src, int mx, int my, int mz,
                                                       bool src_cb, float* __restrict__ dst, bool dst_cb) {
  const int ox = ax == 0 ? mx / 2 : mx, oy = ax == 1 ? my / 2 : my, oz = ax == 2 ? mz / 2 : mz;
  const size_t Nin = static_cast<size_t>(mx) * my * mz;
  const size_t Nout = static_cast<size_t>(ox) * oy * oz;
  const size_t total = 27 * Nout;
  for (size_t it = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; it < total;
       it += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const int d = static_cast<int>(it / Nout);
    const size_t p = it - static_cast<size_t>(d) * Nout;
    int V[3];
    if (dst_cb) {
      vertex_of_pos(p, ox, true, V[0], V[1], V[2]);
    } else {
      const unsigned q = static_cast<unsigned>(p) / static_cast<unsigned>(ox);
      V[0] = static_cast<int>(static_cast<unsigned>(p) - q * static_cast<unsigned>(ox));
      V[2] = static_cast<int>(q / static_cast<unsigned>(oy));
      V[1] = static_cast<int>(q - static_cast<unsigned>(V[2]) * static_cast<unsigned>(oy));
    }
    const int D[3] = {d % 3 - 1, (d / 3) % 3 - 1, d / 9 - 1};
    const int m_ax = ax == 0 ? mx : (ax == 1 ? my : mz);
    float A[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) A[q] = 0.f;
#pragma unroll
    for (int a = -1; a <= 1; ++a) {
      int F[3] = {V[0], V[1], V[2]};
      int fa = 2 * V[ax] + a;
      fa = fa < 0 ? fa + m_ax : (fa >= m_ax ? fa - m_ax : fa);
      F[ax] = fa;
      const size_t pin = src_cb ? stencil_pos(F[0], F[1], F[2], mx, true)
                                : static_cast<size_t>(F[0]) + static_cast<size_t>(mx) *
                                      (F[1] + static_cast<size_t>(my) * F[2]);
      const float wa = a ? 0.5f : 1.f;
#pragma unroll
      for (int e = -1; e <= 1; ++e) {
        const int bax = 2 * D[ax] + e - a;
        if (bax < -1 || bax > 1) continue;
        int B[3] = {D[0], D[1], D[2]};
        B[ax] = bax;
        const int dd = (B[0] + 1) + 3 * (B[1] + 1) + 9 * (B[2] + 1);
        const float ww = wa * (e ? 0.5f : 1.f);
#pragma unroll
        for (int q = 0; q < 9; ++q) A[q] = fmaf(ww, __ldg(src + static_cast<size_t>(9 * dd + q) * Nin + pin), A[q]);
      }
    }
#pragma unroll
    for (int q = 0; q < 9; ++q) dst[static_cast<size_t>(9 * d + q) * Nout + p] = A[q];   // p: output position
  }
}

// Stencil entry as FP32 from FP32 or BF16 storage.
__device__ __forceinline__ float ld_st(const float* p) { return __ldg(p); }
__device__ __forceinline__ float ld_st(const __nv_bfloat16* p) { return __bfloat162float(__ldg(p)); }

__device__ __forceinline__ float st_f32(float v) { return v; }
__device__ __forceinline__ float st_f32(__nv_bfloat16 v) { return __bfloat162float(v); }

// Mixed precision: st16 = BF16 of (A_d(v) + A_-d(v+d)^T) / 2 for every vertex v and
// neighbour d. Both partners of a pair are formed from the same two FP32 blocks (FP32
// addition commutes and the halving is exact), so the rounded operator is exactly
// symmetric. Thread per (d, position); writes the BF16 plane layout of st.
__global__ void __launch_bounds__(256) k_stencil_bf16(const float* __restrict__ st, int n, bool cb,
                                                      __nv_bfloat16* __restrict__ st16) {
  const size_t N = static_cast<size_t>(n) * n * n;
  const size_t total = 27 * N;
  for (size_t it = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; it < total;
       it += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const int d = static_cast<int>(it / N);
    const size_t p = it - static_cast<size_t>(d) * N;
    int X, Y, Z;
    vertex_of_pos(p, n, cb, X, Y, Z);
    const int dx = d % 3 - 1, dy = (d / 3) % 3 - 1, dz = d / 9 - 1;
    const int Xn = (X + dx + n) % n, Yn = (Y + dy + n) % n, Zn = (Z + dz + n) % n;
    const size_t pn = stencil_pos(Xn, Yn, Zn, n, cb);
    const int dm = 26 - d;                      // offset -d seen from the neighbour
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const float a = st[static_cast<size_t>(9 * d + 3 * r + c) * N + p];
        const float b = st[static_cast<size_t>(9 * dm + 3 * c + r) * N + pn];
        st16[static_cast<size_t>(9 * d + 3 * r + c) * N + p] = __float2bfloat16_rn(0.5f * (a + b));
      }
  }
}

// LDL^T factors of the symmetric 3x3 diagonal block S_v (Eq. 16): multipliers l10, l20,
// l21 and the reciprocal pivots i0, i1, i2.
struct Factor3 {
  float l10, l20, l21, i0, i1, i2;
};

__device__ __forceinline__ Factor3 factor3(const float (&S)[9]) {
  Factor3 F;
  const float d0 = S[0];
  F.l10 = S[3] / d0;
  F.l20 = S[6] / d0;
  const float d1 = S[4] - F.l10 * S[1];
  F.l21 = (S[7] - F.l20 * S[1]) / d1;
  const float d2 = S[8] - F.l20 * S[2] - F.l21 * (S[5] - F.l10 * S[2]);
  F.i0 = 1.f / d0;
  F.i1 = 1.f / d1;
  F.i2 = 1.f / d2;
  return F;
}

// Solve S_v x = (y0, y1, y2) in place for one load case.
__device__ __forceinline__ void solve3(const Factor3& F, float& y0, float& y1, float& y2) {
  y1 -= F.l10 * y0;
  y2 -= F.l20 * y0 + F.l21 * y1;
  const float x2 = y2 * F.i2;
  const float x1 = y1 * F.i1 - F.l21 * x2;
  const float x0 = y0 * F.i0 - F.l10 * x1 - F.l20 * x2;
  y0 = x0;
  y1 = x1;
  y2 = x2;
}

__device__ __forceinline__ void solve3x6c(const float (&S)[9], float (&b)[18]) {
  const Factor3 F = factor3(S);
#pragma unroll
  for (int c = 0; c < kCases; ++c) solve3(F, b[3 * c], b[3 * c + 1], b[3 * c + 2]);
}

// One colour pass of block Gauss-Seidel (Eq. 15-16) with the stored stencil. Neighbours
// have other colours and are not written during the pass. first != 0: first sweep from
// x = 0 in colour order 0..7 (higher-colour neighbours are still zero and skipped).
template <typename T>
__global__ void __launch_bounds__(256) k_coarse_gs(const T* __restrict__ st,
                                                   const float* __restrict__ f,
                                                   float* __restrict__ x, int n, int colour,
                                                   int first) {
  const size_t N = static_cast<size_t>(n) * n * n;
  const int h = n >> 1;
  const size_t Nh = static_cast<size_t>(h) * h * h;
  const int cx = colour & 1, cy = (colour >> 1) & 1, cz = colour >> 2;
  for (size_t m = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; m < Nh;
       m += static_cast<size_t>(gridDim.x) * blockDim.x) {
    int i, j, k;
    decode3(static_cast<unsigned>(m), static_cast<unsigned>(h), i, j, k);
    const int X = 2 * i + cx, Y = 2 * j + cy, Z = 2 * k + cz;
    const size_t p = static_cast<size_t>(colour) * Nh + m;
    const size_t v = static_cast<size_t>(X) + static_cast<size_t>(n) * (Y + static_cast<size_t>(n) * Z);
    const Nb nb = make_nb(X, Y, Z, n);
    float rhs[kPlanes];
#pragma unroll
    for (int q = 0; q < kPlanes; ++q) rhs[q] = __ldg(f + q * N + v);
    float S[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) S[q] = ld_st(st + static_cast<size_t>(9 * 13 + q) * N + p);
#pragma unroll
    for (int d = 0; d < 27; ++d) {
      if (d == 13) continue;
      const int dx = d % 3 - 1, dy = (d / 3) % 3 - 1, dz = d / 9 - 1;
      const int odd = (dx != 0) | ((dy != 0) << 1) | ((dz != 0) << 2);
      if (first && (colour ^ odd) > colour) continue;
      float A[9];
#pragma unroll
      for (int q = 0; q < 9; ++q) A[q] = ld_st(st + static_cast<size_t>(9 * d + q) * N + p);
      const size_t w = static_cast<size_t>(nb.X[dx + 1] + nb.Y[dy + 1] + nb.Z[dz + 1]);
      const float* xr = x;
#pragma unroll
      for (int c = 0; c < kCases; ++c) {
        const float u0 = __ldg(xr + (3 * c) * N + w), u1 = __ldg(xr + (3 * c + 1) * N + w),
                    u2 = __ldg(xr + (3 * c + 2) * N + w);
#pragma unroll
        for (int r = 0; r < 3; ++r)
          rhs[3 * c + r] = fmaf(-A[3 * r + 2], u2, fmaf(-A[3 * r + 1], u1, fmaf(-A[3 * r], u0, rhs[3 * c + r])));
      }
    }
    solve3x6c(S, rhs);
#pragma unroll
    for (int q = 0; q < kPlanes; ++q) x[q * N + v] = rhs[q];
  }
}

// One load case of one vertex of a block Gauss-Seidel colour pass (Eq. 15-16): exactly
// the arithmetic of that case in k_coarse_gs (the same FMAs in the same order, the same
// factorisation and solve), so it produces bitwise the same value. The 26 neighbours are
// visited in three z-layers of 9 (d = 0..8, 9..17, 18..26, the order of the FMA chain);
// the 108 stencil and displacement values of a layer are loaded before its FMAs, so a
// thread waits for three rounds of loads instead of one per neighbour (the small coarse
// levels are bound by that latency). COHERENT: x is read through L2 only, for kernels in
// which other CTAs write x between colour passes; otherwise through the read-only path
// (a pass reads only vertices of other colours, which it does not write).
template <typename T, bool COHERENT>
__device__ __forceinline__ void gs_item(const T* __restrict__ st, const float* __restrict__ f, float* x,
                                        int n, size_t N, unsigned Nh, int h, int colour, int fz, int c,
                                        unsigned m) {
  const int cx = colour & 1, cy = (colour >> 1) & 1, cz = colour >> 2;
  int i, j, kk;
  decode3(m, static_cast<unsigned>(h), i, j, kk);
  const int X = 2 * i + cx, Y = 2 * j + cy, Z = 2 * kk + cz;
  const size_t p = static_cast<size_t>(colour) * Nh + m;
  const size_t v = static_cast<size_t>(X) + static_cast<size_t>(n) * (Y + static_cast<size_t>(n) * Z);
  const Nb nb = make_nb(X, Y, Z, n);
  const float* fc = f + static_cast<size_t>(3 * c) * N;
  const float* xc = x + static_cast<size_t>(3 * c) * N;
  float b0 = __ldg(fc + v), b1 = __ldg(fc + N + v), b2 = __ldg(fc + 2 * N + v);
  float S[9];
#pragma unroll
  for (int layer = 0; layer < 3; ++layer) {
    float A[9][9], U[9][3];
#pragma unroll
    for (int e = 0; e < 9; ++e) {
      const int d = 9 * layer + e;
      const int dx = d % 3 - 1, dy = (d / 3) % 3 - 1, dz = d / 9 - 1;
      const int odd = (dx != 0) | ((dy != 0) << 1) | ((dz != 0) << 2);
      if (d == 13) {
#pragma unroll
        for (int q = 0; q < 9; ++q) S[q] = ld_st(st + static_cast<size_t>(9 * 13 + q) * N + p);
        continue;
      }
      if (fz && (colour ^ odd) > colour) continue;
#pragma unroll
      for (int q = 0; q < 9; ++q) A[e][q] = ld_st(st + static_cast<size_t>(9 * d + q) * N + p);
      const size_t w = static_cast<size_t>(nb.X[dx + 1] + nb.Y[dy + 1] + nb.Z[dz + 1]);
      if (COHERENT) {
        U[e][0] = __ldcg(xc + w);
        U[e][1] = __ldcg(xc + N + w);
        U[e][2] = __ldcg(xc + 2 * N + w);
      } else {
        U[e][0] = __ldg(xc + w);
        U[e][1] = __ldg(xc + N + w);
        U[e][2] = __ldg(xc + 2 * N + w);
      }
    }
#pragma unroll
    for (int e = 0; e < 9; ++e) {
      const int d = 9 * layer + e;
      const int dx = d % 3 - 1, dy = (d / 3) % 3 - 1, dz = d / 9 - 1;
      const int odd = (dx != 0) | ((dy != 0) << 1) | ((dz != 0) << 2);
      if (d == 13 || (fz && (colour ^ odd) > colour)) continue;
      const float u0 = U[e][0], u1 = U[e][1], u2 = U[e][2];
      b0 = fmaf(-A[e][2], u2, fmaf(-A[e][1], u1, fmaf(-A[e][0], u0, b0)));
      b1 = fmaf(-A[e][5], u2, fmaf(-A[e][4], u1, fmaf(-A[e][3], u0, b1)));
      b2 = fmaf(-A[e][8], u2, fmaf(-A[e][7], u1, fmaf(-A[e][6], u0, b2)));
    }
  }
  solve3(factor3(S), b0, b1, b2);
  float* xo = x + static_cast<size_t>(3 * c) * N + v;
  if (COHERENT) {
    __stcg(xo, b0);
    __stcg(xo + N, b1);
    __stcg(xo + 2 * N, b2);
  } else {
    xo[0] = b0;
    xo[N] = b1;
    xo[2 * N] = b2;
  }
}

// Work items of a colour pass: one warp per (32 consecutive vertices of the colour, load
// case), the six case warps of a vertex block adjacent, so that a 192-thread CTA covers
// all six cases of its 32 vertices (their stencil rows are shared through L1) and every
// warp's loads are coalesced along the vertex index. Returns false for the padding lanes
// beyond the last vertex.
constexpr int kItemBlock = 192;

__device__ __forceinline__ bool gs_item_index(unsigned it, unsigned Nh, int& c, unsigned& m) {
  const unsigned g = it >> 5;
  const unsigned mb = g / kCases;
  c = static_cast<int>(g - mb * kCases);
  m = mb * 32 + (it & 31);
  return m < Nh;
}

__host__ __device__ inline unsigned gs_items(unsigned Nh) { return (Nh + 31) / 32 * 32 * kCases; }

// One colour pass with a thread per (load case, vertex of the colour): six times the
// threads of k_coarse_gs, each with a sixth of its FMAs and its loads in flight a z-layer
// at a time.
template <typename T>
__global__ void __launch_bounds__(kItemBlock) k_coarse_gs_item(const T* __restrict__ st,
                                                               const float* __restrict__ f, float* x,
                                                               int n, int colour, int first) {
  const size_t N = static_cast<size_t>(n) * n * n;
  const int h = n >> 1;
  const unsigned Nh = static_cast<unsigned>(h) * h * h;
  const unsigned items = gs_items(Nh);
  for (unsigned it = blockIdx.x * blockDim.x + threadIdx.x; it < items; it += gridDim.x * blockDim.x) {
    int c;
    unsigned m;
    if (gs_item_index(it, Nh, c, m)) gs_item<T, false>(st, f, x, n, N, Nh, h, colour, first, c, m);
  }
}

// ---- colour pass with the stencil staged in shared memory
// A CTA takes VERTS consecutive vertices of a colour and all six cases, CASES per thread. The
// 243 stencil values of its vertices arrive by 16-byte asynchronous copies, three z-layers
// as three groups, so that a layer computes while the next ones are in flight: the forms
// above it keep at most a neighbour's or a layer's values in flight per thread, and the
// thread-per-(vertex, case) form loads every stencil value six times. What is left are the
// neighbour values (stride 2 along x) and, per case group, the stencil's shared-memory reads.
// chained: the launch before in the stream is the colour pass before (programmatic dependent
// launch): the copies start while that pass still runs, and only then does the kernel wait
// for its results. The stencil was complete before the first, unchained pass of a chain.
// Arithmetic and order are gs_item's: bitwise the iterates of the other forms.
// Needs 16-byte aligned stencil rows: n a multiple of 4. One sweep with BF16 stencils, against
// the L2 cluster form at 32^3 and the thread-per-vertex form above: 32^3 75 -> 36 us, 64^3
// 216 -> 102 us, 128^3 885 -> 584 us; a 64^3 FP32 V-cycle 613 -> 508 us.
// Start the copies of VERTS vertices' rows (positions m0 .. of the colour) into A[243][VERTS], a
// commit group per z-layer.
template <typename T, int CASES, int VERTS>
__device__ __forceinline__ void stage_stencil(const T* __restrict__ st, size_t N, unsigned Nh, int colour, unsigned m0,
                                              T* A) {
  constexpr int kPer = 16 / static_cast<int>(sizeof(T)), kRowChunks = VERTS / kPer, kLayer = 81;
  constexpr int kTileThreads = VERTS * kCases / CASES;
  const T* src = st + static_cast<size_t>(colour) * Nh + m0;
#pragma unroll 1
  for (int layer = 0; layer < 3; ++layer) {
    for (int t = threadIdx.x; t < kLayer * kRowChunks; t += kTileThreads) {
      const int row = layer * kLayer + t / kRowChunks, c = t % kRowChunks * kPer;
      if (m0 + c < Nh)   // Nh is a multiple of kPer: a chunk is inside or outside
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(
                         static_cast<unsigned>(__cvta_generic_to_shared(A + row * VERTS + c))),
                     "l"(src + static_cast<size_t>(row) * N + c)
                     : "memory");
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  }
}

// The layer's rows are in shared memory for the whole block.
__device__ __forceinline__ void stage_wait(int layer) {
  if (layer == 0) asm volatile("cp.async.wait_group 2;\n" ::: "memory");
  else if (layer == 1) asm volatile("cp.async.wait_group 1;\n" ::: "memory");
  else asm volatile("cp.async.wait_group 0;\n" ::: "memory");
  __syncthreads();
}

template <typename T, int CASES, int VERTS>
__global__ void __launch_bounds__(VERTS * kCases / CASES)
    k_coarse_gs_tile(const T* __restrict__ st, const float* __restrict__ f, float* x, int n, int colour, int fz,
                     int chained) {
  extern __shared__ __align__(16) unsigned char tile_smem[];
  T* A = reinterpret_cast<T*>(tile_smem);                   // [243][VERTS]
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const size_t N = static_cast<size_t>(n) * n * n;
  const int h = n >> 1;
  const unsigned Nh = static_cast<unsigned>(h) * h * h;
  const unsigned m0 = blockIdx.x * VERTS;
  stage_stencil<T, CASES, VERTS>(st, N, Nh, colour, m0, A);
  if (chained) asm volatile("griddepcontrol.wait;" ::: "memory");
  const int j = static_cast<int>(threadIdx.x) % VERTS;
  const int c0 = static_cast<int>(threadIdx.x) / VERTS * CASES;
  const unsigned m = m0 + j;
  const bool live = m < Nh;
  int i, jj, kk;
  decode3(live ? m : 0u, static_cast<unsigned>(h), i, jj, kk);
  const int X = 2 * i + (colour & 1), Y = 2 * jj + ((colour >> 1) & 1), Z = 2 * kk + (colour >> 2);
  const Nb nb = make_nb(X, Y, Z, n);
  const size_t v = static_cast<size_t>(X) + static_cast<size_t>(n) * (Y + static_cast<size_t>(n) * Z);
  const float* fc = f + static_cast<size_t>(3 * c0) * N + v;
  const float* xc = x + static_cast<size_t>(3 * c0) * N;   // plain loads: the pass before wrote it
  float b[3 * CASES];
#pragma unroll
  for (int q = 0; q < 3 * CASES; ++q) b[q] = __ldg(fc + q * N);
  float S[9];
#pragma unroll
  for (int layer = 0; layer < 3; ++layer) {
    float U[9][3 * CASES];
#pragma unroll
    for (int e = 0; e < 9; ++e) {
      const int d = 9 * layer + e;
      const int odd = (d % 3 != 1) | (((d / 3) % 3 != 1) << 1) | ((d / 9 != 1) << 2);
      if (d == 13 || (fz && (colour ^ odd) > colour)) continue;
      const float* xw = xc + (nb.X[d % 3] + nb.Y[(d / 3) % 3] + nb.Z[d / 9]);
#pragma unroll
      for (int q = 0; q < 3 * CASES; ++q) U[e][q] = xw[q * N];
    }
    stage_wait(layer);
    const T* Al = A + layer * 81 * VERTS + j;
#pragma unroll
    for (int e = 0; e < 9; ++e) {
      const int d = 9 * layer + e;
      const int odd = (d % 3 != 1) | (((d / 3) % 3 != 1) << 1) | ((d / 9 != 1) << 2);
      if (d == 13) {
#pragma unroll
        for (int q = 0; q < 9; ++q) S[q] = st_f32(Al[(9 * e + q) * VERTS]);
        continue;
      }
      if (fz && (colour ^ odd) > colour) continue;
      float a[9];
#pragma unroll
      for (int q = 0; q < 9; ++q) a[q] = st_f32(Al[(9 * e + q) * VERTS]);
#pragma unroll
      for (int c = 0; c < CASES; ++c)
#pragma unroll
        for (int r = 0; r < 3; ++r)
          b[3 * c + r] = fmaf(-a[3 * r + 2], U[e][3 * c + 2],
                              fmaf(-a[3 * r + 1], U[e][3 * c + 1], fmaf(-a[3 * r], U[e][3 * c], b[3 * c + r])));
    }
  }
  if (!live) return;
  const Factor3 F = factor3(S);
#pragma unroll
  for (int c = 0; c < CASES; ++c) {
    solve3(F, b[3 * c], b[3 * c + 1], b[3 * c + 2]);
#pragma unroll
    for (int r = 0; r < 3; ++r) x[static_cast<size_t>(3 * (c0 + c) + r) * N + v] = b[3 * c + r];
  }
}

// Every sweep of one smoothing phase on a small level in one launch. Gauss-Seidel does
// not couple the load cases, so the grid is six thread-block clusters of csize CTAs, one
// per case, that never wait on one another: a cluster's colour passes are separated by
// its own hardware barrier (release at arrival, acquire at the wait, cluster scope), so a
// pass sees every value the passes before it wrote; x is read and written through L2.
// Spreading the cases over six clusters puts six times as many SMs on the small levels,
// whose passes are bound by load latency and load issue. Items as in k_coarse_gs_item
// (gs_item per vertex and case), so the iterates are bitwise those of the per-colour
// launches. sweeps >= 1; reverse: colours 7..0; first: the first sweep starts from x = 0
// (forward order only, as in k_coarse_gs).
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

constexpr int kClusterBlock = 256;

template <typename T>
__global__ void __launch_bounds__(kClusterBlock) k_coarse_gs_cluster(const T* __restrict__ st,
                                                                     const float* __restrict__ f,
                                                                     float* x, int n, int sweeps,
                                                                     int reverse, int first, int csize) {
  const size_t N = static_cast<size_t>(n) * n * n;
  const int h = n >> 1;
  const unsigned Nh = static_cast<unsigned>(h) * h * h;
  const int c = static_cast<int>(blockIdx.x) / csize;   // load case of this cluster
  const unsigned nthreads = static_cast<unsigned>(csize) * blockDim.x;
  const unsigned tid = (blockIdx.x - static_cast<unsigned>(c * csize)) * blockDim.x + threadIdx.x;
  for (int s = 0; s < sweeps; ++s) {
    const int fz = first && s == 0 && !reverse ? 1 : 0;
    for (int k = 0; k < 8; ++k) {
      const int colour = reverse ? 7 - k : k;
      for (unsigned m = tid; m < Nh; m += nthreads) gs_item<T, true>(st, f, x, n, N, Nh, h, colour, fz, c, m);
      cluster_barrier();
    }
  }
}

// ---- on-chip form of the small-level smoother
// Six clusters again, one per load case; CTA `rank` of a cluster owns positions
// [rank Mper, (rank + 1) Mper) of every colour. Everything a phase reads twice stays on the
// chip: each CTA keeps a copy of its case's displacement in shared memory (16 bytes per
// vertex, colour by colour, so that a quarter warp's neighbour loads are one conflict-free
// 128-byte line), and the stencil rows of its own vertices in registers, one block row of
// one vertex (26 x 3 values) per thread and colour. A pass is then the 78-FMA chain of a
// row on register and shared-memory operands, three shuffles that gather the vertex's
// rows, the solve with factors made once per phase, one 16-byte store per CTA that reads
// the vertex, and the cluster barrier: bound by that chain and the barrier, not by loads.
// kRegColours colour groups of threads: with 8 (Mper <= 16) a group serves one colour; with
// 4 (Mper <= 32) it serves colours g and g + 4, the second one's rows in shared memory (the
// registers hold 512 x 78 values, half of what 32 vertices of 8 colours need).
// Warps of a group: 8 vertices each, lane = 8 row + vertex (lanes 24..31 idle).
// The arithmetic per vertex is gs_item's, on the same values in the same order (the first
// sweep from zero multiplies the zeros it skips elsewhere): bitwise the same iterates.
// Against streaming each pass's rows through shared memory (three threads per vertex, one pass
// 3.0 / 3.7 us at 8^3 / 16^3, the copies' issue and waits): one
// sweep at 16^3 / 8^3, launch and setup included, 45.2 / 30.9 -> 22.7 / 16.9 us,
// the coarse smoothing of a 64^3 V-cycle 810 -> 340 us, of a mixed 256^3 one 16.1 -> 5.3 ms.
constexpr int kResThreads = 512;
constexpr int kResRow = 84;       // floats per stored row: 78 rounded up, quarter warps on distinct banks
constexpr int kResTargets = 6;    // a lane's share (a third) of at most 16 CTAs

__device__ __forceinline__ unsigned smem_addr(const void* p) {
  return static_cast<unsigned>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

// address of the same shared-memory location in CTA `rank` of the cluster
__device__ __forceinline__ unsigned map_rank(unsigned local, unsigned rank) {
  unsigned remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(rank));
  return remote;
}

// Dynamic shared memory: displacement (4 N floats), factors (8 colours x Mper x 8 floats) and,
// with 4 colour groups, the rows of colours 4..7.
__host__ __device__ inline size_t resident_smem_bytes(size_t N, int Mper, int groups) {
  return sizeof(float) * (4 * N + 64 * static_cast<size_t>(Mper) +
                          (groups == 4 ? static_cast<size_t>(4) * Mper * 3 * kResRow : 0));
}

// Index parts of the neighbours of half-grid position (i, j, k) of a colour in the
// colour-blocked displacement: neighbour d sits at X[dx + 1] + Y[dy + 1] + Z[dz + 1].
struct ResNb {
  int X[3], Y[3], Z[3];
};

__device__ __forceinline__ ResNb res_nb(unsigned m, int colour, int h, int Nh) {
  int i, j, k;
  decode3(m, static_cast<unsigned>(h), i, j, k);
  const int cx = colour & 1, cy = (colour >> 1) & 1, cz = colour >> 2;
  ResNb nb;
  // an even coordinate 2i has neighbours 2(i-1)+1 and 2i+1, an odd one 2i+1 has 2i and 2(i+1)
  auto lo = [h](int a, int odd) { return odd ? a : (a == 0 ? h - 1 : a - 1); };
  auto hi = [h](int a, int odd) { return odd ? (a == h - 1 ? 0 : a + 1) : a; };
  nb.X[1] = cx * Nh + i;
  nb.X[0] = (1 - cx) * Nh + lo(i, cx);
  nb.X[2] = (1 - cx) * Nh + hi(i, cx);
  nb.Y[1] = 2 * cy * Nh + h * j;
  nb.Y[0] = 2 * (1 - cy) * Nh + h * lo(j, cy);
  nb.Y[2] = 2 * (1 - cy) * Nh + h * hi(j, cy);
  nb.Z[1] = 4 * cz * Nh + h * h * k;
  nb.Z[0] = 4 * (1 - cz) * Nh + h * h * lo(k, cz);
  nb.Z[2] = 4 * (1 - cz) * Nh + h * h * hi(k, cz);
  return nb;
}

// b minus the off-diagonal part of one block row: the FMA chain of the row, in the order of
// every other form. row(e) is neighbour e's three values (e = 0..25, the diagonal skipped).
template <typename Row>
__device__ __forceinline__ float res_chain(float b, const float4* us, const ResNb& nb, Row row) {
#pragma unroll
  for (int d = 0; d < 27; ++d) {
    if (d == 13) continue;
    const int e = d < 13 ? d : d - 1;
    const float4 u = us[nb.X[d % 3] + nb.Y[(d / 3) % 3] + nb.Z[d / 9]];
    b = fmaf(-row(3 * e + 2), u.z, fmaf(-row(3 * e + 1), u.y, fmaf(-row(3 * e), u.x, b)));
  }
  return b;
}

// Where a resident smoother's rows come from: load(colour, position m, r, row, S) gives block row
// r of the 26 neighbour blocks (78 values, diagonal skipped) and, if S, the diagonal block.
template <typename T>
struct StoredRows {   // a coarse level's stencil
  const T* st;
  __device__ __forceinline__ float mean(int) const { return 0.f; }
  template <typename Put>
  __device__ __forceinline__ void load(int colour, unsigned m, int n, int r, Put put, float (&S)[9]) const {
    const size_t N = static_cast<size_t>(n) * n * n;
    const int h = n >> 1;
    const size_t p = static_cast<size_t>(colour) * h * h * h + m;
#pragma unroll
    for (int e = 0; e < 26; ++e)
#pragma unroll
      for (int k = 0; k < 3; ++k) put(3 * e + k, ld_st(st + static_cast<size_t>(9 * (e < 13 ? e : e + 1) + 3 * r + k) * N + p));
#pragma unroll
    for (int k = 0; k < 9; ++k) S[k] = ld_st(st + static_cast<size_t>(9 * 13 + k) * N + p);
  }
};

struct FineRows {   // the finest level: built from the moduli, as its other kernels do
  const KeParam& K;
  const float* E;
  const float* fmean;
  __device__ __forceinline__ float mean(int q) const { return fmean ? __ldg(fmean + q) : 0.f; }
  template <typename Put>
  __device__ __forceinline__ void load(int colour, unsigned m, int n, int r, Put put, float (&S)[9]) const {
    int i, j, k;
    decode3(m, static_cast<unsigned>(n >> 1), i, j, k);
    const Nb nb = make_nb(2 * i + (colour & 1), 2 * j + ((colour >> 1) & 1), 2 * k + (colour >> 2), n);
    float Et[8];
    load_E8(E, nb, Et);
#pragma unroll
    for (int d = 0; d < 27; ++d) {
      float A[9];
      nb_block(K, Et, d % 3 - 1, (d / 3) % 3 - 1, d / 9 - 1, A);
      if (d == 13) {
#pragma unroll
        for (int q = 0; q < 9; ++q) S[q] = A[q];
        continue;
      }
#pragma unroll
      for (int q = 0; q < 3; ++q) put(3 * (d < 13 ? d : d - 1) + q, r == 0 ? A[q] : (r == 1 ? A[3 + q] : A[6 + q]));
    }
  }
};

template <int kGroups, typename Rows>
__device__ __forceinline__ void gs_resident(const Rows& src, const float* __restrict__ f, float* x, int n,
                                            int sweeps, int reverse, int first, int csize, int Mper) {
  extern __shared__ __align__(16) float sm[];
  __shared__ unsigned need_s;
  constexpr int kWarps = kResThreads / 32 / kGroups;       // warps (8 vertices each) per group
  const int N = n * n * n, h = n >> 1, Nh = h * h * h;
  const int c = static_cast<int>(blockIdx.x) / csize;      // load case of this cluster
  const int rank = static_cast<int>(blockIdx.x) - c * csize;
  const int m0 = rank * Mper;
  const int mcount = m0 >= Nh ? 0 : min(Mper, Nh - m0);
  float4* us = reinterpret_cast<float4*>(sm);
  float4* fac = us + N;                                    // [8][Mper][2]: l10 l20 l21 i0 | i1 i2
  float* rows = sm + 4 * N + 64 * Mper;                    // [4][Mper][3][kResRow]
  const float* fc = f + static_cast<size_t>(3 * c) * N;
  float* xc = x + static_cast<size_t>(3 * c) * N;
  const int warp = static_cast<int>(threadIdx.x) >> 5, lane = static_cast<int>(threadIdx.x) & 31;
  const int group = warp / kWarps;
  const int r = lane >> 3, jj = lane & 7;                  // block row (3: idle) and vertex in the warp
  const int j = (warp - group * kWarps) * 8 + jj;
  const bool own = r < 3 && j < mcount;

  // displacement, colour by colour (zero where the first sweep starts from zero)
  if (threadIdx.x == 0) need_s = 0u;
  const bool from_zero = first && !reverse;
  for (int v = threadIdx.x; v < N; v += kResThreads) {
    int a, b, d;
    decode3(static_cast<unsigned>(v), static_cast<unsigned>(n), a, b, d);
    const int pos = ((a & 1) + 2 * (b & 1) + 4 * (d & 1)) * Nh + (a >> 1) + h * ((b >> 1) + h * (d >> 1));
    us[pos] = from_zero ? make_float4(0.f, 0.f, 0.f, 0.f)
                        : make_float4(__ldcg(xc + v), __ldcg(xc + N + v), __ldcg(xc + 2 * static_cast<size_t>(N) + v), 0.f);
  }
  // this thread's stencil rows and right-hand sides
  float A[78], rhs[8 / kGroups];
#pragma unroll
  for (int q = 0; q < 8 / kGroups; ++q) rhs[q] = 0.f;
#pragma unroll
  for (int e = 0; e < 78; ++e) A[e] = 0.f;
  if (own) {
    int a, b, d;
    decode3(static_cast<unsigned>(m0 + j), static_cast<unsigned>(h), a, b, d);
#pragma unroll
    for (int q = 0; q < 8 / kGroups; ++q) {
      const int colour = group + 4 * q;
      const size_t v = static_cast<size_t>(2 * a + (colour & 1)) +
                       static_cast<size_t>(n) * ((2 * b + ((colour >> 1) & 1)) + static_cast<size_t>(n) * (2 * d + (colour >> 2)));
      rhs[q] = __ldg(fc + static_cast<size_t>(r) * N + v) - src.mean(3 * c + r);
      float* dst = rows + ((static_cast<size_t>(group) * Mper + j) * 3 + r) * kResRow;
      float S[9];
      src.load(colour, static_cast<unsigned>(m0 + j), n, r, [&](int e, float val) {
        if (q == 0) A[e] = val;
        else dst[e] = val;
      }, S);
      if (r == 0) {
        const Factor3 F = factor3(S);
        fac[2 * (colour * Mper + j)] = make_float4(F.l10, F.l20, F.l21, F.i0);
        fac[2 * (colour * Mper + j) + 1] = make_float4(F.i1, F.i2, 0.f, 0.f);
      }
    }
  }
  __syncthreads();
  // the CTAs that read this one's vertices: owners of positions at most one half-grid step away
  unsigned mine = 0u;
  for (int t = threadIdx.x; t < 27 * mcount; t += kResThreads) {
    const int d = t / mcount;
    int a, b, k;
    decode3(static_cast<unsigned>(m0 + t - d * mcount), static_cast<unsigned>(h), a, b, k);
    a = (a + d % 3 - 1 + h) % h;
    b = (b + (d / 3) % 3 - 1 + h) % h;
    k = (k + d / 9 - 1 + h) % h;
    mine |= 1u << ((a + h * (b + h * k)) / Mper);
  }
  mine = __reduce_or_sync(0xffffffffu, mine);   // one atomic per warp, not one per neighbour
  if (lane == 0 && mine) atomicOr(&need_s, mine);
  __syncthreads();
  unsigned target[kResTargets];   // displacement copies this lane writes (rows split them), 0: none
#pragma unroll
  for (int q = 0; q < kResTargets; ++q) target[q] = 0u;
  {
    const unsigned need = need_s;
    const unsigned base = smem_addr(us);
    int seen = 0;
    for (int t = 0; t < csize; ++t) {
      if (!((need >> t) & 1u)) continue;
#pragma unroll
      for (int q = 0; q < kResTargets; ++q)
        if (seen == 3 * q + r) target[q] = map_rank(base, static_cast<unsigned>(t));
      ++seen;
    }
  }
  cluster_arrive();   // every copy of the displacement is complete before any owner writes into it

  const int total = sweeps * 8;
  for (int pass = 0; pass < total; ++pass) {
    const int colour = reverse ? 7 - (pass & 7) : pass & 7;
    if (colour % kGroups == group) {
      const ResNb nb = res_nb(static_cast<unsigned>(own ? m0 + j : 0), colour, h, Nh);
      const float4 f0 = fac[2 * (colour * Mper + (own ? j : 0))], f1 = fac[2 * (colour * Mper + (own ? j : 0)) + 1];
      const Factor3 F = {f0.x, f0.y, f0.z, f0.w, f1.x, f1.y};
      cluster_wait();
      float br;
      if (kGroups == 8 || colour < 4) {
        br = res_chain(rhs[0], us, nb, [&](int e) { return A[e]; });
      } else {
        const float4* row = reinterpret_cast<const float4*>(
            rows + ((static_cast<size_t>(group) * Mper + (own ? j : 0)) * 3 + (r < 3 ? r : 0)) * kResRow);
        br = res_chain(rhs[8 / kGroups - 1], us, nb, [&](int e) {
          const float4 q4 = row[e / 4];   // the compiler merges the loads of one float4
          return e % 4 == 0 ? q4.x : e % 4 == 1 ? q4.y : e % 4 == 2 ? q4.z : q4.w;
        });
      }
      float y0 = __shfl_sync(0xffffffffu, br, jj), y1 = __shfl_sync(0xffffffffu, br, 8 + jj),
            y2 = __shfl_sync(0xffffffffu, br, 16 + jj);
      solve3(F, y0, y1, y2);
      if (own) {
        const unsigned off = 16u * static_cast<unsigned>(colour * Nh + m0 + j);
#pragma unroll
        for (int q = 0; q < kResTargets; ++q)
          if (target[q])
            asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(target[q] + off), "f"(y0),
                         "f"(y1), "f"(y2), "f"(0.f)
                         : "memory");
      }
    } else {
      cluster_wait();
    }
    cluster_arrive();
  }
  cluster_wait();
  // every vertex is owned by one CTA: write the owned values back
  for (int i = threadIdx.x; i < 8 * mcount; i += kResThreads) {
    const int colour = i / mcount, q = i - colour * mcount;
    int a, b, d;
    decode3(static_cast<unsigned>(m0 + q), static_cast<unsigned>(h), a, b, d);
    const size_t v = static_cast<size_t>(2 * a + (colour & 1)) +
                     static_cast<size_t>(n) * ((2 * b + ((colour >> 1) & 1)) + static_cast<size_t>(n) * (2 * d + (colour >> 2)));
    const float4 u = us[colour * Nh + m0 + q];
    __stcg(xc + v, u.x);
    __stcg(xc + N + v, u.y);
    __stcg(xc + 2 * static_cast<size_t>(N) + v, u.z);
  }
}

template <typename T, int kGroups>
__global__ void __launch_bounds__(kResThreads, 1) k_coarse_gs_resident(const T* __restrict__ st,
                                                                     const float* __restrict__ f, float* x,
                                                                     int n, int sweeps, int reverse, int first,
                                                                     int csize, int Mper) {
  gs_resident<kGroups>(StoredRows<T>{st}, f, x, n, sweeps, reverse, first, csize, Mper);
}

// One sweep of the finest level of a cell of at most 16^3 in one launch: as many launches of
// colour pairs are all launch and load latency there (16^3: 11 us each, four a sweep).
template <int kGroups>
__global__ void __launch_bounds__(kResThreads, 1) k_fine_gs_resident(const __grid_constant__ KeParam K,
                                                                    const float* __restrict__ E,
                                                                    const float* __restrict__ f, float* x, int n,
                                                                    int reverse, int first,
                                                                    const float* __restrict__ fmean, int csize,
                                                                    int Mper) {
  gs_resident<kGroups>(FineRows{K, E, fmean}, f, x, n, 1, reverse, first, csize, Mper);
}

// out = b - K x with the stored stencil; threads walk stencil positions (coalesced).
template <typename T>
__global__ void __launch_bounds__(256) k_coarse_residual(const T* __restrict__ st,
                                                         const float* __restrict__ b,
                                                         const float* __restrict__ x,
                                                         float* __restrict__ out, int n, bool cb) {
  const size_t N = static_cast<size_t>(n) * n * n;
  // vertices in lexicographic order: x, b and out are read and written in whole sectors;
  // with colour-blocked stencils a warp's stencil reads are two contiguous runs
  for (size_t v = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; v < N;
       v += static_cast<size_t>(gridDim.x) * blockDim.x) {
    int X, Y, Z;
    decode3(static_cast<unsigned>(v), static_cast<unsigned>(n), X, Y, Z);
    const size_t p = stencil_pos(X, Y, Z, n, cb);
    const Nb nb = make_nb(X, Y, Z, n);
    float acc[kPlanes];
#pragma unroll
    for (int q = 0; q < kPlanes; ++q) acc[q] = 0.f;
#pragma unroll
    for (int d = 0; d < 27; ++d) {
      const int dx = d % 3 - 1, dy = (d / 3) % 3 - 1, dz = d / 9 - 1;
      float A[9];
#pragma unroll
      for (int q = 0; q < 9; ++q) A[q] = ld_st(st + static_cast<size_t>(9 * d + q) * N + p);
      const size_t w = static_cast<size_t>(nb.X[dx + 1] + nb.Y[dy + 1] + nb.Z[dz + 1]);
#pragma unroll
      for (int c = 0; c < kCases; ++c) {
        const float u0 = __ldg(x + (3 * c) * N + w), u1 = __ldg(x + (3 * c + 1) * N + w),
                    u2 = __ldg(x + (3 * c + 2) * N + w);
#pragma unroll
        for (int r = 0; r < 3; ++r)
          acc[3 * c + r] = fmaf(A[3 * r], u0, fmaf(A[3 * r + 1], u1, fmaf(A[3 * r + 2], u2, acc[3 * c + r])));
      }
    }
#pragma unroll
    for (int q = 0; q < kPlanes; ++q) out[q * N + v] = __ldg(b + q * N + v) - acc[q];
  }
}

// The same in the staged form of k_coarse_gs_tile (the stencil of VERTS vertices of one colour
// through shared memory, CASES load cases per thread, n a multiple of 4), with the FMA order of
// k_coarse_residual: a thread of that kernel waits for 27 neighbours one after another
// (8^3: 25 -> 6 us).
template <typename T, int CASES, int VERTS>
__global__ void __launch_bounds__(VERTS * kCases / CASES)
    k_coarse_residual_tile(const T* __restrict__ st, const float* __restrict__ bv, const float* x,
                           float* out, int n, unsigned blocks_per_colour) {
  extern __shared__ __align__(16) unsigned char tile_smem[];
  T* A = reinterpret_cast<T*>(tile_smem);                   // [243][VERTS]
  const size_t N = static_cast<size_t>(n) * n * n;
  const int h = n >> 1;
  const unsigned Nh = static_cast<unsigned>(h) * h * h;
  const int colour = static_cast<int>(blockIdx.x / blocks_per_colour);
  const unsigned m0 = (blockIdx.x - colour * blocks_per_colour) * VERTS;
  stage_stencil<T, CASES, VERTS>(st, N, Nh, colour, m0, A);
  const int j = static_cast<int>(threadIdx.x) % VERTS;
  const int c0 = static_cast<int>(threadIdx.x) / VERTS * CASES;
  const unsigned m = m0 + j;
  const bool live = m < Nh;
  int i, jj, kk;
  decode3(live ? m : 0u, static_cast<unsigned>(h), i, jj, kk);
  const int X = 2 * i + (colour & 1), Y = 2 * jj + ((colour >> 1) & 1), Z = 2 * kk + (colour >> 2);
  const Nb nb = make_nb(X, Y, Z, n);
  const size_t v = static_cast<size_t>(X) + static_cast<size_t>(n) * (Y + static_cast<size_t>(n) * Z);
  const float* xc = x + static_cast<size_t>(3 * c0) * N;
  float acc[3 * CASES], b[3 * CASES];
#pragma unroll
  for (int q = 0; q < 3 * CASES; ++q) {
    acc[q] = 0.f;
    b[q] = __ldg(bv + (3 * c0 + q) * N + v);
  }
#pragma unroll
  for (int layer = 0; layer < 3; ++layer) {
    float U[9][3 * CASES];
#pragma unroll
    for (int e = 0; e < 9; ++e) {
      const float* xw = xc + (nb.X[e % 3] + nb.Y[e / 3] + nb.Z[layer]);
#pragma unroll
      for (int q = 0; q < 3 * CASES; ++q) U[e][q] = xw[q * N];   // plain loads: kept before the barrier
    }
    stage_wait(layer);
    const T* Al = A + layer * 81 * VERTS + j;
#pragma unroll
    for (int e = 0; e < 9; ++e) {
      float a[9];
#pragma unroll
      for (int q = 0; q < 9; ++q) a[q] = st_f32(Al[(9 * e + q) * VERTS]);
#pragma unroll
      for (int c = 0; c < CASES; ++c)
#pragma unroll
        for (int r = 0; r < 3; ++r)
          acc[3 * c + r] = fmaf(a[3 * r], U[e][3 * c], fmaf(a[3 * r + 1], U[e][3 * c + 1],
                                fmaf(a[3 * r + 2], U[e][3 * c + 2], acc[3 * c + r])));
    }
  }
  if (!live) return;
#pragma unroll
  for (int q = 0; q < 3 * CASES; ++q) out[static_cast<size_t>(3 * c0 + q) * N + v] = b[q] - acc[q];
}

// Chebyshev step with the stored stencil (threads walk vertices in lexicographic order):
// mode 0: out = x_in + c0 S^-1 (b - K x_in); mode 1: out = x_in + c0 (x_in - out) +
// c1 S^-1 (b - K x_in), the previous iterate read from out and replaced in place.
// x_in == null stands for x_in = 0 (first step from zero). mode 2: out = S^-1 K x_in
// (power iteration for the largest eigenvalue of D^-1 K).
template <typename T>
__global__ void __launch_bounds__(256) k_coarse_cheb(const T* __restrict__ st,
                                                     const float* __restrict__ b,
                                                     const float* __restrict__ xin, float* out,
                                                     int n, bool cb, int mode, float c0, float c1) {
  const size_t N = static_cast<size_t>(n) * n * n;
  for (size_t v = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; v < N;
       v += static_cast<size_t>(gridDim.x) * blockDim.x) {
    int X, Y, Z;
    decode3(static_cast<unsigned>(v), static_cast<unsigned>(n), X, Y, Z);
    const size_t p = stencil_pos(X, Y, Z, n, cb);
    float acc[kPlanes];
#pragma unroll
    for (int q = 0; q < kPlanes; ++q) acc[q] = 0.f;
    if (xin) {
      const Nb nb = make_nb(X, Y, Z, n);
#pragma unroll
      for (int d = 0; d < 27; ++d) {
        const int dx = d % 3 - 1, dy = (d / 3) % 3 - 1, dz = d / 9 - 1;
        float A[9];
#pragma unroll
        for (int q = 0; q < 9; ++q) A[q] = ld_st(st + static_cast<size_t>(9 * d + q) * N + p);
        const size_t w = static_cast<size_t>(nb.X[dx + 1] + nb.Y[dy + 1] + nb.Z[dz + 1]);
#pragma unroll
        for (int c = 0; c < kCases; ++c) {
          const float u0 = __ldg(xin + (3 * c) * N + w), u1 = __ldg(xin + (3 * c + 1) * N + w),
                      u2 = __ldg(xin + (3 * c + 2) * N + w);
#pragma unroll
          for (int r = 0; r < 3; ++r)
            acc[3 * c + r] = fmaf(A[3 * r], u0, fmaf(A[3 * r + 1], u1, fmaf(A[3 * r + 2], u2, acc[3 * c + r])));
        }
      }
    }
    float S[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) S[q] = ld_st(st + static_cast<size_t>(9 * 13 + q) * N + p);
    if (mode != 2) {
#pragma unroll
      for (int q = 0; q < kPlanes; ++q) acc[q] = __ldg(b + q * N + v) - acc[q];
    }
    solve3x6c(S, acc);
#pragma unroll
    for (int q = 0; q < kPlanes; ++q) {
      const size_t o = q * N + v;
      const float xc = xin ? __ldg(xin + o) : 0.f;
      if (mode == 0) out[o] = fmaf(c0, acc[q], xc);
      else if (mode == 1) out[o] = fmaf(c1, acc[q], fmaf(c0, xc - out[o], xc));
      else if (mode == 3) out[o] = fmaf(c1, acc[q], fmaf(c0, xc, xc));   // previous iterate 0
      else out[o] = acc[q];
    }
  }
}

__global__ void k_fill_hash(float* __restrict__ x, size_t count, unsigned seed) {
  for (size_t i = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < count;
       i += static_cast<size_t>(gridDim.x) * blockDim.x) {
    unsigned h = static_cast<unsigned>(i) * 0x9E3779B1u ^ seed;
    h ^= h >> 16;
    h *= 0x85EBCA6Bu;
    h ^= h >> 13;
    h *= 0xC2B2AE35u;
    h ^= h >> 16;
    x[i] = static_cast<float>(h) * (2.f / 4294967296.f) - 1.f;
  }
}

// coarse[V] = sum over fine 2V + a, a in {-1,0,1}^3, of w(a) fine[2V + a] (R = I^T).
// Thread per (coarse vertex, load case; the case is blockIdx.y): six times the threads of one
// thread for all 18 planes, which left the small levels with a handful of warps waiting on
// 486 loads each, and a working set of 3 planes that stays in L1 on the large ones.
__global__ void __launch_bounds__(256) k_restrict(const float* __restrict__ fine, int nf,
                                                  float* __restrict__ coarse) {
  const int nc = nf / 2;
  const size_t Nf = static_cast<size_t>(nf) * nf * nf;
  const unsigned Nc = static_cast<unsigned>(nc) * nc * nc;
  fine += 3 * blockIdx.y * Nf;
  coarse += 3 * blockIdx.y * static_cast<size_t>(Nc);
  for (unsigned V = blockIdx.x * blockDim.x + threadIdx.x; V < Nc; V += gridDim.x * blockDim.x) {
    int X, Y, Z;
    decode3(V, static_cast<unsigned>(nc), X, Y, Z);
    const Nb nb = make_nb(2 * X, 2 * Y, 2 * Z, nf);
    float acc[3] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int d = 0; d < 27; ++d) {
      const int dx = d % 3 - 1, dy = (d / 3) % 3 - 1, dz = d / 9 - 1;
      const float w = (dx ? 0.5f : 1.f) * (dy ? 0.5f : 1.f) * (dz ? 0.5f : 1.f);
      const size_t o = static_cast<size_t>(nb.X[dx + 1] + nb.Y[dy + 1] + nb.Z[dz + 1]);
#pragma unroll
      for (int q = 0; q < 3; ++q) acc[q] = fmaf(w, __ldg(fine + q * Nf + o), acc[q]);
    }
#pragma unroll
    for (int q = 0; q < 3; ++q) coarse[q * static_cast<size_t>(Nc) + V] = acc[q];
  }
}

// fine (+)= I coarse. One thread per coarse cell (X..X+1, Y..Y+1, Z..Z+1) and load case
// (blockIdx.y): its 8 corner values give the 8 fine vertices (2X+a, 2Y+b, 2Z+c), a,b,c in
// {0,1}, by trilinear weights (1 on an even fine coordinate, 1/2 to each neighbour on an
// odd one). PAIRS: the two fine vertices of an x pair move as one 8-byte access (fine is
// 8-byte aligned and nf even, so every pair is); otherwise one by one.
template <bool PAIRS>
__global__ void __launch_bounds__(256) k_prolong(const float* __restrict__ coarse, int nf,
                                                 float* __restrict__ fine, int overwrite) {
  const int nc = nf / 2;
  const size_t Nf = static_cast<size_t>(nf) * nf * nf;
  const unsigned Nc = static_cast<unsigned>(nc) * nc * nc;
  coarse += 3 * blockIdx.y * static_cast<size_t>(Nc);
  fine += 3 * blockIdx.y * Nf;
  for (unsigned V = blockIdx.x * blockDim.x + threadIdx.x; V < Nc; V += gridDim.x * blockDim.x) {
    int X, Y, Z;
    decode3(V, static_cast<unsigned>(nc), X, Y, Z);
    const int X1 = X + 1 == nc ? 0 : X + 1, Y1 = Y + 1 == nc ? 0 : Y + 1, Z1 = Z + 1 == nc ? 0 : Z + 1;
    size_t cidx[8];
#pragma unroll
    for (int k = 0; k < 8; ++k)
      cidx[k] = static_cast<size_t>((k & 1) ? X1 : X) +
                static_cast<size_t>(nc) * (((k >> 1) & 1 ? Y1 : Y) + static_cast<size_t>(nc) * ((k >> 2) ? Z1 : Z));
    size_t fidx[4];
#pragma unroll
    for (int k = 0; k < 4; ++k)
      fidx[k] = static_cast<size_t>(2 * X) +
                static_cast<size_t>(nf) * ((2 * Y + (k & 1)) + static_cast<size_t>(nf) * (2 * Z + (k >> 1)));
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const float* cq = coarse + q * static_cast<size_t>(Nc);
      float c[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) c[k] = __ldg(cq + cidx[k]);
      // interpolate along x, then y, then z
      float ax[8];
#pragma unroll
      for (int k = 0; k < 8; k += 2) {
        ax[k] = c[k];
        ax[k + 1] = 0.5f * (c[k] + c[k + 1]);
      }
      float ay[8];
#pragma unroll
      for (int zc = 0; zc < 2; ++zc)
#pragma unroll
        for (int a = 0; a < 2; ++a) {
          const float lo = ax[4 * zc + a], hi = ax[4 * zc + 2 + a];
          ay[4 * zc + a] = lo;
          ay[4 * zc + 2 + a] = 0.5f * (lo + hi);
        }
      float* fq = fine + q * Nf;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int e = 2 * k;
        const float v0 = (e >> 2) ? 0.5f * (ay[e & 3] + ay[4 + (e & 3)]) : ay[e];
        const float v1 = (e >> 2) ? 0.5f * (ay[(e & 3) + 1] + ay[5 + (e & 3)]) : ay[e + 1];
        float* o = fq + fidx[k];
        if (PAIRS) {
          float2 t = overwrite ? make_float2(0.f, 0.f) : *reinterpret_cast<const float2*>(o);
          t.x = overwrite ? v0 : t.x + v0;
          t.y = overwrite ? v1 : t.y + v1;
          *reinterpret_cast<float2*>(o) = t;
        } else {
          o[0] = overwrite ? v0 : o[0] + v0;
          o[1] = overwrite ? v1 : o[1] + v1;
        }
      }
    }
  }
}

// Coarsest operator (Sec. 4.2 "eight corner vertices ... fixed"): the pinned inverse in FP64
// by Gauss-Jordan elimination without pivoting (SPD pivots are positive), blocked. Step t
// of the elimination, with c = column t and r = row t before it and ip = 1 / A[t][t], is
//   A[i][j] -= (c[i] r[j]) ip,  A[t][j] = r[j] ip,  A[i][t] = -c[i] ip,  A[t][t] = ip.
// A panel of kSw steps needs its columns, rows and diagonal block step by step, but every
// other entry only the saved c, r and ip of the panel's steps, which it applies in order:
// the same FP64 operations on the same values as the unblocked elimination, so G is bitwise
// the inverse it gives (the solution in the void regions follows a change of the
// preconditioner in its last bits). The m - 3 unknowns are padded to mp, a multiple of kSw,
// with an identity block. Per panel two launches: the panel's row and column tiles, then
// every other tile; the tile of the next diagonal block also runs that block's own steps
// (look-ahead), so no third launch stands in the chain.
// Bound by the FP64 pipe (2 per clock and SM; 2 m^3 operations) and, for small m, by the chain
// of 2 m / kSw launches. Against the one-CTA elimination over global memory it replaced
// (every step a pass over the matrix by one SM): the setup of a 16^3
// cell (m = 192) 7.1 -> 0.41 ms, of a 96^3 cell (m = 648) 254.6 -> 2.3 ms.
constexpr int kSw = 16;

__host__ __device__ inline int sweep_size(int m) { return (m - 3 + kSw - 1) / kSw * kSw; }

// Saved values of one panel: the columns' c (mp x kSw, [row][step]) and the rows' r ([column][step])
// outside the diagonal block, and the block's own c, r and ip per step.
struct SweepBuf {
  double* col;
  double* row;
  double* dcol;   // [row in block][step]
  double* drow;   // [step][column in block]
  double* ip;
};

// Dense FP64 matrix of the coarsest stencil without the 3 pinned unknowns: entry
// (3v + r - 3, 3w + c - 3) = block (v, d)[r][c], w = v + d wrapped (nc >= 3, so the 27
// neighbours are distinct). A is cleared before; the padding gets a unit diagonal.
__global__ void __launch_bounds__(256) k_coarsest_dense(const float* __restrict__ st, int nc, bool cb, int mp,
                                                        double* __restrict__ A) {
  const int Nc = nc * nc * nc, m0 = 3 * Nc - 3;
  const int gid = blockIdx.x * blockDim.x + threadIdx.x;
  for (int i = m0 + gid; i < mp; i += gridDim.x * blockDim.x) A[static_cast<size_t>(i) * mp + i] = 1.0;
  for (int it = gid; it < 27 * Nc; it += gridDim.x * blockDim.x) {
    const int d = it / Nc;
    const int v = it - d * Nc;
    const int x = v % nc, y = (v / nc) % nc, z = v / (nc * nc);
    const int xw = (x + d % 3 - 1 + nc) % nc, yw = (y + (d / 3) % 3 - 1 + nc) % nc, zw = (z + d / 9 - 1 + nc) % nc;
    const int w = xw + nc * (yw + nc * zw);
    if (v == 0 || w == 0) continue;
    const size_t p = stencil_pos(x, y, z, nc, cb);
    for (int r = 0; r < 3; ++r)
      for (int c = 0; c < 3; ++c)
        A[static_cast<size_t>(3 * v + r - 3) * mp + 3 * w + c - 3] =
            static_cast<double>(st[static_cast<size_t>(9 * d + 3 * r + c) * Nc + p]);
  }
}

// a - (c r) ip with the product rounded first, as in the elimination step above.
__device__ __forceinline__ double sweep_update(double a, double c, double r, double ip) {
  return fma(-__dmul_rn(c, r), ip, a);
}

// The kSw steps of diagonal block D (256 threads, one entry each); leaves its final values in
// D and saves the steps' c, r and ip. A pivot that is not positive sets *status.
__device__ __forceinline__ void sweep_diagonal(double (&D)[kSw][kSw + 1], double& ip_s, const SweepBuf& b,
                                               int* status) {
  const int r = threadIdx.x / kSw, c = threadIdx.x % kSw;
  for (int t = 0; t < kSw; ++t) {
    __syncthreads();
    if (threadIdx.x == 0) {
      const double piv = D[t][t];
      if (!(piv > 0.0)) *status = 1;
      ip_s = 1.0 / piv;
      b.ip[t] = ip_s;
    }
    __syncthreads();
    const double ip = ip_s, cv = D[r][t], rv = D[t][c], av = D[r][c];
    if (c == t) b.dcol[r * kSw + t] = cv;
    if (r == t) b.drow[t * kSw + c] = rv;
    // one product and one FMA in every lane: r[j] ip = fma(r[j], ip, 0), and so on
    double p = __dmul_rn(cv, rv);
    p = r == t ? (c == t ? -1.0 : -rv) : (c == t ? cv : p);
    const double val = fma(-p, ip, r == t || c == t ? 0.0 : av);
    __syncthreads();
    D[r][c] = val;
  }
  __syncthreads();
}

// Diagonal block 0 (one CTA), before the first panel.
__global__ void __launch_bounds__(kSw * kSw) k_coarsest_first(double* __restrict__ A, int mp, SweepBuf b,
                                                             int* __restrict__ status) {
  __shared__ double D[kSw][kSw + 1];
  __shared__ double ip_s;
  const int r = threadIdx.x / kSw, c = threadIdx.x % kSw;
  D[r][c] = A[static_cast<size_t>(r) * mp + c];
  sweep_diagonal(D, ip_s, b, status);
  A[static_cast<size_t>(r) * mp + c] = D[r][c];
}

// Panel k: tile b < nb is the column tile (b, k), nb + b the row tile (k, b); b = k skipped (its own
// steps ran before). Two CTAs of eight rows (columns) per tile: half a warp holds a tile row
// (column) of kSw values, lane s its value s; step t broadcasts value t within the half
// warp. The steps are a chain of two FP64 instructions, whose issue (a warp's takes 16
// clocks) is what the small CTAs spread over the SMs.
__global__ void __launch_bounds__(kSw * kSw / 2) k_coarsest_panel(double* __restrict__ A, int mp, int k, SweepBuf b) {
  const int nb = mp / kSw;
  const int id = static_cast<int>(blockIdx.x) >> 1;
  const bool is_row = id >= nb;
  const int tile = is_row ? id - nb : id;
  if (tile == k) return;
  __shared__ double dv[kSw][kSw + 1], ips[kSw], T[kSw / 2][kSw + 1];
  const int il = threadIdx.x / kSw, s = threadIdx.x % kSw;
  const int i = il + (blockIdx.x & 1) * (kSw / 2);
  // dv[t][s]: what step t multiplies value t with to update value s
  for (int e = threadIdx.x; e < kSw * kSw; e += kSw * kSw / 2) {
    const int x = e / kSw, y = e % kSw;
    dv[is_row ? y : x][is_row ? x : y] = is_row ? b.dcol[e] : b.drow[e];
  }
  if (threadIdx.x < kSw) ips[threadIdx.x] = b.ip[threadIdx.x];
  // a row tile is transposed on the way: lane s of half warp il takes row s of column i
  const int half = kSw / 2;
  const size_t at = is_row ? static_cast<size_t>(kSw * k + threadIdx.x / half) * mp + kSw * tile +
                                 (blockIdx.x & 1) * half + threadIdx.x % half
                           : static_cast<size_t>(kSw * tile + i) * mp + kSw * k + s;
  double v = A[at];
  if (is_row) T[threadIdx.x % half][threadIdx.x / half] = v;
  __syncthreads();
  if (is_row) v = T[il][s];
  double save = 0.0;
#pragma unroll
  for (int t = 0; t < kSw; ++t) {
    const double x = __shfl_sync(0xffffffffu, v, t, kSw);
    double p = __dmul_rn(x, dv[t][s]);
    if (s == t) {
      save = x;
      p = is_row ? -x : x;
    }
    v = fma(-p, ips[t], s == t ? 0.0 : v);
  }
  (is_row ? b.row : b.col)[static_cast<size_t>(kSw * tile + i) * kSw + s] = save;
  if (is_row) {
    __syncthreads();
    T[il][s] = v;
    __syncthreads();
    v = T[threadIdx.x % half][threadIdx.x / half];
  }
  A[at] = v;
}

// Every tile outside panel k's rows and columns: the panel's kSw steps in order. The tile of
// the next diagonal block then runs that block's own steps into nb.
__global__ void __launch_bounds__(kSw * kSw) k_coarsest_rest(double* __restrict__ A, int mp, int k, SweepBuf b,
                                                            SweepBuf next, int* __restrict__ status) {
  const int bi = blockIdx.y, bj = blockIdx.x;
  if (bi == k || bj == k) return;
  __shared__ double cs[kSw][kSw + 1], rs[kSw][kSw + 1], ips[kSw];
  __shared__ double ip_s;
  const int r = threadIdx.x / kSw, c = threadIdx.x % kSw;
  const size_t at = static_cast<size_t>(kSw * bi + r) * mp + kSw * bj + c;
  cs[r][c] = b.col[static_cast<size_t>(kSw * bi + r) * kSw + c];
  rs[r][c] = b.row[static_cast<size_t>(kSw * bj + r) * kSw + c];
  if (threadIdx.x < kSw) ips[threadIdx.x] = b.ip[threadIdx.x];
  double a = A[at];
  __syncthreads();
#pragma unroll
  for (int t = 0; t < kSw; ++t) a = sweep_update(a, cs[r][t], rs[c][t], ips[t]);
  if (bi == k + 1 && bj == k + 1) {
    __syncthreads();
    cs[r][c] = a;
    sweep_diagonal(cs, ip_s, next, status);
    a = cs[r][c];
  }
  A[at] = a;
}

// The three component means of row i of the embedded inverse X (rows and columns 0..2 zero),
// rmean[3 i + b], summed in column order; a thread per (row, component).
__global__ void __launch_bounds__(128) k_coarsest_means(const double* __restrict__ A, int m, int mp,
                                                        double* __restrict__ rmean) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int i = t / 3, b = t - 3 * i;
  if (i >= m) return;
  double s = 0.0;
  if (i >= 3) {
    const double* row = A + static_cast<size_t>(i - 3) * mp + b;
#pragma unroll 8
    for (int w = 1; w < m / 3; ++w) s += row[3 * w - 3];
  }
  rmean[t] = s / (m / 3);
}

// G = P X P with P the projector removing the 3 rigid translations (per-component means): the
// centred pseudo-inverse of the coarsest operator (Sec. 4.2 null-space removal).
__global__ void __launch_bounds__(256) k_coarsest_centre(const double* __restrict__ A, int m, int mp,
                                                         const double* __restrict__ rmean, double* __restrict__ G) {
  extern __shared__ double rms[];   // the 3 m row means: every block sums them in the same order
  __shared__ double tot[9];
  const int nv = m / 3;
  for (int t = threadIdx.x; t < 3 * m; t += blockDim.x) rms[t] = rmean[t];
  __syncthreads();
  if (threadIdx.x < 9) {
    const int a = threadIdx.x / 3, b = threadIdx.x % 3;
    double s = 0.0;
    for (int v = 0; v < nv; ++v) s += rms[(3 * v + a) * 3 + b];
    tot[threadIdx.x] = s / nv;
  }
  __syncthreads();
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < m * m; e += gridDim.x * blockDim.x) {
    const int i = e / m, j = e - i * m;
    const int a = i % 3, b = j % 3;
    const double x = i < 3 || j < 3 ? 0.0 : A[static_cast<size_t>(i - 3) * mp + j - 3];
    // X symmetric: column mean of column j over rows of component a = rms[j][a]
    G[e] = x - rms[3 * i + b] - rms[3 * j + a] + tot[3 * a + b];
  }
}

// x = G b for the 6 cases (FP64 dot products), a warp per ROWS output rows for all cases, each in
// a CTA of its own: the FP64 pipe (2 operations per clock and SM, a conversion from FP32
// costing one) bounds it, so the rows spread over every SM, and where there are more rows
// than that a warp shares the converted right-hand sides between two.
template <int ROWS>
__global__ void __launch_bounds__(32) k_coarsest_apply(const double* __restrict__ G, int m,
                                                       const float* __restrict__ b,
                                                       float* __restrict__ x) {
  const int nv = m / 3, lane = threadIdx.x;
  const int i0 = blockIdx.x * ROWS;
  double s[ROWS][kCases] = {};
#pragma unroll 2
  for (int j = lane; j < m; j += 32) {
    const int w = j / 3, k = j - 3 * w;
    double g[ROWS];
#pragma unroll
    for (int r = 0; r < ROWS; ++r) g[r] = i0 + r < m ? __ldg(G + static_cast<size_t>(i0 + r) * m + j) : 0.0;
#pragma unroll
    for (int c = 0; c < kCases; ++c) {
      const double v = static_cast<double>(__ldg(b + static_cast<size_t>(3 * c + k) * nv + w));
#pragma unroll
      for (int r = 0; r < ROWS; ++r) s[r][c] = fma(g[r], v, s[r][c]);
    }
  }
#pragma unroll
  for (int r = 0; r < ROWS; ++r) {
    const int i = i0 + r;
#pragma unroll
    for (int c = 0; c < kCases; ++c) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s[r][c] += __shfl_down_sync(0xffffffffu, s[r][c], o);
      if (lane == 0 && i < m) x[static_cast<size_t>(3 * c + i % 3) * nv + i / 3] = static_cast<float>(s[r][c]);
    }
  }
}

// Export a stencil in vertex-major order out[(v*27 + d)*9 + q].
__global__ void k_stencil_export(const float* __restrict__ st, int n, bool cb,
                                 float* __restrict__ out) {
  const size_t N = static_cast<size_t>(n) * n * n;
  for (size_t it = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; it < N * kStencil;
       it += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const size_t v = it / kStencil;
    const int k = static_cast<int>(it % kStencil);
    const int x = static_cast<int>(v % n), y = static_cast<int>((v / n) % n),
              z = static_cast<int>(v / (static_cast<size_t>(n) * n));
    out[it] = st[static_cast<size_t>(k) * N + stencil_pos(x, y, z, n, cb)];
  }
}

}  // namespace

cudaError_t launch_level1_assemble(const homo_ctx* c, const Level& L1) {
  // the 18 KB table travels in the kernel's parameter bank (limit 32 KB)
  BfParam B;
  for (int i = 0; i < 8 * 576; ++i) B.b[i] = c->hBf[i];
  k_level1<<<grid_for(L1.N, 128), 128, 0, c->stream>>>(B, c->E, c->n, L1.st, L1.n, L1.colour_blocked);
  return cudaGetLastError();
}

cudaError_t launch_galerkin(const Level& Lf, const Level& Lc, float* tmp1, float* tmp2, cudaStream_t s) {
  const int n = Lf.n, h = n / 2;
  if (Lc.n != h || !Lf.colour_blocked) return cudaErrorInvalidValue;
  const size_t n1 = static_cast<size_t>(h) * n * n, n2 = static_cast<size_t>(h) * h * n;
  // x: level stencil -> (h, n, n) in tmp1; y: -> (h, h, n) in tmp2; z: -> the coarse level
  k_galerkin_axis<0><<<grid_for(27 * n1, 256), 256, 0, s>>>(Lf.st, n, n, n, true, tmp1, false);
  k_galerkin_axis<1><<<grid_for(27 * n2, 256), 256, 0, s>>>(tmp1, h, n, n, false, tmp2, false);
  k_galerkin_axis<2><<<grid_for(27 * Lc.N, 256), 256, 0, s>>>(tmp2, h, h, n, false, Lc.st, Lc.colour_blocked);
  return cudaGetLastError();
}

namespace {

template <typename T, int CASES, int VERTS>
cudaError_t tile_launch(const Level& L, const T* st, int colour, int first, int chained, const float* f, float* x,
                        cudaStream_t s) {
  const size_t h = static_cast<size_t>(L.n / 2), Nh = h * h * h;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>((Nh + VERTS - 1) / VERTS));
  cfg.blockDim = dim3(VERTS * kCases / CASES);
  cfg.dynamicSmemBytes = static_cast<size_t>(kStencil) * VERTS * sizeof(T);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = chained ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k_coarse_gs_tile<T, CASES, VERTS>, st, f, x, L.n, colour, first, chained);
}

// A colour pass in the staged form: a case per thread up to kTileSplitN cells per axis (the
// threads to fill the chip), three above (the stencil's shared-memory reads per case).
constexpr int kTileSplitN = 96;

template <typename T>
cudaError_t tile_pass(const Level& L, const T* st, int colour, int first, int chained, const float* f, float* x,
                      cudaStream_t s) {
  return L.n <= kTileSplitN ? tile_launch<T, 1, 32>(L, st, colour, first, chained, f, x, s)
                            : tile_launch<T, 3, 64>(L, st, colour, first, chained, f, x, s);
}

template <typename T, int CASES, int VERTS>
cudaError_t tile_attr() {
  constexpr int shm = static_cast<int>(kStencil * VERTS * sizeof(T));
  const cudaError_t e = cudaFuncSetAttribute(k_coarse_gs_tile<T, CASES, VERTS>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, shm);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_coarse_residual_tile<T, CASES, VERTS>, cudaFuncAttributeMaxDynamicSharedMemorySize, shm);
}

}  // namespace

bool coarse_tile_ok(const Level& L) { return L.n % 4 == 0; }

namespace {
template <typename T, int CASES, int VERTS>
void residual_tile(const Level& L, const T* st, const float* b, const float* x, float* out, cudaStream_t s) {
  const size_t h = static_cast<size_t>(L.n / 2);
  const unsigned blocks = static_cast<unsigned>((h * h * h + VERTS - 1) / VERTS);
  k_coarse_residual_tile<T, CASES, VERTS><<<8 * blocks, VERTS * kCases / CASES, kStencil * VERTS * sizeof(T), s>>>(
      st, b, x, out, L.n, blocks);
}

template <typename T>
cudaError_t residual_launch(const Level& L, const T* st, const float* b, const float* x, float* out, cudaStream_t s) {
  if (!coarse_tile_ok(L))
    k_coarse_residual<<<grid_for(L.N, 256), 256, 0, s>>>(st, b, x, out, L.n, L.colour_blocked);
  else if (L.n <= kTileSplitN)
    residual_tile<T, 1, 32>(L, st, b, x, out, s);
  else
    residual_tile<T, 3, 64>(L, st, b, x, out, s);
  return cudaGetLastError();
}
}  // namespace

cudaError_t launch_coarse_residual(const Level& L, const float* b, const float* x, float* out,
                                   cudaStream_t s) {
  return L.sth ? residual_launch(L, static_cast<const __nv_bfloat16*>(L.sth), b, x, out, s)
               : residual_launch(L, static_cast<const float*>(L.st), b, x, out, s);
}

cudaError_t launch_coarse_gs_tile(const Level& L, int colour, const float* f, float* x, int first, int chained,
                                  cudaStream_t s) {
  return L.sth ? tile_pass(L, static_cast<const __nv_bfloat16*>(L.sth), colour, first, chained, f, x, s)
               : tile_pass(L, static_cast<const float*>(L.st), colour, first, chained, f, x, s);
}

cudaError_t launch_coarse_gs(const Level& L, int colour, const float* f, float* x, int first,
                             cudaStream_t s) {
  const size_t h = static_cast<size_t>(L.n / 2);
  if (L.sth) k_coarse_gs<<<grid_for(h * h * h, 256), 256, 0, s>>>(L.sth, f, x, L.n, colour, first);
  else k_coarse_gs<<<grid_for(h * h * h, 256), 256, 0, s>>>(L.st, f, x, L.n, colour, first);
  return cudaGetLastError();
}

namespace {

template <typename T>
int cluster_fits(int size) {
  const void* fn = reinterpret_cast<const void*>(k_coarse_gs_cluster<T>);
  if (cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, size > 8 ? 1 : 0) != cudaSuccess)
    return 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(size);
  cfg.blockDim = dim3(kClusterBlock);
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = size;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int count = 0;
  if (cudaOccupancyMaxActiveClusters(&count, fn, &cfg) != cudaSuccess) return 0;
  return count;
}

std::mutex g_cluster_mu;
int g_cluster_size[256] = {};    // per device: 0 = not queried, -1 = no cluster launch
int g_resident_size[256] = {};   // per device: largest resident-form cluster, -1 = none
constexpr int kResidentSmemMax = 216 * 1024;   // dynamic shared memory of the resident form, at most

int resident_fits(int size, const void* fn) {
  if (cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, size > 8 ? 1 : 0) != cudaSuccess ||
      cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kResidentSmemMax) != cudaSuccess)
    return 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(size);
  cfg.blockDim = dim3(kResThreads);
  cfg.dynamicSmemBytes = kResidentSmemMax;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = size;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int count = 0;
  if (cudaOccupancyMaxActiveClusters(&count, fn, &cfg) != cudaSuccess) return 0;
  return count;
}

// Cluster size, vertices per colour and CTA, and colour groups of the resident form on level
// L, or false when the level does not qualify. 8 groups (every row in registers) wherever
// at most cluster_max CTAs of 16 vertices hold a colour, else 4 groups of 32.
bool resident_shape(const Level& L, int cluster_max, int& csize, int& Mper, int& groups, size_t& smem) {
  if (cluster_max < 1 || L.n % 2 || L.n > 16) return false;
  const int h = L.n / 2, Nh = h * h * h;
  groups = Nh <= 16 * cluster_max ? 8 : 4;
  const int verts = groups == 8 ? 16 : 32;
  int size = 1;
  while (size < cluster_max && size * verts < Nh) size *= 2;
  if (size * verts < Nh) return false;
  csize = size;
  Mper = (Nh + size - 1) / size;
  smem = resident_smem_bytes(L.N, Mper, groups);
  return smem <= static_cast<size_t>(kResidentSmemMax);
}

}  // namespace

int coarse_cluster_size() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 256) {
    cudaGetLastError();
    return -1;
  }
  std::lock_guard<std::mutex> lk(g_cluster_mu);
  if (g_cluster_size[dev] == 0) {
    int best = -1;
    for (int size : {16, 8, 4}) {
      if (cluster_fits<float>(size) > 0 && cluster_fits<__nv_bfloat16>(size) > 0) {
        best = size;
        break;
      }
    }
    int res = -1;
    for (int size : {16, 8, 4, 2, 1}) {
      const void* forms[] = {reinterpret_cast<const void*>(k_coarse_gs_resident<float, 8>),
                             reinterpret_cast<const void*>(k_coarse_gs_resident<float, 4>),
                             reinterpret_cast<const void*>(k_coarse_gs_resident<__nv_bfloat16, 8>),
                             reinterpret_cast<const void*>(k_coarse_gs_resident<__nv_bfloat16, 4>),
                             reinterpret_cast<const void*>(k_fine_gs_resident<8>),
                             reinterpret_cast<const void*>(k_fine_gs_resident<4>)};
      if (std::all_of(std::begin(forms), std::end(forms), [size](const void* fn) { return resident_fits(size, fn) > 0; })) {
        res = size;
        break;
      }
    }
    cudaGetLastError();   // a refused size leaves its error behind
    g_cluster_size[dev] = best;
    g_resident_size[dev] = res;
  }
  return g_cluster_size[dev];
}

int coarse_resident_size() {
  coarse_cluster_size();   // runs the per-device queries once
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 256) {
    cudaGetLastError();
    return -1;
  }
  std::lock_guard<std::mutex> lk(g_cluster_mu);
  return g_resident_size[dev] == 0 ? -1 : g_resident_size[dev];
}

bool coarse_resident_ok(const Level& L, int cluster_max) {
  int csize, Mper, groups;
  size_t smem;
  return resident_shape(L, cluster_max, csize, Mper, groups, smem);
}

namespace {
// Launch configuration of a resident smoother on level L.
struct ResidentLaunch {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  int csize = 0, Mper = 0, groups = 0;
  bool set(const Level& L, int cluster_max, cudaStream_t s) {
    size_t smem;
    if (!resident_shape(L, cluster_max, csize, Mper, groups, smem)) return false;
    cfg.gridDim = dim3(kCases * csize);
    cfg.blockDim = dim3(kResThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = csize;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return true;
  }
};

template <typename T>
cudaError_t resident_launch(const Level& L, const T* st, int sweeps, int reverse, int first, const float* f, float* x,
                            int cluster_max, cudaStream_t s) {
  ResidentLaunch r;
  if (!r.set(L, cluster_max, s)) return cudaErrorInvalidValue;
  return cudaLaunchKernelEx(&r.cfg, r.groups == 8 ? k_coarse_gs_resident<T, 8> : k_coarse_gs_resident<T, 4>, st, f, x,
                            L.n, sweeps, reverse, first, r.csize, r.Mper);
}
}  // namespace

cudaError_t launch_fine_gs_resident(const homo_ctx* c, int reverse, const float* f, float* u, int first,
                                    const float* fmean) {
  ResidentLaunch r;
  if (!r.set(c->lev[0], c->gs_resident, c->stream)) return cudaErrorInvalidValue;
  const float* E = c->E;
  return cudaLaunchKernelEx(&r.cfg, r.groups == 8 ? k_fine_gs_resident<8> : k_fine_gs_resident<4>, c->ke, E, f, u,
                            c->n, reverse, first, fmean, r.csize, r.Mper);
}

cudaError_t launch_coarse_gs_resident(const Level& L, int sweeps, int reverse, int first, const float* f,
                                      float* x, int cluster_max, cudaStream_t s) {
  return L.sth ? resident_launch(L, static_cast<const __nv_bfloat16*>(L.sth), sweeps, reverse, first, f, x, cluster_max, s)
               : resident_launch(L, static_cast<const float*>(L.st), sweeps, reverse, first, f, x, cluster_max, s);
}

cudaError_t launch_coarse_gs_sweeps(const Level& L, int sweeps, int reverse, int first, const float* f,
                                    float* x, int cluster_max, cudaStream_t s) {
  const unsigned h = static_cast<unsigned>(L.n / 2);
  const size_t Nh = static_cast<size_t>(h) * h * h;
  // per case: the smallest power-of-two cluster with a thread per vertex of a colour, at
  // most cluster_max CTAs
  const size_t need = (Nh + kClusterBlock - 1) / kClusterBlock;
  int size = 1;
  while (size < cluster_max && static_cast<size_t>(size) < need) size *= 2;
  if (size > cluster_max) size = cluster_max;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kCases * size);
  cfg.blockDim = dim3(kClusterBlock);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = size;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (L.sth)
    return cudaLaunchKernelEx(&cfg, k_coarse_gs_cluster<__nv_bfloat16>, L.sth, f, x, L.n, sweeps, reverse, first, size);
  return cudaLaunchKernelEx(&cfg, k_coarse_gs_cluster<float>, L.st, f, x, L.n, sweeps, reverse, first, size);
}

cudaError_t launch_coarse_gs_item(const Level& L, int colour, const float* f, float* x, int first,
                                  cudaStream_t s) {
  const unsigned h = static_cast<unsigned>(L.n / 2);
  const int g = grid_for(gs_items(h * h * h), kItemBlock);
  if (L.sth) k_coarse_gs_item<<<g, kItemBlock, 0, s>>>(L.sth, f, x, L.n, colour, first);
  else k_coarse_gs_item<<<g, kItemBlock, 0, s>>>(L.st, f, x, L.n, colour, first);
  return cudaGetLastError();
}

cudaError_t launch_coarse_cheb(const Level& L, const float* b, const float* x_in, float* out, int mode,
                               float c0, float c1, cudaStream_t s) {
  if (L.sth) k_coarse_cheb<<<grid_for(L.N, 256), 256, 0, s>>>(L.sth, b, x_in, out, L.n, L.colour_blocked, mode, c0, c1);
  else k_coarse_cheb<<<grid_for(L.N, 256), 256, 0, s>>>(L.st, b, x_in, out, L.n, L.colour_blocked, mode, c0, c1);
  return cudaGetLastError();
}

cudaError_t launch_coarse_dinvk(const Level& L, const float* x, float* y, cudaStream_t s) {
  if (L.sth) k_coarse_cheb<<<grid_for(L.N, 256), 256, 0, s>>>(L.sth, nullptr, x, y, L.n, L.colour_blocked, 2, 0.f, 0.f);
  else k_coarse_cheb<<<grid_for(L.N, 256), 256, 0, s>>>(L.st, nullptr, x, y, L.n, L.colour_blocked, 2, 0.f, 0.f);
  return cudaGetLastError();
}

cudaError_t launch_fill_hash(float* x, size_t count, unsigned seed, cudaStream_t s) {
  k_fill_hash<<<grid_for(count, 256), 256, 0, s>>>(x, count, seed);
  return cudaGetLastError();
}

cudaError_t launch_restrict(int nf, const float* fine, float* coarse, cudaStream_t s) {
  const size_t nc = static_cast<size_t>(nf / 2);
  k_restrict<<<dim3(grid_for(nc * nc * nc, 256), kCases), 256, 0, s>>>(fine, nf, coarse);
  return cudaGetLastError();
}

cudaError_t launch_prolong_add(int nf, const float* coarse, float* fine, int overwrite,
                               cudaStream_t s) {
  const size_t Nf = static_cast<size_t>(nf) * nf * nf;
  const dim3 grid(grid_for(Nf / 8, 256), kCases);
  if (reinterpret_cast<uintptr_t>(fine) % 8 == 0) k_prolong<true><<<grid, 256, 0, s>>>(coarse, nf, fine, overwrite);
  else k_prolong<false><<<grid, 256, 0, s>>>(coarse, nf, fine, overwrite);
  return cudaGetLastError();
}

size_t coarsest_work_doubles(int m) {   // A, two sets of saved panel values, row means
  const size_t mp = static_cast<size_t>(sweep_size(m));
  return mp * mp + 2 * (2 * mp * kSw + 2 * kSw * kSw + kSw) + 3 * static_cast<size_t>(m);
}

int coarsest_setup_kernels(int m) { return 4 + 2 * (sweep_size(m) / kSw); }

cudaError_t launch_coarsest_setup(homo_ctx* c) {
  const Level& L = c->lev[c->nlev - 1];
  const int m = c->mc, mp = sweep_size(m), np = mp / kSw;
  double* at = c->A + static_cast<size_t>(mp) * mp;
  SweepBuf buf[2];
  for (SweepBuf& b : buf) {
    b = {at, at + mp * kSw, at + 2 * mp * kSw, at + 2 * mp * kSw + kSw * kSw, at + 2 * mp * kSw + 2 * kSw * kSw};
    at = b.ip + kSw;
  }
  double* rmean = at;
  cudaError_t e = cudaMemsetAsync(c->A, 0, sizeof(double) * mp * mp, c->stream);
  if (e != cudaSuccess) return e;
  int* status = reinterpret_cast<int*>(c->scal + S_OC + 63);
  e = cudaMemsetAsync(status, 0, sizeof(int), c->stream);
  if (e != cudaSuccess) return e;
  k_coarsest_dense<<<grid_for(27 * L.N, 256), 256, 0, c->stream>>>(L.st, L.n, L.colour_blocked, mp, c->A);
  k_coarsest_first<<<1, kSw * kSw, 0, c->stream>>>(c->A, mp, buf[0], status);
  for (int k = 0; k < np; ++k) {
    k_coarsest_panel<<<4 * np, kSw * kSw / 2, 0, c->stream>>>(c->A, mp, k, buf[k & 1]);
    k_coarsest_rest<<<dim3(np, np), kSw * kSw, 0, c->stream>>>(c->A, mp, k, buf[k & 1], buf[(k + 1) & 1], status);
  }
  k_coarsest_means<<<(3 * m + 127) / 128, 128, 0, c->stream>>>(c->A, m, mp, rmean);
  k_coarsest_centre<<<std::min(grid_for(static_cast<size_t>(m) * m, 256), 304), 256, sizeof(double) * 3 * m, c->stream>>>(
      c->A, m, mp, rmean, c->G);
  return cudaGetLastError();
}

cudaError_t coarse_init() {   // shared-memory limits, before any capture
  cudaError_t e = tile_attr<float, 1, 32>();
  if (e == cudaSuccess) e = tile_attr<float, 3, 64>();
  if (e == cudaSuccess) e = tile_attr<__nv_bfloat16, 1, 32>();
  if (e == cudaSuccess) e = tile_attr<__nv_bfloat16, 3, 64>();
  return e;
}

cudaError_t launch_coarsest_apply(const homo_ctx* c, const float* b, float* x) {
  const int m = c->mc;
  if (m <= 2 * 152) k_coarsest_apply<1><<<m, 32, 0, c->stream>>>(c->G, m, b, x);
  else k_coarsest_apply<2><<<(m + 1) / 2, 32, 0, c->stream>>>(c->G, m, b, x);
  return cudaGetLastError();
}

cudaError_t launch_stencil_bf16(const Level& L, cudaStream_t s) {
  if (!L.sth || !L.st) return cudaErrorInvalidValue;
  k_stencil_bf16<<<grid_for(27 * L.N, 256), 256, 0, s>>>(L.st, L.n, L.colour_blocked, L.sth);
  return cudaGetLastError();
}

cudaError_t launch_stencil_export(const Level& L, float* out, cudaStream_t s) {
  k_stencil_export<<<grid_for(L.N * kStencil, 256), 256, 0, s>>>(L.st, L.n, L.colour_blocked, out);
  return cudaGetLastError();
}

}  // namespace homo
