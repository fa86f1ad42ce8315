// Finest-level kernels. The level-0 stiffness is never stored (Sec. 4.1): every kernel
// rebuilds what it needs from the element moduli E and the element matrix K0, which sits
// in the kernel's parameter (constant) bank.
//
// Vertex form of K u (Eq. 13): incident element t = a + 2b + 4c of vertex v has origin
// v - (1,1,1) + (a,b,c) and v is its local vertex 7 - t. The 3x3 coupling block between v
// and its neighbour v + d is
//     A_d = sum over (t, j) with bits(t) + bits(j) - 1 = d of E_t * K0[7 - t, j],
// built once per vertex and applied to all 6 load cases (the 6 cases share E and K0).
#include <cstring>
#include <mutex>
#include <string>

#include "dev_common.cuh"
#include "stencil.cuh"

#include <utility>

namespace homo {

namespace {

// Error-free transformations (Knuth TwoSum, FMA-based TwoProduct) with operations the
// compiler may not contract or reorder.
__device__ __forceinline__ f32x2 fmul2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bb = __fadd_rn(s, -a);
  e = __fadd_rn(__fadd_rn(a, -__fadd_rn(s, -bb)), __fadd_rn(b, -bb));
}

// Macro-strain loads in vertex form (Eq. 11): f_(i,v) = sum_t E_t (K0 chi_i)[7 - t].
// In a uniform medium the 8 element forces at a vertex cancel exactly (sum_t (K0
// chi_i)[7 - t] = 0), so the kernel sums (E_t - E_0) (K0 chi_i)[7 - t]: the loads are
// exactly zero where E is locally uniform and carry no cancellation error elsewhere.
// The sum is formed in double-float arithmetic (the difference E_t - E_0 and K0 chi split
// exactly, error-free products and sums) and stored as f + flo: an FP32 load rounded
// against the largest of its terms perturbs the weakly held soft-region displacements,
// whose strain energies the sensitivities of Eq. 9 weigh.
__global__ void __launch_bounds__(256) k_loads(const __grid_constant__ LoadParam L,
                                               const float* __restrict__ E,
                                               float* __restrict__ f, float* __restrict__ flo, int n) {
  const size_t N = static_cast<size_t>(n) * n * n;
  for (size_t v = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; v < N;
       v += static_cast<size_t>(gridDim.x) * blockDim.x) {
    int x, y, z;
    decode3(static_cast<unsigned>(v), static_cast<unsigned>(n), x, y, z);
    const Nb nb = make_nb(x, y, z, n);
    float Et[8];
    load_E8(E, nb, Et);
    float dh[8], dl[8];
#pragma unroll
    for (int t = 1; t < 8; ++t) two_sum(Et[t], -Et[0], dh[t], dl[t]);   // E_t - E_0 = dh + dl
#pragma unroll
    for (int c = 0; c < kCases; ++c)
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        float hi = 0.f, lo = 0.f;
#pragma unroll
        for (int t = 1; t < 8; ++t) {
          const float a = L.fe[c][3 * (7 - t) + r], al = L.fe_lo[c][3 * (7 - t) + r];
          const float p = __fmul_rn(dh[t], a);
          const float pe = fmaf(dh[t], a, -p);               // dh a = p + pe exactly
          float s, e;
          two_sum(hi, p, s, e);
          hi = s;
          lo = __fadd_rn(lo, __fadd_rn(__fadd_rn(e, pe), fmaf(dh[t], al, __fmul_rn(dl[t], a))));
        }
        const float s2 = __fadd_rn(hi, lo);
        const size_t o = static_cast<size_t>(3 * c + r) * N + v;
        f[o] = s2;
        flo[o] = __fadd_rn(lo, -__fadd_rn(s2, -hi));          // FastTwoSum: f + flo = hi + lo
      }
  }
}


// The signed sums of moduli that the blocks A_d are products of: with F the axes where d is 0,
// a block needs, for every subset g of F, the sum over the contributing elements (in the order
// of t) of E_t times the signs of t along g. 8 corners need 1, 12 edges 2, 6 faces 4.
constexpr int kDSums = 56;

struct DBlocks {
  float k[27][9];            // K0[0][|d|][r][c] with the signs d_a d_b of the axes where d is not 0
  unsigned char o[27][4];    // which sum: diagonal, (0,1), (0,2), (1,2)
};

__host__ __device__ constexpr int dsum_slot(int d, int sub) {   // sub: bit k = sign along axis k
  int base = 0;
  for (int e = 0; e < d; ++e) {
    const int f = (e % 3 == 1) + (e / 3 % 3 == 1) + (e / 9 == 1);
    base += f == 3 ? 0 : 1 << f;
  }
  int pos = 0, bit = 0;
  const int D[3] = {d % 3 - 1, d / 3 % 3 - 1, d / 9 - 1};
  for (int k = 0; k < 3; ++k)
    if (D[k] == 0) {
      if (sub >> k & 1) pos |= 1 << bit;
      ++bit;
    }
  return base + pos;
}

DBlocks make_dblocks(const KeParam& K) {
  DBlocks B;
  for (int d = 0; d < 27; ++d) {
    const int D[3] = {d % 3 - 1, d / 3 % 3 - 1, d / 9 - 1};
    const int m = (D[0] != 0 ? 1 : 0) + (D[1] != 0 ? 2 : 0) + (D[2] != 0 ? 4 : 0);
    for (int r = 0; r < 3; ++r)
      for (int c = 0; c < 3; ++c) {
        float v = K.k[24 * r + 3 * m + c];
        if (r != c) v *= static_cast<float>((D[r] != 0 ? D[r] : 1) * (D[c] != 0 ? D[c] : 1));
        B.k[d][3 * r + c] = v;
      }
    const int ax[4][2] = {{0, 0}, {0, 1}, {0, 2}, {1, 2}};
    for (int i = 0; i < 4; ++i) {
      int sub = 0;
      if (i > 0) sub = (D[ax[i][0]] == 0 ? 1 << ax[i][0] : 0) | (D[ax[i][1]] == 0 ? 1 << ax[i][1] : 0);
      B.o[d][i] = static_cast<unsigned char>(d == 13 ? 0 : dsum_slot(d, sub));
    }
  }
  return B;
}

constexpr int kTrueResThreads = 128;

// Sum for block i / 8 and axes i % 8, if the block has it, stored with stride kTrueResThreads.
template <int i>
__device__ __forceinline__ void store_dsum(const float (&Et)[8], float* s) {
  constexpr int d = i / 8, sub = i % 8, dx = d % 3 - 1, dy = d / 3 % 3 - 1, dz = d / 9 - 1;
  if constexpr (d != 13 && !((sub & 1) && dx != 0) && !((sub & 2) && dy != 0) && !((sub & 4) && dz != 0)) {
    constexpr int slot = dsum_slot(d, sub);
    float acc = 0.f;
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const int a = t & 1, b = t >> 1 & 1, c = t >> 2;
      if ((dx != 0 && a != (dx > 0)) || (dy != 0 && b != (dy > 0)) || (dz != 0 && c != (dz > 0))) continue;
      const bool neg = ((sub & 1) && !a) != (((sub & 2) && !b) != ((sub & 4) && !c));
      acc += neg ? -Et[t] : Et[t];
    }
    s[slot * kTrueResThreads] = acc;
  }
}

template <int... i>
__device__ __forceinline__ void store_dsums(const float (&Et)[8], float* s, std::integer_sequence<int, i...>) {
  (store_dsum<i>(Et, s), ...);
}

// r = (b + blo) - K (u + ulo) evaluated in double-float arithmetic (difference form, products
// and sums error-free up to the final rounding), then partials of ||r_c||^2 and of the
// 18 plane sums. This is the accurate true residual the CG driver restarts from; it uses
// exactly the FP32 blocks A_d of the CG product, so both see the same operator.
//
// Bound by the FMA pipe (69 % busy with 12 warps an SM): 369 two-lane operations per neighbour,
// two cycles each. Around them a block costs 4 shared loads (its signed sums, formed once per
// vertex) and 9 products with uniform constants; rebuilt from the 8 moduli at a runtime d it
// took as many instructions as a third of the arithmetic. 160^3: 3.52 -> 3.27 ms.
__global__ void __launch_bounds__(kTrueResThreads) k_fine_true_residual(const __grid_constant__ DBlocks B,
                                                                     const float* __restrict__ E,
                                                                     const float* __restrict__ u,
                                                                     const float* __restrict__ ulo,
                                                                     const float* __restrict__ b,
                                                                     const float* __restrict__ blo,
                                                                     float* __restrict__ out, int n,
                                                                     double* __restrict__ part) {
  __shared__ float ssum[kDSums][kTrueResThreads];   // each thread its own column
  const size_t N = static_cast<size_t>(n) * n * n;
  float red[kCases + kPlanes];
#pragma unroll
  for (int c = 0; c < kCases + kPlanes; ++c) red[c] = 0.f;
  for (size_t v = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; v < N;
       v += static_cast<size_t>(gridDim.x) * blockDim.x) {
    int x, y, z;
    decode3(static_cast<unsigned>(v), static_cast<unsigned>(n), x, y, z);
    const Nb nb = make_nb(x, y, z, n);
    {
      float Et[8];
      load_E8(E, nb, Et);
      store_dsums(Et, &ssum[0][threadIdx.x], std::make_integer_sequence<int, 27 * 8>{});
    }
    // The 6 cases advance in pairs (2p, 2p + 1) on the two lanes of f32x2 registers. Every
    // lane performs exactly the scalar operations of the double-float recurrence below,
    // in the same order (the negated-operand forms are exact: round to nearest is
    // symmetric), so the result is bitwise that of a scalar evaluation:
    //   dh + e = u_(v+d) - u_v (two-sum), dl = e + (ulo_(v+d) - ulo_v),
    //   p = a dh, pe = a dh - p (FMA), hi + e' = hi + p (two-sum),
    //   lo += e' + (a dl + pe).
    f32x2 hi[9], lo[9], nown[9], ownlo[9];
    const unsigned v32 = static_cast<unsigned>(v);
#pragma unroll
    for (int p = 0; p < 3; ++p)
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const int q0 = 6 * p + k, q1 = q0 + 3;
        hi[3 * p + k] = 0ull;
        lo[3 * p + k] = 0ull;
        nown[3 * p + k] = pack2(-__ldg(u + q0 * N + v32), -__ldg(u + q1 * N + v32));
        ownlo[3 * p + k] = pack2(__ldg(ulo + q0 * N + v32), __ldg(ulo + q1 * N + v32));
      }
#pragma unroll 1
    for (int d = 0; d < 27; ++d) {
      if (d == 13) continue;
      const int rx = d % 3, ry = (d / 3) % 3, rz = d / 9;
      const int yz = (ry == 0 ? nb.Y[0] : (ry == 1 ? nb.Y[1] : nb.Y[2])) +
                     (rz == 0 ? nb.Z[0] : (rz == 1 ? nb.Z[1] : nb.Z[2]));
      const float s0 = ssum[B.o[d][0]][threadIdx.x], s01 = ssum[B.o[d][1]][threadIdx.x],
                  s02 = ssum[B.o[d][2]][threadIdx.x], s12 = ssum[B.o[d][3]][threadIdx.x];
      const float* C = B.k[d];
      const float A[9] = {C[0] * s0,  C[1] * s01, C[2] * s02, C[3] * s01, C[4] * s0,
                          C[5] * s12, C[6] * s02, C[7] * s12, C[8] * s0};
      f32x2 Ap[9], An[9];
#pragma unroll
      for (int e = 0; e < 9; ++e) {
        Ap[e] = pack2(A[e], A[e]);
        An[e] = pack2(-A[e], -A[e]);
      }
      const unsigned w = static_cast<unsigned>((rx == 0 ? nb.X[0] : (rx == 1 ? nb.X[1] : nb.X[2])) + yz);
#pragma unroll
      for (int p = 0; p < 3; ++p) {
        f32x2 dh[3], dl[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const size_t q0 = static_cast<size_t>(6 * p + k) * N, q1 = q0 + 3 * N;
          const f32x2 a = pack2(__ldg(u + q0 + w), __ldg(u + q1 + w));
          const f32x2 b = nown[3 * p + k];
          const f32x2 s = fadd2(a, b);                      // two-sum of u_(v+d) and -u_v
          const f32x2 bb = fsub2(s, a);
          const f32x2 e = fadd2(fsub2(a, fsub2(s, bb)), fsub2(b, bb));
          dh[k] = s;
          dl[k] = fadd2(e, fsub2(pack2(__ldg(ulo + q0 + w), __ldg(ulo + q1 + w)), ownlo[3 * p + k]));
        }
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            const f32x2 pr = fmul2(Ap[3 * r + k], dh[k]);
            const f32x2 npe = ffma2(An[3 * r + k], dh[k], pr);      // = -(a dh - p) exactly
            const f32x2 h = hi[3 * p + r];
            const f32x2 s = fadd2(h, pr);                            // two-sum of hi and p
            const f32x2 bb = fsub2(s, h);
            const f32x2 e = fadd2(fsub2(h, fsub2(s, bb)), fsub2(pr, bb));
            hi[3 * p + r] = s;
            // e + (a dl + pe) = e - (-a dl - pe) = e - fma(-a, dl, -pe)
            lo[3 * p + r] = fadd2(lo[3 * p + r], fsub2(e, ffma2(An[3 * r + k], dl[k], npe)));
          }
      }
    }
    float hs[kPlanes], ls[kPlanes];
#pragma unroll
    for (int p = 0; p < 3; ++p)
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        unpack2(hi[3 * p + r], hs[6 * p + r], hs[6 * p + 3 + r]);
        unpack2(lo[3 * p + r], ls[6 * p + r], ls[6 * p + 3 + r]);
      }
#pragma unroll
    for (int q = 0; q < kPlanes; ++q) {
      const size_t o = static_cast<size_t>(q) * N + v;
      float s, e;
      two_sum(__ldg(b + o), -hs[q], s, e);
      const float val = __fadd_rn(s, __fadd_rn(e, __fadd_rn(__ldg(blo + o), -ls[q])));
      out[o] = val;
      red[q / 3] = fmaf(val, val, red[q / 3]);
      red[kCases + q] += val;
    }
  }
  block_sum_store<kCases + kPlanes>(red, part);
}

// First Chebyshev step from x = 0: out_v = c0 S_v^-1 (b_v - bmean), S_v the diagonal
// block (the Gauss-Seidel diagonal solve of Eq. 16).
__global__ void __launch_bounds__(256) k_fine_jacobi_start(const __grid_constant__ KeParam K,
                                                           const float* __restrict__ E,
                                                           const float* __restrict__ b,
                                                           const float* __restrict__ bmean,
                                                           float* __restrict__ out, int n, float c0) {
  const size_t N = static_cast<size_t>(n) * n * n;
  for (size_t v = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; v < N;
       v += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const int x = static_cast<int>(v % n), y = static_cast<int>((v / n) % n),
              z = static_cast<int>(v / (static_cast<size_t>(n) * n));
    const Nb nb = make_nb(x, y, z, n);
    float Et[8];
    load_E8(E, nb, Et);
    float S[9];
    nb_block(K, Et, 0, 0, 0, S);
    float rhs[kPlanes];
#pragma unroll
    for (int q = 0; q < kPlanes; ++q)
      rhs[q] = __ldg(b + q * N + v) - (bmean ? __ldg(bmean + q) : 0.f);
    solve3x6(S, rhs);
#pragma unroll
    for (int q = 0; q < kPlanes; ++q) out[q * N + v] = c0 * rhs[q];
  }
}

// Level-0 stencil written out (used only when the finest level is also the coarsest and
// is solved directly): st[(9d + q) * N + pos(v)] = A_d[q].
__global__ void __launch_bounds__(256) k_fine_stencil(const __grid_constant__ KeParam K,
                                                      const float* __restrict__ E, int n, bool cb,
                                                      float* __restrict__ st) {
  const size_t N = static_cast<size_t>(n) * n * n;
  for (size_t v = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; v < N;
       v += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const int x = static_cast<int>(v % n), y = static_cast<int>((v / n) % n),
              z = static_cast<int>(v / (static_cast<size_t>(n) * n));
    const Nb nb = make_nb(x, y, z, n);
    float Et[8];
    load_E8(E, nb, Et);
    const size_t p = stencil_pos(x, y, z, n, cb);
#pragma unroll
    for (int d = 0; d < 27; ++d) {
      float A[9];
      nb_block(K, Et, d % 3 - 1, (d / 3) % 3 - 1, d / 9 - 1, A);
#pragma unroll
      for (int q = 0; q < 9; ++q) st[static_cast<size_t>(9 * d + q) * N + p] = A[q];
    }
  }
}

__global__ void k_simp(const float* __restrict__ rin, float* __restrict__ rout,
                       float* __restrict__ E, size_t N, float p, float E0, float Emin) {
  for (size_t e = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; e < N;
       e += static_cast<size_t>(gridDim.x) * blockDim.x) {
    float r = rin[e];
    r = fminf(fmaxf(r, 0.f), 1.f);
    rout[e] = r;
    E[e] = Emin + powf(r, p) * (E0 - Emin);
  }
}

struct ElemParam {
  float mu[kCases];           // eigenvalues of the symmetrised objective gradient G
  float vec[kCases][kCases];  // vec[k][i]: component i of the eigenvector of mu[k]
  float p, dE;                // SIMP exponent, E0 - Emin
  float invN;
};

struct KePairs {   // k[c][r] = (K0[r][c], K0[r][c]) for two-lane FMAs
  f32x2 k[24][24];
};

constexpr int kElemCases = kCases;            // one warp per load case
constexpr int kElemBlock = 32 * kElemCases;   // 32 lanes x 6 cases, two elements per lane
constexpr int kElemPad = 25;                  // w row stride in shared memory (bank spread)

// Pair slot of (i, j) in the row-major upper triangle of the 6x6 C^H (i <= j).
__host__ __device__ constexpr int pair_slot(int i, int j) {
  return i <= j ? i * kCases - i * (i - 1) / 2 + (j - i) : j * kCases - j * (j - 1) / 2 + (i - j);
}

// Per element q_ij = w_i^T K0 w_j, w_i = chi_i - (u_i - u_i at local vertex 0): the
// summand of Eq. 7 (subtracting the element's own translation leaves K0 w unchanged and
// keeps FP32 round-off independent of the field's magnitude, cf. Sec. 4.2 "relative
// coordinate"). Six threads per element, one per load case i and each in its own warp,
// so a warp's loads cover 32 consecutive elements: thread i gathers w_i (both parts of
// the double-float field), forms y_i = K0 w_i and the products q_ij = y_i . w_j of the
// pairs dealt to it (q_ij = q_ji: the diagonal, i+1, i+2 and, for i < 3, i+3 mod 6, so
// 3 or 4 each), reading the other w_j from shared memory.
// A thread takes its elements of two consecutive grid steps at once, on the two lanes of
// f32x2 registers (each lane rounded as the scalar chain): every constant of K0 (a pair in
// the parameter bank) and every instruction then serves two elements, where
// the scalar form spent an instruction per constant as well (1700 a thread and element, 850
// of them FMA-pipe). The rows of y come in two halves of 12, which keeps the registers
// at 2 blocks per SM. 192^3, C^H and sensitivities together: 5.27 -> 4.85 ms.
// MODE 0: block partial sums of E_e q_ij (21 values, Kahan-compensated per thread).
// MODE 1: sensitivity (Eq. 8-9) p rho^(p-1) dE sum_ij g_ij q_ij / N, evaluated as
// sum_k mu_k z_k^T K0 z_k with G = sym(g) = sum_k mu_k v_k v_k^T and z_k = sum_i v_k[i] w_i
// (thread k forms z_k from the six w_i in shared memory): each term is a non-negative
// quadratic form, so the sum does not cancel across the 21 products (for the bulk
// objective G has rank one and the sensitivity is a single quadratic form).
template <int MODE>
__global__ void __launch_bounds__(kElemBlock, 2) k_fine_elem(const __grid_constant__ KePairs K,
                                                             const __grid_constant__ ChiParam X,
                                                             const __grid_constant__ ElemParam P,
                                                             const float* __restrict__ E,
                                                             const float* __restrict__ rho,
                                                             const float* __restrict__ u,
                                                             const float* __restrict__ ulo, int n,
                                                             float* __restrict__ sens,
                                                             double* __restrict__ part) {
  __shared__ f32x2 ws[kElemCases][32][kElemPad];
  __shared__ f32x2 sp[kElemCases][32];
  __shared__ double sacc[21];
  const int lane = threadIdx.x & 31, i = threadIdx.x >> 5;   // element slot, load case
  const unsigned N = static_cast<unsigned>(n) * n * n;       // n <= 1024
  const int npair = i < 3 ? 4 : 3;
  int jp[4], slot[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    jp[k] = (i + k) % kCases;
    slot[k] = pair_slot(i, jp[k]);
  }
  float cs[4] = {0.f, 0.f, 0.f, 0.f}, cc[4] = {0.f, 0.f, 0.f, 0.f};
  const unsigned stride = gridDim.x * 32;
  const float* ui = u + static_cast<size_t>(3 * i) * N;
  const float* li = ulo + static_cast<size_t>(3 * i) * N;
  for (size_t e0 = static_cast<size_t>(blockIdx.x) * 32; e0 < N; e0 += 2 * static_cast<size_t>(stride)) {
    const size_t el[2] = {e0 + lane, e0 + lane + stride};
    const bool live[2] = {el[0] < N, el[1] < N};
    f32x2 w[24];
    {
      float wv[2][24];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const unsigned e = live[h] ? static_cast<unsigned>(el[h]) : 0u;
        int x, y, z;
        decode3(e, static_cast<unsigned>(n), x, y, z);
        const int xs[2] = {x, x == n - 1 ? 0 : x + 1};
        const int ys[2] = {y * n, (y == n - 1 ? 0 : y + 1) * n};
        const int zs[2] = {z * n * n, (z == n - 1 ? 0 : z + 1) * n * n};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const float* uq = ui + static_cast<size_t>(k) * N;
          const float* lq = li + static_cast<size_t>(k) * N;
          const float h0 = __ldg(uq + e), l0 = __ldg(lq + e);
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const unsigned vj = static_cast<unsigned>(xs[j & 1] + ys[(j >> 1) & 1] + zs[j >> 2]);
            const float du = (__ldg(uq + vj) - h0) + (__ldg(lq + vj) - l0);
            wv[h][3 * j + k] = live[h] ? X.chi[i][3 * j + k] - du : 0.f;
          }
        }
      }
#pragma unroll
      for (int r = 0; r < 24; ++r) w[r] = pack2(wv[0][r], wv[1][r]);
    }
#pragma unroll
    for (int r = 0; r < 24; ++r) ws[i][lane][r] = w[r];
    __syncthreads();
    if (MODE == 1) {   // z_k = sum_i v_k[i] w_i replaces w: thread i now stands for mode k = i
#pragma unroll
      for (int r = 0; r < 24; ++r) {
        f32x2 zr = 0ull;
#pragma unroll
        for (int c = 0; c < kCases; ++c) zr = ffma2(pack2(P.vec[i][c], P.vec[i][c]), ws[c][lane][r], zr);
        w[r] = zr;
      }
    }
    f32x2 q[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      f32x2 yv[12];
#pragma unroll
      for (int r = 0; r < 12; ++r) yv[r] = 0ull;
#pragma unroll
      for (int k = 0; k < 24; ++k) {
#pragma unroll
        for (int r = 0; r < 12; ++r) yv[r] = ffma2(K.k[k][12 * half + r], w[k], yv[r]);
      }
      if (MODE == 1) {
#pragma unroll
        for (int r = 0; r < 12; ++r) q[0] = ffma2(yv[r], w[12 * half + r], q[0]);
      } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          if (k < npair) {
            const f32x2* wj = ws[jp[k]][lane] + 12 * half;
#pragma unroll
            for (int r = 0; r < 12; ++r) q[k] = ffma2(yv[r], wj[r], q[k]);
          }
        }
      }
    }
    float qv[4][2];
#pragma unroll
    for (int k = 0; k < (MODE == 1 ? 1 : 4); ++k) unpack2(q[k], qv[k][0], qv[k][1]);
    if (MODE == 0) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (!live[h]) continue;
        const float Ee = __ldg(E + el[h]);
#pragma unroll
        for (int k = 0; k < 4; ++k) {   // Kahan summation of E_e q_e,k
          const float yk = fmaf(Ee, qv[k][h], -cc[k]);
          const float t = cs[k] + yk;
          cc[k] = (t - cs[k]) - yk;
          cs[k] = t;
        }
      }
    } else {
      sp[i][lane] = pack2(P.mu[i] * qv[0][0], P.mu[i] * qv[0][1]);
    }
    __syncthreads();
    const size_t eo = i == 0 ? el[0] : el[1];
    if (MODE == 1 && i < 2 && eo < N) {   // warp h finishes element h of each lane
      float sg = 0.f;
#pragma unroll
      for (int c = 0; c < kElemCases; ++c) {
        float v0, v1;
        unpack2(sp[c][lane], v0, v1);
        sg += i == 0 ? v0 : v1;
      }
      const float r = __ldg(rho + eo);
      sens[eo] = P.p * powf(r, P.p - 1.f) * P.dE * sg * P.invN;
    }
  }
  if (MODE == 0) {
    // each pair slot belongs to exactly one warp: reduce the warp's 32 sums per slot
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      float v = cs[k];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
      if (lane == 0 && k < npair) sacc[slot[k]] = static_cast<double>(v);
    }
    __syncthreads();
    if (threadIdx.x < 21) part[static_cast<size_t>(blockIdx.x) * 21 + threadIdx.x] = sacc[threadIdx.x];
  }
}

}  // namespace

cudaError_t launch_simp(const float* rho_in, float* rho_out, float* E, size_t N, float p,
                        float E0, float Emin, cudaStream_t s) {
  k_simp<<<grid_for(N, 256), 256, 0, s>>>(rho_in, rho_out, E, N, p, E0, Emin);
  return cudaGetLastError();
}

cudaError_t launch_fine_jacobi_start(const homo_ctx* c, const float* b, const float* bmean, float* out,
                                     float c0) {
  k_fine_jacobi_start<<<grid_for(c->N, 256), 256, 0, c->stream>>>(c->ke, c->E, b, bmean, out, c->n, c0);
  return cudaGetLastError();
}

cudaError_t launch_fine_stencil(const homo_ctx* c, const Level& L0) {
  k_fine_stencil<<<grid_for(c->N, 256), 256, 0, c->stream>>>(c->ke, c->E, c->n, L0.colour_blocked, L0.st);
  return cudaGetLastError();
}

cudaError_t launch_loads(const homo_ctx* c, float* f) {
  k_loads<<<grid_for(c->N, 256), 256, 0, c->stream>>>(c->ld, c->E, f, c->flo, c->n);
  return cudaGetLastError();
}

cudaError_t launch_fine_apply(const homo_ctx* c, const float* u, float* out, double* part,
                              int* grid_out) {
  return launch_fine_tiled(c, part ? 1 : 7, u, nullptr, out, part, grid_out);
}

cudaError_t launch_fine_residual(const homo_ctx* c, const float* b, const float* u,
                                 const float* ulo, float* out, double* part, int* grid_out,
                                 const float* bmean) {
  if (ulo) {
    const int g = grid_for(c->N, kTrueResThreads);
    if (grid_out) *grid_out = g;
    k_fine_true_residual<<<g, kTrueResThreads, 0, c->stream>>>(make_dblocks(c->ke), c->E, u, ulo, b, c->flo, out, c->n,
                                                               part);
    return cudaGetLastError();
  }
  return launch_fine_tiled(c, 3, u, b, out, nullptr, grid_out, bmean);
}


cudaError_t launch_fine_elem(const homo_ctx* c, int mode, const double* g36, float* sens,
                             double* part, int* grid_out) {
  ElemParam P{};
  if (g36) {   // sum_ij g_ij q_ij = sum_ij G_ij q_ij, G = (g + g^T) / 2 = sum_k mu_k v_k v_k^T
    double G[kCases * kCases], V[kCases * kCases];
    for (int i = 0; i < kCases; ++i)
      for (int j = 0; j < kCases; ++j) G[i * kCases + j] = 0.5 * (g36[6 * i + j] + g36[6 * j + i]);
    sym_eigen(kCases, G, V);
    for (int k = 0; k < kCases; ++k) {
      P.mu[k] = static_cast<float>(G[k * kCases + k]);
      for (int i = 0; i < kCases; ++i) P.vec[k][i] = static_cast<float>(V[i * kCases + k]);
    }
  }
  P.p = static_cast<float>(c->p);
  P.dE = static_cast<float>(c->E0 - c->Emin);
  P.invN = static_cast<float>(1.0 / static_cast<double>(c->N));
  const int g = grid_for((c->N + 31) / 32, 1);   // one block per 32 elements, capped
  if (grid_out) *grid_out = g;
  KePairs kp;
  for (int col = 0; col < 24; ++col)
    for (int row = 0; row < 24; ++row) {
      uint32_t b;
      std::memcpy(&b, &c->ke.k[row * 24 + col], 4);
      kp.k[col][row] = (static_cast<f32x2>(b) << 32) | b;
    }
  if (mode == 0)
    k_fine_elem<0><<<g, kElemBlock, 0, c->stream>>>(kp, c->chi, P, c->E, c->rho, c->u, c->ulo,
                                                   c->n, sens, part);
  else
    k_fine_elem<1><<<g, kElemBlock, 0, c->stream>>>(kp, c->chi, P, c->E, c->rho, c->u, c->ulo,
                                                   c->n, sens, part);
  return cudaGetLastError();
}

void set_thread_error(const std::string& msg);

// ---------------------------------------------------------------- allocation-free C^H
// A second way to evaluate C^H for callers that cannot allocate device memory while
// they run. Its per-block partial sums go to one fixed array in device memory that the
// library reserves when it is loaded, instead of to context buffers from cudaMalloc.
namespace {

constexpr int kNoAllocBlocks = 1216;   // partial-sum rows: 152 SMs x 8 blocks
constexpr int kNoAllocMaxN = 1024;     // largest cell per axis (indices stay in int)

// Rows 0..kNoAllocBlocks-1: 21 partial sums per block; last row: the 21 totals.
// Every GPU that loads the library holds this array (about 200 KB) until exit.
static __device__ __align__(256) double g_noalloc_scratch[(kNoAllocBlocks + 1) * 21];

std::mutex g_noalloc_mu;
double* g_noalloc_ptr[256] = {};   // device address of g_noalloc_scratch, per device

// Thread per element, its 144 w values and 21 products in a shared-memory row.
constexpr int kNoAllocElemBlock = 128;
constexpr int kNoAllocStride = 165;   // 144 w values + 21 products per thread row (odd: bank spread)

// The element arithmetic of Eq. 7 (w_i = chi_i - relative displacement, q_ij = w_i^T K0
// w_j, Kahan sums of E_e q_ij) with one thread per element; ulo may be null (read as 0).
__global__ void __launch_bounds__(kNoAllocElemBlock) k_ch_noalloc(const __grid_constant__ KeParam K,
                                                           const __grid_constant__ ChiParam X,
                                                           const float* __restrict__ E,
                                                           const float* __restrict__ u,
                                                           const float* __restrict__ ulo, int n,
                                                           double* __restrict__ scratch) {
  extern __shared__ float wsh[];
  float* w = wsh + threadIdx.x * kNoAllocStride;
  const size_t N = static_cast<size_t>(n) * n * n;
  float cs[21], cc[21];
#pragma unroll
  for (int k = 0; k < 21; ++k) cs[k] = cc[k] = 0.f;
  for (size_t e = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; e < N;
       e += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const int x = static_cast<int>(e % n), y = static_cast<int>((e / n) % n),
              z = static_cast<int>(e / (static_cast<size_t>(n) * n));
    const int xs[2] = {x, x == n - 1 ? 0 : x + 1};
    const int ys[2] = {y * n, (y == n - 1 ? 0 : y + 1) * n};
    const int zs[2] = {z * n * n, (z == n - 1 ? 0 : z + 1) * n * n};
#pragma unroll
    for (int q = 0; q < kPlanes; ++q) {
      const float* uq = u + static_cast<size_t>(q) * N;
      const float* lq = ulo ? ulo + static_cast<size_t>(q) * N : nullptr;
      const float h0 = __ldg(uq + e), l0 = lq ? __ldg(lq + e) : 0.f;
      const int c = q / 3, k = q % 3;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const size_t vj = static_cast<size_t>(xs[j & 1] + ys[(j >> 1) & 1] + zs[j >> 2]);
        const float du = (__ldg(uq + vj) - h0) + (lq ? (__ldg(lq + vj) - l0) : 0.f);
        w[c * 24 + 3 * j + k] = X.chi[c][3 * j + k] - du;
      }
    }
    float* q = w + 144;
#pragma unroll 1
    for (int i = 0, idx = 0; i < kCases; ++i) {
      float yv[24];
#pragma unroll
      for (int r = 0; r < 24; ++r) yv[r] = 0.f;
#pragma unroll
      for (int k = 0; k < 24; ++k) {
        const float wk = w[i * 24 + k];
#pragma unroll
        for (int r = 0; r < 24; ++r) yv[r] = fmaf(K.k[r * 24 + k], wk, yv[r]);
      }
#pragma unroll 1
      for (int j = i; j < kCases; ++j, ++idx) {
        float s = 0.f;
#pragma unroll
        for (int k = 0; k < 24; ++k) s = fmaf(yv[k], w[j * 24 + k], s);
        q[idx] = s;
      }
    }
    const float Ee = __ldg(E + e);
#pragma unroll
    for (int k = 0; k < 21; ++k) {
      const float yk = fmaf(Ee, q[k], -cc[k]);
      const float t = cs[k] + yk;
      cc[k] = (t - cs[k]) - yk;
      cs[k] = t;
    }
  }
  block_sum_store<21>(cs, scratch);
}

// totals[k] = sum over the nblk rows written by this call, fixed order.
__global__ void k_ch_noalloc_total(double* __restrict__ scratch, int nblk) {
  const int k = threadIdx.x;
  if (k >= 21) return;
  double s = 0.0;
  for (int b = 0; b < nblk; ++b) s += scratch[static_cast<size_t>(b) * 21 + k];
  scratch[static_cast<size_t>(kNoAllocBlocks) * 21 + k] = s;
}

int noalloc_fail(int code, const std::string& msg) {
  set_thread_error(msg);
  return code;
}

}  // namespace

}  // namespace homo

extern "C" int homo_CH_noalloc(int n, double nu, const float* E, const float* u, const float* ulo,
                               double CH[36], void* cuda_stream) {
  using namespace homo;
  if (n < 4 || n > kNoAllocMaxN)
    return noalloc_fail(HOMO_EINVAL, "homo_CH_noalloc: n = " + std::to_string(n) +
                                         " is outside [4, " + std::to_string(kNoAllocMaxN) +
                                         "], the largest cell its fixed scratch array serves");
  if (!(nu > -1.0 && nu < 0.5) || !E || !u || !CH)
    return noalloc_fail(HOMO_EINVAL, "homo_CH_noalloc: bad nu or null pointer");
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || dev < 0 || dev >= 256)
    return noalloc_fail(HOMO_ECUDA, std::string("homo_CH_noalloc: cudaGetDevice: ") + cudaGetErrorString(e));
  double* scratch = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
      void* p = nullptr;
      e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
      if (e != cudaSuccess || !p)
        return noalloc_fail(HOMO_ECUDA, std::string("homo_CH_noalloc: cudaGetSymbolAddress: ") +
                                            cudaGetErrorString(e));
      g_noalloc_ptr[dev] = static_cast<double*>(p);
    }
    scratch = g_noalloc_ptr[dev];
  }
  KeParam ke;
  LoadParam ld;
  ChiParam chi;
  build_element_matrix(nu, ke, ld, chi);
  const size_t N = static_cast<size_t>(n) * n * n;
  size_t blocks = (N + kNoAllocElemBlock - 1) / kNoAllocElemBlock;
  if (blocks > static_cast<size_t>(kNoAllocBlocks)) blocks = kNoAllocBlocks;
  const size_t shm = static_cast<size_t>(kNoAllocElemBlock) * kNoAllocStride * sizeof(float);
  e = cudaFuncSetAttribute(k_ch_noalloc, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(shm));
  if (e == cudaSuccess) {
    k_ch_noalloc<<<static_cast<int>(blocks), kNoAllocElemBlock, shm, s>>>(ke, chi, E, u, ulo, n, scratch);
    k_ch_noalloc_total<<<1, 32, 0, s>>>(scratch, static_cast<int>(blocks));
    e = cudaGetLastError();
  }
  double tot[21];
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(tot, scratch + static_cast<size_t>(kNoAllocBlocks) * 21, sizeof(tot),
                        cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess)
    return noalloc_fail(HOMO_ECUDA, std::string("homo_CH_noalloc: ") + cudaGetErrorString(e));
  const double invN = 1.0 / static_cast<double>(N);
  int idx = 0;
  for (int i = 0; i < kCases; ++i)
    for (int j = i; j < kCases; ++j) {
      CH[6 * i + j] = CH[6 * j + i] = tot[idx++] * invN;
    }
  return HOMO_OK;
}
