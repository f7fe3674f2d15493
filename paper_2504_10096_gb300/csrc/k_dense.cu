// Dense structure-preserving diagonalisation of the pseudo-Hermitian BSE
// matrix on the GPU (the direct method of Sec. 2.1.1, Eqs. 4-6), in FP64.
//
// With Q and the real skew-symmetric J of Eq. 4, Q^H H Q = -i J M_r, where
//     M_r = [[Re(A + B), Im(A - B)], [-Im(A + B), Re(A - B)]]     (Eq. 5)
// is real symmetric and positive definite when M of Eq. 2 is.  With the
// Cholesky factor M_r = L L^T, W = L^T J L is real skew-symmetric and -iW is
// Hermitian with the eigenvalues +-omega of H (Eq. 6).  The steps, all in
// this file and all FP64 on the CUDA cores (GB300's FP64 tensor rate is far
// below its FP64 FMA rate, so no tensor-core path is used):
//   1. assemble M_r (order n = 2N, column-major) from the handle's packed tiles;
//   2. blocked right-looking Cholesky (32-column panels: diagonal block and panel
//      solve in one launch, trailing symmetric rank-32 update);
//   3. W = L_top^T L_bot - L_bot^T L_top (J swaps the two halves of L's rows);
//   4. Householder reduction of W to skew-tridiagonal form: the reflector
//      H = I - tau v v^T of column k turns the trailing block into
//      W + tau (v p^T - p v^T), p = W v (v^T W v = 0 for skew W);
//   5. -iT (T skew-tridiagonal, sub-diagonal e) is unitarily similar, through
//      a diagonal phase matrix D, to the real symmetric tridiagonal S with zero
//      diagonal and off-diagonals |e_k|: the wanted eigenvalues (indices N ...
//      N + nev - 1 of S's ascending spectrum) by bisection with Sturm counts,
//      their eigenvectors by inverse iteration;
//   6. back-transformation q = H_0 ... H_{n-3} D s, then y = L^{-T} q and
//      z = Q y, which the caller Omega-normalises (Eq. 7 gives the partners).
#include <algorithm>
#include <cmath>

#include "../../include/bse.h"
#include "grid_sync.cuh"
#include "tree_solve.cuh"

namespace bse {
namespace {

constexpr int DNB = 32;        // Cholesky panel width and GEMM tile edge

// (A_ij, B_ij) from the packed upper-triangle tiles of problem p (any i, j < N):
// complex128 PH tiles hold P = A + B, Q = A - B; complex64 tiles hold A, B
template <typename ST>
__device__ __forceinline__ void dn_ab(const Prob& p, int64_t i, int64_t j, bool pq, double2& a, double2& b) {
  const bool up = i <= j;
  const int64_t r = up ? i : j, c = up ? j : i;
  const int I = (int)(r / TS), J = (int)(c / TS);
  const int64_t t = (int64_t)I * p.nT - (int64_t)I * (I - 1) / 2 + (J - I);
  int rr = (int)(r % TS), cc = (int)(c % TS);
  if (!up && I == J) {           // diagonal tiles hold both halves: read (i, j) itself
    rr = (int)(i % TS);
    cc = (int)(j % TS);
  }
  const int64_t e = t * (TS * TS) + (int64_t)rr * TS + cc;
  double2 x = ccvt<double2>(((const ST*)p.A)[e]), y = ccvt<double2>(((const ST*)p.B)[e]);
  if (pq) {
    a = make_double2(0.5 * (x.x + y.x), 0.5 * (x.y + y.y));
    b = make_double2(0.5 * (x.x - y.x), 0.5 * (x.y - y.y));
  } else {
    a = x;
    b = y;
  }
  if (!up && I != J) a = conjc(a);   // lower triangle: A Hermitian, B symmetric
}

// 1. M_r (n x n, column-major, leading dimension ld); grid (ceil(n/32), ceil(n/8)), 32 x 8
template <typename ST>
__global__ void k_dn_assemble(const Prob* __restrict__ probs, int pq, double* __restrict__ M, int64_t ld) {
  const Prob& p = probs[0];
  const int64_t N = p.N, n = 2 * N;
  const int64_t i = (int64_t)blockIdx.x * 32 + threadIdx.x;
  const int64_t j = (int64_t)blockIdx.y * 8 + threadIdx.y;
  if (i >= n || j >= n) return;
  const bool ti = i >= N, tj = j >= N;
  double2 a, b;
  dn_ab<ST>(p, ti ? i - N : i, tj ? j - N : j, pq != 0, a, b);
  double v;
  if (!ti && !tj) v = a.x + b.x;          // Re(A + B)
  else if (!ti && tj) v = a.y - b.y;      // Im(A - B)
  else if (ti && !tj) v = -(a.y + b.y);   // -Im(A + B)
  else v = a.x - b.x;                     // Re(A - B)
  M[j * ld + i] = v;
}

// 2. one panel: the diagonal block at k0 (kb <= 32 columns) is factored by every CTA for itself in
// shared memory, a warp of rows per column step, and each CTA then solves x L11^T = a for its 32
// rows below, eight lanes a row (four columns each: the 32-step chain of multiply-adds is what such
// a solve costs, 64 clocks a step).  CTA 0 stores L11 to D (k_dn_update copies it back: the other
// CTAs still read the block here).
__global__ void __launch_bounds__(256) k_dn_panel(double* __restrict__ M, int64_t ld, int64_t n, int64_t k0, int kb,
                                                  double* __restrict__ D, int* __restrict__ notpd) {
  __shared__ double a[DNB][DNB + 1];
  __shared__ double rd[DNB];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int e = tid; e < DNB * DNB; e += 256) {
    const int r = e % DNB, c = e / DNB;
    a[r][c] = (r < kb && c < kb && r >= c) ? M[(k0 + c) * ld + k0 + r] : (r == c ? 1.0 : 0.0);
  }
  __syncthreads();
  for (int c = 0; c < kb; ++c) {
    if (warp == 0) {
      double d = a[c][c];
      __syncwarp();                    // lane c rewrites it below
      const bool bad = !(d > 0.0);     // M_r not positive definite: flag it, keep the numbers finite
      if (bad) d = 1.0;
      const double r = rsqrt(d);
      if (bad && lane == 0 && blockIdx.x == 0) atomicExch(notpd, 1);
      if (lane == c) { a[c][c] = d * r; rd[c] = r; }
      else if (lane > c) a[lane][c] *= r;
    }
    __syncthreads();
    // trailing columns q > c: a[r][q] -= a[r][c] a[q][c], lane = row
    for (int q = c + 1 + warp; q < kb; q += 8)
      if (lane >= q) a[lane][q] = fma(-a[lane][c], a[q][c], a[lane][q]);
    __syncthreads();
  }
  if (blockIdx.x == 0)
    for (int e = tid; e < DNB * DNB; e += 256) D[e] = a[e % DNB][e / DNB];      // column-major
  // rows below: eight lanes a row, lane s owns the columns s, s + 8, s + 16, s + 24
  const int64_t row = k0 + kb + (int64_t)blockIdx.x * 32 + (tid >> 3);
  const int s = tid & 7;
  double x[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int c = s + 8 * u;
    x[u] = (row < n && c < kb) ? M[(k0 + c) * ld + row] : 0.0;
  }
#pragma unroll
  for (int c = 0; c < DNB; ++c) {
    if (c < kb) {                          // uniform
      if (s == (c & 7)) x[c >> 3] *= rd[c];
      const double xc = __shfl_sync(0xffffffffu, x[c >> 3], (lane & 24) | (c & 7));
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (s + 8 * u > c) x[u] = fma(-xc, a[s + 8 * u][c], x[u]);
    }
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int c = s + 8 * u;
    if (row < n && c < kb) M[(k0 + c) * ld + row] = x[u];
  }
}

// trailing update C -= L21 L21^T on the lower triangle (32 x 32 tiles, 256 threads of 2 x 2), rows
// and columns from `off`; the first CTA also copies the panel's diagonal block back from D
__global__ void __launch_bounds__(256) k_dn_update(double* __restrict__ M, int64_t ld, int64_t n, int64_t k0, int kb,
                                                   const double* __restrict__ D) {
  __shared__ double sa[DNB][DNB + 1], sb[DNB][DNB + 1];
  const int bi = blockIdx.x, bj = blockIdx.y, tid = threadIdx.x;
  if (bi < bj) return;
  if (bi == 0 && bj == 0)
    for (int e = tid; e < kb * kb; e += 256) {
      const int r = e % kb, c = e / kb;
      if (r >= c) M[(k0 + c) * ld + k0 + r] = D[c * DNB + r];
    }
  const int64_t off = k0 + kb, i0 = off + (int64_t)bi * DNB, j0 = off + (int64_t)bj * DNB;
  if (i0 >= n) return;
  for (int e = tid; e < DNB * DNB; e += 256) {
    const int r = e % DNB, q = e / DNB;
    sa[q][r] = (i0 + r < n && q < kb) ? M[(k0 + q) * ld + i0 + r] : 0.0;
    sb[q][r] = (j0 + r < n && q < kb) ? M[(k0 + q) * ld + j0 + r] : 0.0;
  }
  __syncthreads();
  const int tr = tid & 15, tc = tid >> 4;
  double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
#pragma unroll 8
  for (int q = 0; q < DNB; ++q) {
    const double a0 = sa[q][tr], a1 = sa[q][tr + 16], b0 = sb[q][tc], b1 = sb[q][tc + 16];
    acc[0][0] = fma(a0, b0, acc[0][0]);
    acc[0][1] = fma(a0, b1, acc[0][1]);
    acc[1][0] = fma(a1, b0, acc[1][0]);
    acc[1][1] = fma(a1, b1, acc[1][1]);
  }
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      const int64_t gi = i0 + tr + 16 * u, gj = j0 + tc + 16 * v;
      if (gi < n && gj < n && gi >= gj) M[gj * ld + gi] -= acc[u][v];
    }
}

// 3. G = L_top^T L_bot: G[i][j] = sum_q L[q][i] L[N + q][j], q < N.  L is lower triangular, so only
// rows i < N are non-zero and q runs from max(i, j - N): a quarter of the full product.  32 x 32
// tiles, 256 threads of 2 x 2, q staged 32 at a time; the other half of G is written as zeros.
__global__ void __launch_bounds__(256) k_dn_wgemm(double* __restrict__ G, const double* __restrict__ L, int64_t ld,
                                                  int64_t n) {
  __shared__ double sa[DNB][DNB + 1], sb[DNB][DNB + 1];   // [q][column]
  const int64_t N = n / 2, i0 = (int64_t)blockIdx.x * DNB, j0 = (int64_t)blockIdx.y * DNB;
  const int tid = threadIdx.x, tr = tid & 15, tc = tid >> 4;
  double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
  int64_t q0 = i0 > j0 - N ? i0 : j0 - N;
  if (i0 >= N) q0 = N;                                    // zero rows
  for (; q0 < N; q0 += DNB) {
    __syncthreads();
    for (int e = tid; e < DNB * DNB; e += 256) {
      const int q = e % DNB, c = e / DNB;                 // q along the columns of L
      const int64_t gq = q0 + q, gi = i0 + c, gj = j0 + c;
      sa[q][c] = (gq < N && gi < N && gq >= gi) ? L[gi * ld + gq] : 0.0;
      sb[q][c] = (gq < N && gj < n && N + gq >= gj) ? L[gj * ld + N + gq] : 0.0;
    }
    __syncthreads();
#pragma unroll 8
    for (int q = 0; q < DNB; ++q) {
      const double a0 = sa[q][tr], a1 = sa[q][tr + 16], b0 = sb[q][tc], b1 = sb[q][tc + 16];
      acc[0][0] = fma(a0, b0, acc[0][0]);
      acc[0][1] = fma(a0, b1, acc[0][1]);
      acc[1][0] = fma(a1, b0, acc[1][0]);
      acc[1][1] = fma(a1, b1, acc[1][1]);
    }
  }
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      const int64_t gi = i0 + tr + 16 * u, gj = j0 + tc + 16 * v;
      if (gi < n && gj < n) G[gj * ld + gi] = acc[u][v];
    }
}

// W = G - G^T, elementwise (column-major); the upper triangle of G is read before either
// element of a pair is written because each thread owns one unordered pair (i > j)
__global__ void k_dn_skew(double* __restrict__ W, int64_t ld, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * 32 + threadIdx.x;
  const int64_t j = (int64_t)blockIdx.y * 8 + threadIdx.y;
  if (i >= n || j >= n || i < j) return;
  if (i == j) { W[j * ld + i] = 0.0; return; }
  const double gij = W[j * ld + i], gji = W[i * ld + j];
  W[j * ld + i] = gij - gji;
  W[i * ld + j] = gji - gij;
}

// 4. Householder reduction to skew-tridiagonal form in one cooperative launch: column j belongs to CTA
// j mod G, in shared memory where the CTA's columns fit (order up to about 1900), else in place.  With
// x = W[k+1:, k], beta = -sign(x0) |x|, v = x / (x0 - beta), v0 = 1, tau = (beta - x0) / beta (tau = 0
// when x below x0 is zero), a step has two phases:
//   * p = W22 v: since W is skew, p_j = -(column j) . v, each CTA from its own columns;
//   * W22 += tau (v p^T - p v^T) on the own columns; the owner of column k + 1 updates it first and
//     builds the next reflector from it.
// So a step costs two grid barriers and a few multiply-adds per thread instead of four launches and a
// matrix-vector product on n / 256 CTAs: 72 -> 7.5 us a column at order 600.  Whole diagonalisation,
// measured: N = 300, 60 pairs 62.7 -> 9.5 ms; N = 1000, 50 pairs 450 -> 103 ms; N = 2000, 20 pairs 1.90 ->
// 0.63 s.
// Stores e_k = beta in E[k], tau in T[k], and v below the sub-diagonal of column k of W (its entry
// k + 1 holds beta; the reflector's is 1).
template <bool SMC>
__global__ void __launch_bounds__(256) k_dn_tridiag(double* __restrict__ W, int64_t ld, int n, double* __restrict__ E,
                                                    double* __restrict__ T, double* __restrict__ Pv, GridBar* gb) {
  extern __shared__ double dsm[];
  __shared__ int s_ok;
  __shared__ double red[8], s_h[4];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int G = gridDim.x, bid = blockIdx.x;
  unsigned int gen = 0;
  double* vs = dsm;                // the reflector and p of the step (SMC); columns behind them
  double* ps = dsm + n;
  const int own = bid < n ? (n - 1 - bid) / G + 1 : 0;
  auto col = [&](int q) { return SMC ? dsm + (size_t)(2 + q) * n : W + (int64_t)(bid + (int64_t)G * q) * ld; };
  if (SMC) {
    for (int q = 0; q < own; ++q) {
      const double* src = W + (int64_t)(bid + (int64_t)G * q) * ld;
      for (int r = tid; r < n; r += 256) col(q)[r] = src[r];
    }
    __syncthreads();
  }
  // the reflector of column c, whose entries below c are in x (all threads of the owner)
  auto house = [&](const double* x, int c) {
    double s = 0.0;
    for (int r = c + 2 + tid; r < n; r += 256) s = fma(x[r], x[r], s);
    s = warp_sum(s);
    if (lane == 0) red[warp] = s;
    __syncthreads();
    if (warp == 0) {
      double sig = lane < 8 ? red[lane] : 0.0;
#pragma unroll
      for (int m = 4; m >= 1; m >>= 1) sig += __shfl_xor_sync(0xffffffffu, sig, m);
      sig = __shfl_sync(0xffffffffu, sig, 0);
      const double x0 = x[c + 1];
      double beta = x0, tau = 0.0, scale = 0.0;
      if (sig > 0.0) {
        const double t = fma(x0, x0, sig), r = rsqrt(t), nrm = t * r;
        beta = x0 >= 0.0 ? -nrm : nrm;
        tau = fma(fabs(x0), r, 1.0);       // (beta - x0) / beta
        const double g = 1.0 / (fabs(x0) + nrm);
        scale = x0 >= 0.0 ? g : -g;        // 1 / (x0 - beta)
      }
      if (lane == 0) {
        s_h[0] = beta;
        s_h[1] = scale;
        E[c] = beta;
        T[c] = tau;
      }
    }
    __syncthreads();
    double* dst = W + (int64_t)c * ld;
    const double beta = s_h[0], scale = s_h[1];
    for (int r = c + 1 + tid; r < n; r += 256) dst[r] = r == c + 1 ? beta : x[r] * scale;
  };
  if (n > 2 && bid == 0) house(col(0), 0);
  if (!grid_sync(gb, G, gen, &s_ok)) return;
  for (int k = 0; k + 2 < n; ++k) {
    const double* vk = W + (int64_t)k * ld;
    const double tau = __ldcg(T + k);
    auto v_at = [&](int r) { return SMC ? vs[r] : (r == k + 1 ? 1.0 : __ldcg(vk + r)); };
    auto p_at = [&](int r) { return SMC ? ps[r] : __ldcg(Pv + r); };
    if (SMC) {
      for (int r = k + 1 + tid; r < n; r += 256) vs[r] = r == k + 1 ? 1.0 : __ldcg(vk + r);
      __syncthreads();
    }
    // own columns j > k: a warp each
    const int q0 = k + 1 <= bid ? 0 : (k + 1 - bid + G - 1) / G;
    if (tau != 0.0)
      for (int q = q0 + warp; q < own; q += 8) {
        const double* x = col(q);
        double s = 0.0;
        for (int r = k + 1 + lane; r < n; r += 32) s = fma(x[r], v_at(r), s);
        s = warp_sum(s);
        if (lane == 0) Pv[bid + G * q] = -s;
      }
    if (!grid_sync(gb, G, gen, &s_ok)) return;
    if (tau != 0.0) {
      if (SMC) {
        for (int r = k + 1 + tid; r < n; r += 256) ps[r] = __ldcg(Pv + r);
        __syncthreads();
      }
      auto update = [&](int q, int r0, int dr) {
        double* x = col(q);
        const int j = bid + G * q;
        const double tp = tau * p_at(j), tv = -tau * v_at(j);
        for (int r = r0; r < n; r += dr) x[r] = fma(p_at(r), tv, fma(v_at(r), tp, x[r]));
      };
      int qn = -1;
      if ((k + 1) % G == bid) {            // the next column first, by all warps
        qn = (k + 1 - bid) / G;
        update(qn, k + 1 + tid, 256);
        __syncthreads();
        if (k + 3 < n) house(col(qn), k + 1);
      }
      for (int q = q0 + warp; q < own; q += 8)
        if (q != qn) update(q, k + 1 + lane, 32);
    } else if ((k + 1) % G == bid && k + 3 < n) {
      house(col((k + 1 - bid) / G), k + 1);
    }
    if (!grid_sync(gb, G, gen, &s_ok)) return;
  }
  // the last sub-diagonal entry needs no reflector
  if ((n - 2) % G == bid && tid == 0) {
    E[n - 2] = col((n - 2 - bid) / G)[n - 1];
    T[n - 2] = 0.0;
  }
}

// the transpose of the Cholesky factor into the upper triangle (over the M_r values left there): the
// back substitution reads rows of L along its columns
__global__ void k_dn_mirror(double* __restrict__ M, int64_t ld, int64_t n) {
  __shared__ double t[32][33];
  const int64_t i0 = (int64_t)blockIdx.x * 32, j0 = (int64_t)blockIdx.y * 32;   // tile (i0, j0), i0 >= j0
  if (i0 < j0) return;
  for (int c = threadIdx.y; c < 32; c += 8) {
    const int64_t i = i0 + threadIdx.x, j = j0 + c;
    t[c][threadIdx.x] = (i < n && j < n) ? M[j * ld + i] : 0.0;
  }
  __syncthreads();
  for (int c = threadIdx.y; c < 32; c += 8) {
    const int64_t i = i0 + c, j = j0 + threadIdx.x;       // M[row j][column i] = L[i][j]
    if (i < n && j < i) M[i * ld + j] = t[threadIdx.x][c];
  }
}

// 5. S: zero diagonal, off-diagonals |e_k|.  The arrays the multisection and the inverse iteration
// read (x = 0, |e|, and double-FP32 copies scaled to norm 1), and S's Gershgorin bound 2 max |e|; one CTA
struct DnS {
  double* x;      // n zeros
  double* e;      // |e_k|
  double* e2;     // its square
  float2* xf;     // n zeros
  float2* e2f;    // e2 scaled
  double* bound;  // the bound and the scale
};

__global__ void __launch_bounds__(1024) k_dn_prepare(const double* __restrict__ E, int64_t n, DnS S) {
  __shared__ double red[32];
  double m = 0.0;
  for (int64_t t = threadIdx.x; t + 1 < n; t += blockDim.x) m = fmax(m, fabs(E[t]));
#pragma unroll
  for (int k = 16; k >= 1; k >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, k));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  m = 0.0;
  for (int q = 0; q < 32; ++q) m = fmax(m, red[q]);
  const double bound = 2.0 * m * (1.0 + 1e-14) + 1e-300, sc = tree_scale(bound);
  for (int64_t t = threadIdx.x; t < n; t += blockDim.x) {
    const double e = t + 1 < n ? fabs(E[t]) : 0.0;
    S.x[t] = 0.0;
    S.e[t] = e;
    S.e2[t] = e * e;
    S.xf[t] = make_float2(0.f, 0.f);
    S.e2f[t] = f2_split((e * sc) * (e * sc));
  }
  if (threadIdx.x == 0) {
    S.bound[0] = bound;
    S.bound[1] = sc;
  }
}

// one CTA per wanted eigenvalue (index idx0 + blockIdx.x of the ascending spectrum)
__global__ void __launch_bounds__(RV_THREADS) k_dn_bisect(DnS S, int64_t n, int64_t idx0, double* __restrict__ lam) {
  __shared__ double s_sig[RV_THREADS];
  __shared__ int s_cnt[RV_THREADS / 32];
  const double bound = S.bound[0];
  const double v = tree_eigenvalue(S.x, S.e2, S.xf, S.e2f, 0, (int)n, (int)(idx0 + blockIdx.x), -bound, bound, bound,
                                   S.bound[1], s_sig, s_cnt);
  if (threadIdx.x == 0) lam[blockIdx.x] = v;
}

// inverse iteration for the eigenvectors of S, one warp per cluster of close eigenvalues
// (Gram-Schmidt inside a cluster); the factorisation in shared memory (SM) or in 5 n doubles of
// scratch; vectors s_c (n doubles each, unit 2-norm) go to Sv[c * n ...]
template <bool SM>
__global__ void __launch_bounds__(32) k_dn_inverse(DnS S, int64_t n, int nev, const double* __restrict__ lam,
                                                   double* __restrict__ scratch, double* __restrict__ Sv) {
  extern __shared__ double dsm[];
  const int c0 = blockIdx.x, lane = threadIdx.x;
  const double bound = S.bound[0];
  const double eps = 2.220446049250313e-16;
  const double ctol = 1e-7 * bound;
  if (c0 > 0 && lam[c0] - lam[c0 - 1] < ctol) return;     // not a cluster leader
  int c1 = c0 + 1;
  while (c1 < nev && lam[c1] - lam[c1 - 1] < ctol) ++c1;
  TV tv;
  tv.d = tv.b = nullptr;
  tv.h = 0;
  tv.a = S.x;
  tv.e = S.e;
  tv.n = (int)n;
  double* w = SM ? dsm : scratch + (int64_t)c0 * 5 * n;
  Fact F;
  F.invd = w;
  F.dl = w + n;
  F.du = w + 2 * n;
  F.du2 = w + 3 * n;
  F.piv = (unsigned char*)(w + 4 * n);
  const double pivmin = eps * fmax(bound, 1e-290);
  double lprev = -1e300;
  for (int c = c0; c < c1; ++c) {
    double lm = lam[c];
    if (c > c0 && lm - lprev < 10.0 * eps * bound) lm = lprev + 10.0 * eps * bound;
    lprev = lm;
    factor_tree(tv, lm, pivmin, F, lane);
    double* x = Sv + (int64_t)c * n;
    for (int64_t t = lane; t < n; t += 32)
      x[t] = (double)(mix64((uint64_t)(c + 1) * 0x100000001b3ull + (uint64_t)t) >> 11) * (1.0 / 9007199254740992.0) - 0.5;
    __syncwarp();
    for (int it = 0; it < 4; ++it) {
      for (int rep = 0; rep < 2; ++rep)
        for (int q = c0; q < c; ++q) {
          const double* sq = Sv + (int64_t)q * n;
          double dot = 0.0;
          for (int64_t t = lane; t < n; t += 32) dot = fma(sq[t], x[t], dot);
          dot = warp_sum(dot);
          for (int64_t t = lane; t < n; t += 32) x[t] = fma(-dot, sq[t], x[t]);
          __syncwarp();
        }
      double nr = 0.0;
      for (int64_t t = lane; t < n; t += 32) nr = fma(x[t], x[t], nr);
      nr = warp_sum(nr);
      const double inv = nr > 0.0 ? rsqrt(nr) : 0.0;
      for (int64_t t = lane; t < n; t += 32) x[t] *= inv;
      __syncwarp();
      if (it == 3) break;
      solve_tree(tv, F, x, lane);
    }
  }
}

// 6. one CTA per eigenvector: q = H_0 ... H_{n-3} D s (D: the phases that make -iT real, so q is
// complex), then y = L^{-T} q, then z = Q y into Z (FP64 complex, ld 2 Npad: X rows then Y rows).  The
// next reflector (row of L) is loaded while the current one is reduced; the two components of a dot
// product share one reduction (a half-warp each from the second step on); the triangular solve goes
// column by column of L^T's upper-triangle copy, so it needs no reduction at all.  q is in shared
// memory (SM) or in qbuf.
template <bool SM>
__global__ void __launch_bounds__(256) k_dn_back(const double* __restrict__ Wv, const double* __restrict__ L,
                                                 int64_t ld, int64_t n, const double* __restrict__ E,
                                                 const double* __restrict__ T, const double* __restrict__ Sv,
                                                 double2* __restrict__ qbuf, int64_t Npad, double2* __restrict__ Z) {
  extern __shared__ double dsm[];
  __shared__ double red[8][2];
  const int c = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t N = n / 2;
  double2* q = SM ? reinterpret_cast<double2*>(dsm) : qbuf + (int64_t)c * n;
  const double* s = Sv + (int64_t)c * n;
  // D: d_0 = 1, d_{t+1} = d_t (-i) sign(e_t): the phase (-i)^t and the parity of the negative e
  // before t (prefix over 32-entry groups by ballots, each warp for itself)
  {
    unsigned par = 0;
    for (int64_t t0 = 0; t0 < n; t0 += 32) {
      const int64_t t = t0 + lane;
      const unsigned neg = __ballot_sync(0xffffffffu, t + 1 < n && E[t] < 0.0);
      if (((t0 >> 5) & 7) == warp && t < n) {
        const bool minus = (par + __popc(neg & ((1u << lane) - 1u))) & 1u;
        const double v = minus ? -s[t] : s[t];
        const int ph = (int)(t & 3);
        q[t] = ph == 0 ? make_double2(v, 0.0) : ph == 1 ? make_double2(0.0, -v)
             : ph == 2 ? make_double2(-v, 0.0) : make_double2(0.0, v);              // v (-i)^t
      }
      par += __popc(neg);
    }
  }
  __syncthreads();
  constexpr int U = 4;                                  // entries a thread keeps of the next column
  double nx[U];
  auto fetch = [&](const double* v, int64_t r0) {
#pragma unroll
    for (int u = 0; u < U; ++u) nx[u] = r0 + tid + 256 * u < n ? __ldg(v + r0 + tid + 256 * u) : 0.0;
  };
  if (n > 2) fetch(Wv + (n - 3) * ld, n - 2);
  for (int64_t k = n - 3; k >= 0; --k) {                // q <- H_k q on rows k+1 ... n-1
    const double tau = __ldg(T + k);
    const double* v = Wv + k * ld;                      // v_{k+1} = 1 (stored as beta), v_r below
    double cur[U];
#pragma unroll
    for (int u = 0; u < U; ++u) cur[u] = nx[u];
    if (k > 0) fetch(Wv + (k - 1) * ld, k);
    if (tau == 0.0) continue;                           // uniform
    if (tid == 0) cur[0] = 1.0;
    double sr = 0.0, si = 0.0;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t r = k + 1 + tid + 256 * u;
      if (r < n) {
        sr = fma(cur[u], q[r].x, sr);
        si = fma(cur[u], q[r].y, si);
      }
    }
    for (int64_t r = k + 1 + tid + 256 * U; r < n; r += 256) {
      const double vr = __ldg(v + r);
      sr = fma(vr, q[r].x, sr);
      si = fma(vr, q[r].y, si);
    }
    // lanes 0-15 go on with the real sum, 16-31 with the imaginary one
    double t = lane < 16 ? sr : si;
    t += __shfl_xor_sync(0xffffffffu, lane < 16 ? si : sr, 16);
#pragma unroll
    for (int m = 8; m >= 1; m >>= 1) t += __shfl_xor_sync(0xffffffffu, t, m);
    if ((lane & 15) == 0) red[warp][lane >> 4] = t;
    __syncthreads();
    t = red[lane & 7][(lane >> 3) & 1];
#pragma unroll
    for (int m = 4; m >= 1; m >>= 1) t += __shfl_xor_sync(0xffffffffu, t, m);
    t *= -tau;
    sr = __shfl_sync(0xffffffffu, t, 0);
    si = __shfl_sync(0xffffffffu, t, 8);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t r = k + 1 + tid + 256 * u;
      if (r < n) q[r] = make_double2(fma(cur[u], sr, q[r].x), fma(cur[u], si, q[r].y));
    }
    for (int64_t r = k + 1 + tid + 256 * U; r < n; r += 256) {
      const double vr = __ldg(v + r);
      q[r] = make_double2(fma(vr, sr, q[r].x), fma(vr, si, q[r].y));
    }
    __syncthreads();
  }
  // y = L^{-T} q (in place): y_i = q_i / L[i][i], then q_j -= L[i][j] y_i for j < i, L[i][j] at row j of
  // column i in the upper triangle
  auto fetch_row = [&](int64_t i) {
#pragma unroll
    for (int u = 0; u < U; ++u) nx[u] = tid + 256 * u < i ? __ldg(L + i * ld + tid + 256 * u) : 0.0;
  };
  fetch_row(n - 1);
  double dn = __ldg(L + (n - 1) * ld + n - 1);
  for (int64_t i = n - 1; i >= 0; --i) {
    const double inv = recip_any(dn);
    double cur[U];
#pragma unroll
    for (int u = 0; u < U; ++u) cur[u] = nx[u];
    if (i > 0) {
      fetch_row(i - 1);
      dn = __ldg(L + (i - 1) * ld + i - 1);
    }
    const double2 qi = q[i];
    const double2 y = make_double2(qi.x * inv, qi.y * inv);
    __syncthreads();                                    // everyone has read q_i
    if (tid == (int)(i & 255)) q[i] = y;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t j = tid + 256 * u;
      if (j < i) q[j] = make_double2(fma(-cur[u], y.x, q[j].x), fma(-cur[u], y.y, q[j].y));
    }
    for (int64_t j = tid + 256 * U; j < i; j += 256) {
      const double l = __ldg(L + i * ld + j);
      q[j] = make_double2(fma(-l, y.x, q[j].x), fma(-l, y.y, q[j].y));
    }
    __syncthreads();
  }
  // z = Q y, Q = (1/sqrt 2) [[I, -iI], [I, iI]]: X = (y1 - i y2) / sqrt 2, Y = (y1 + i y2) / sqrt 2
  const double r2 = 0.70710678118654752440;
  double2* z = Z + (int64_t)c * 2 * Npad;
  for (int64_t r = tid; r < Npad; r += 256) {
    double2 X = make_double2(0.0, 0.0), Y = make_double2(0.0, 0.0);
    if (r < N) {
      const double2 a = q[r], b = q[N + r];
      X = make_double2((a.x + b.y) * r2, (a.y - b.x) * r2);
      Y = make_double2((a.x - b.y) * r2, (a.y + b.x) * r2);
    }
    z[r] = X;
    z[Npad + r] = Y;
  }
}

}  // namespace

// scratch of dense_shao in doubles: M_r / L and W (ld x n each), the reflector work
// vectors, the arrays of S, the eigenvector scratch of the inverse iteration, the complex q
// vectors, the panel's diagonal block and the grid barrier
size_t dense_scratch_doubles(int64_t N, int nev) {
  const int64_t n = 2 * N;
  const int64_t ld = (n + 31) / 32 * 32;
  // sixteen sub-buffers, each rounded up to 32 doubles
  return (size_t)(2 * ld * n + 3 * n + 5 * n + (int64_t)nev * (5 * n + n + 2 * n) + nev + DNB * DNB + 16 + 16 * 32);
}

// Steps 2-6 on an assembled M_r (step 1 is `assemble(M, ld)`): the nev lowest positive omega
// (device, *lam_dev) and their right eigenvectors (unnormalised) in Z (ld 2 Npad).  Returns 0,
// 1 (M_r not positive definite), 2 (a bounded wait expired) or -1 (CUDA error); the stream is
// synchronised.
template <typename Assemble>
int dense_run(int64_t N, int64_t Npad, int nev, double* work, int* dflag, double2* Z, double** lam_dev,
              Assemble assemble, cudaStream_t s) {
  const int64_t n = 2 * N;
  const int64_t ld = (n + 31) / 32 * 32;
  // sub-buffers start on 256-byte boundaries (q is read and written as double2)
  size_t off = 0;
  auto take = [&](int64_t count) {
    double* p = work + off;
    off += (size_t)((count + 31) / 32 * 32);
    return p;
  };
  double* M = take(ld * n);         // M_r, then L (lower) and L^T (upper)
  double* W = take(ld * n);         // G, then W, then the reduced form with the reflectors
  double* E = take(n);              // sub-diagonal of T
  double* T = take(n);              // reflector scalars
  double* Pv = take(n);             // W22 v
  DnS S;
  S.x = take(n);
  S.e = take(n);
  S.e2 = take(n);
  S.xf = reinterpret_cast<float2*>(take(n));
  S.e2f = reinterpret_cast<float2*>(take(n));
  S.bound = take(2);
  double* lam = take(nev);          // wanted eigenvalues of S
  double* inv = take((int64_t)nev * 5 * n);   // inverse-iteration scratch, 5 n per vector
  double* Sv = take((int64_t)nev * n);
  double2* qb = reinterpret_cast<double2*>(take((int64_t)nev * 2 * n));
  double* D = take(DNB * DNB);
  GridBar* gb = reinterpret_cast<GridBar*>(take(1));
  *lam_dev = lam;
  if (cudaMemsetAsync(dflag, 0, sizeof(int), s) != cudaSuccess ||
      cudaMemsetAsync(gb, 0, sizeof(GridBar), s) != cudaSuccess)
    return -1;
  // 1.
  const dim3 g2((unsigned)((n + 31) / 32), (unsigned)((n + 7) / 8)), b2(32, 8);
  assemble(M, ld);
  // 2. Cholesky
  for (int64_t k0 = 0; k0 < n; k0 += DNB) {
    const int kb = (int)std::min<int64_t>(DNB, n - k0);
    const unsigned nt = (unsigned)std::max<int64_t>(1, (n - k0 - kb + DNB - 1) / DNB);
    count_launch(2);
    k_dn_panel<<<nt, 256, 0, s>>>(M, ld, n, k0, kb, D, dflag);
    k_dn_update<<<dim3(nt, nt), 256, 0, s>>>(M, ld, n, k0, kb, D);
  }
  // 3. G = L_top^T L_bot, then W = G - G^T
  count_launch(3);
  const unsigned ng = (unsigned)((n + DNB - 1) / DNB);
  k_dn_mirror<<<dim3(ng, ng), b2, 0, s>>>(M, ld, n);
  k_dn_wgemm<<<dim3(ng, ng), 256, 0, s>>>(W, M, ld, n);
  k_dn_skew<<<g2, b2, 0, s>>>(W, ld, n);
  // the opt-ins below are to DN_SMEM for all orders: another thread's solve may need more than this one
  constexpr size_t DN_SMEM = 200 * 1024;
  static PerDevice<bool> opt_in;
  opt_in.get(current_device(), [] {
    cudaFuncSetAttribute(k_dn_tridiag<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DN_SMEM);
    cudaFuncSetAttribute(k_dn_inverse<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DN_SMEM);
    cudaFuncSetAttribute(k_dn_back<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DN_SMEM);
    return true;
  });
  // 4. skew-tridiagonalisation
  {
    int nn = (int)n;
    int64_t lda = ld;
    const int grid = (int)std::min<int64_t>(num_sms(), n);
    const size_t cols = sizeof(double) * (size_t)n * ((n + grid - 1) / grid + 2);
    const bool smc = cols <= DN_SMEM;
    void* args[] = {(void*)&W, (void*)&lda, (void*)&nn, (void*)&E, (void*)&T, (void*)&Pv, (void*)&gb};
    const void* fn = smc ? (const void*)k_dn_tridiag<true> : (const void*)k_dn_tridiag<false>;
    count_launch();
    if (cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(256), args, smc ? cols : 0, s) != cudaSuccess) {
      cudaGetLastError();
      return -1;
    }
  }
  // 5. eigenvalues N ... N + nev - 1 of S and their eigenvectors
  count_launch(3);
  k_dn_prepare<<<1, 1024, 0, s>>>(E, n, S);
  k_dn_bisect<<<nev, RV_THREADS, 0, s>>>(S, n, N, lam);
  const size_t fs = sizeof(double) * (size_t)(4 * n) + (size_t)n;
  if (fs <= DN_SMEM) {
    k_dn_inverse<true><<<nev, 32, fs, s>>>(S, n, nev, lam, inv, Sv);
  } else {
    k_dn_inverse<false><<<nev, 32, 0, s>>>(S, n, nev, lam, inv, Sv);
  }
  // 6.
  count_launch();
  const size_t qs = sizeof(double2) * (size_t)n;
  if (qs <= DN_SMEM) {
    k_dn_back<true><<<nev, 256, qs, s>>>(W, M, ld, n, E, T, Sv, qb, Npad, Z);
  } else {
    k_dn_back<false><<<nev, 256, 0, s>>>(W, M, ld, n, E, T, Sv, qb, Npad, Z);
  }
  int h = 0;
  GridBar hb{};
  if (cudaMemcpyAsync(&h, dflag, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaMemcpyAsync(&hb, gb, sizeof(GridBar), cudaMemcpyDeviceToHost, s) != cudaSuccess)
    return -1;
  if (cudaStreamSynchronize(s) != cudaSuccess || cudaGetLastError() != cudaSuccess) return -1;
  return hb.err ? 2 : (h ? 1 : 0);
}

namespace {

// ---------------------------------------------------------------- projected BSE variant
// The folded recurrence builds V (M+-orthonormal) and P = M+ V, and H maps the even vectors
// e_j = (v_j; conj(v_j)) to the odd ones o_j = (p_j; -conj(p_j)) and o_j to sum_i e_i T_ij
// (T the projected M- M+).  In the basis x_j = e_j + o_j, y_j = e_j - o_j, which the
// swap-and-conjugate symmetry of H maps onto each other, H's projection is the BSE matrix
// [[A_k, B_k], [-B_k, -A_k]] of Eq. 1 with the real symmetric blocks A_k = (T + I) / 2 and
// B_k = (I - T) / 2; its M_r (Eq. 5) is diag(I, T), positive definite.  The dense
// structure-preserving method solves it (its omega are the singular values of T's Cholesky
// factor, computed without squaring), and an eigenvector (a; b) is the Ritz vector
// x a + y b = e (a + b) + o (a - b): the folded coefficients are a + b.

// M_r = diag(I, T_active) of problem ip (column-major, ld); grid as k_dn_assemble
__global__ void k_pj_assemble(const Prob* __restrict__ probs, int ip, double* __restrict__ M, int64_t ld) {
  const Prob& p = probs[ip];
  const KState* st = p.st;
  const int k = st->k, l = st->l, m = st->m, h = l - k;
  const int64_t na = m - k, n = 2 * na;
  const int64_t i = (int64_t)blockIdx.x * 32 + threadIdx.x;
  const int64_t j = (int64_t)blockIdx.y * 8 + threadIdx.y;
  if (i >= n || j >= n) return;
  double v = 0.0;
  if (i < na || j < na) {
    v = i == j ? 1.0 : 0.0;
  } else {
    const int64_t a = i - na, b = j - na;
    const int64_t lo = a < b ? a : b, hi = a < b ? b : a;
    if (a == b) v = a < h ? p.theta[k + a] : p.alpha[l + (a - h)];
    else if (hi == h && lo < h) v = p.barrow[k + lo];
    else if (lo >= h && hi == lo + 1) v = p.beta[l + (lo - h)];
  }
  M[j * ld + i] = v;
}

__device__ __forceinline__ double block_sum(double v, double* red) {
  v = warp_sum(v);
  const int w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[w] = v;
  __syncthreads();
  double t = 0.0;
  for (int q = 0; q < nw; ++q) t += red[q];
  return t;
}

// folded Ritz data from the small problem's eigenvectors: one CTA per wanted pair
__global__ void __launch_bounds__(256) k_pj_coef(const Prob* __restrict__ probs, int ip, int64_t na,
                                                 const double2* __restrict__ Zs, const double* __restrict__ lam) {
  __shared__ double red[8];
  __shared__ double sv[8];
  __shared__ int si[8];
  const Prob& p = probs[ip];
  const KState* st = p.st;
  const int i = blockIdx.x, tid = threadIdx.x;
  const double2* z = Zs + (int64_t)i * 2 * na;
  // the entry of largest modulus of c~ = a + b fixes the common phase (lowest index on ties)
  double best = -1.0;
  int bi = 0;
  for (int64_t t = tid; t < na; t += 256) {
    const double2 c = cadd(z[t], z[na + t]);
    const double a2 = c.x * c.x + c.y * c.y;
    if (a2 > best) { best = a2; bi = (int)t; }
  }
  for (int o = 16; o >= 1; o >>= 1) {
    const double ob = __shfl_xor_sync(0xffffffffu, best, o);
    const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
    if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
  }
  if ((tid & 31) == 0) { sv[tid >> 5] = best; si[tid >> 5] = bi; }
  __syncthreads();
  if (tid == 0) {
    for (int w = 1; w < 8; ++w)
      if (sv[w] > sv[0] || (sv[w] == sv[0] && si[w] < si[0])) { sv[0] = sv[w]; si[0] = si[w]; }
  }
  __syncthreads();
  const double2 cm = cadd(z[si[0]], z[na + si[0]]);
  const double cmn = sqrt(cm.x * cm.x + cm.y * cm.y);
  const double2 ph = cmn > 0.0 ? make_double2(cm.x / cmn, -cm.y / cmn) : make_double2(1.0, 0.0);  // conj phase
  double* S = p.S + (int64_t)i * p.ncv;
  double nr = 0.0;
  for (int64_t t = tid; t < na; t += 256) {
    const double2 c = cadd(z[t], z[na + t]);
    const double v = c.x * ph.x - c.y * ph.y;   // Re(c e^{-i phi})
    S[t] = v;
    nr += v * v;
  }
  nr = block_sum(nr, red);
  const double inv = nr > 0.0 ? 1.0 / sqrt(nr) : 0.0;
  for (int64_t t = tid; t < na; t += 256) S[t] *= inv;
  __syncthreads();
  if (tid == 0) {
    p.ritz[i] = lam[i] * lam[i];
    p.rest[i] = fabs(p.beta[st->m - 1] * S[na - 1]);
  }
}

__global__ void k_pj_fail(const Prob* __restrict__ probs, int ip) {
  KState* st = probs[ip].st;
  if (threadIdx.x == 0 && st->status == ST_OK) st->status = ST_NOTPD;
}

}  // namespace

// Dense diagonalisation of problem 0 of a PH handle: the nev lowest positive omega and
// their right eigenvectors (unnormalised) in Z (ld 2 Npad).  Returns 0, 1 (M_r not positive
// definite) or -1 (CUDA error).  `work` holds dense_scratch_doubles(N, nev) doubles.
int dense_shao(const Prob* dprobs, int64_t N, int64_t Npad, bool tiles64, bool pq, int nev, double* work,
               int* dflag, double2* Z, double* lam_out, cudaStream_t s) {
  const int64_t n = 2 * N;
  const dim3 g2((unsigned)((n + 31) / 32), (unsigned)((n + 7) / 8)), b2(32, 8);
  double* lam = nullptr;
  const int rc = dense_run(N, Npad, nev, work, dflag, Z, &lam, [&](double* M, int64_t ld) {
    count_launch();
    if (tiles64) k_dn_assemble<float2><<<g2, b2, 0, s>>>(dprobs, pq ? 1 : 0, M, ld);
    else k_dn_assemble<double2><<<g2, b2, 0, s>>>(dprobs, pq ? 1 : 0, M, ld);
  }, s);
  if (rc) return rc;
  if (lam_out && (cudaMemcpyAsync(lam_out, lam, sizeof(double) * nev, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
                  cudaStreamSynchronize(s) != cudaSuccess))
    return -1;
  return 0;
}

size_t projected_scratch_doubles(int n, int nw) { return (size_t)4 * n * nw + 64; }

int projected_ritz(const Prob* dprobs, int iprob, int n, int nw, double* work, int* dflag, cudaStream_t s) {
  if (n < 1 || nw < 1) return 0;
  const int64_t n2 = 2 * (int64_t)n;
  const dim3 g2((unsigned)((n2 + 31) / 32), (unsigned)((n2 + 7) / 8)), b2(32, 8);
  const size_t dsz = (dense_scratch_doubles(n, nw) + 31) / 32 * 32;
  double2* Zs = reinterpret_cast<double2*>(work + dsz);
  double* lam = nullptr;
  const int rc = dense_run(n, n, nw, work, dflag, Zs, &lam, [&](double* M, int64_t ld) {
    count_launch();
    k_pj_assemble<<<g2, b2, 0, s>>>(dprobs, iprob, M, ld);
  }, s);
  if (rc < 0 || rc == 2) return rc;
  count_launch();
  if (rc == 1) {
    k_pj_fail<<<1, 32, 0, s>>>(dprobs, iprob);
    return cudaGetLastError() == cudaSuccess ? 1 : -1;
  }
  k_pj_coef<<<nw, 256, 0, s>>>(dprobs, iprob, n, Zs, lam);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}


}  // namespace bse
