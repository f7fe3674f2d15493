// Eigenvalues by multisection and eigenvectors by inverse iteration of a symmetric matrix whose
// graph is a star of leaves around the first vertex (the hub) of a path: the projected problems of
// the restart (k_ritz.cu) and, without leaves, the tridiagonal matrix of the dense method
// (k_dense.cu).
//
// What bounds them is latency: a warp-wide FP64 instruction holds its scheduler's FP64 pipe for 64
// clocks whatever its active lanes, and a division is some nine of them (measured: 570 clocks), so
// a Sturm count with one division per row took 860 clocks a row.  Therefore
//   * the multisection narrows each eigenvalue to about 2^-40 of ||T|| with counts in double-FP32
//     arithmetic (FP32 pipes), and FP64 counts take over from there: they check that the bracket
//     holds the wanted index (else they start from the whole interval) and finish to FP64
//     accuracy, so the result does not rest on the FP32 counts;
//   * reciprocals are the hardware's 20-bit one and one step of the third-order iteration (three
//     FMAs, recip), signs and magnitudes are compared as integers;
//   * in the factorisation and the solves the leaves go over the lanes, and only the path part
//     (the new Lanczos vectors of the cycle) is sequential, with the pivots' reciprocals kept.
#pragma once

#include "bse_internal.cuh"

namespace bse {

struct TV {        // view of the matrix
  const double* d; // leaves' diagonal
  const double* b; // leaves' couplings to the hub
  int h;           // number of leaves
  const double* a; // hub and path diagonal
  const double* e; // path off-diagonal: e[t] couples a[t] and a[t+1]
  int n;           // order
};

__device__ __forceinline__ int mag_hi(double v) { return __double2hiint(v) & 0x7fffffff; }

// 1 / q within an ulp, for a normal q with a normal reciprocal: the hardware's approximation r (20 bits)
// and one step of the third-order iteration r (1 + e + e^2), e = 1 - q r (the first terms of the
// geometric series of 1 / (1 - e)): what is left of r's error is its cube, 2^-60.  The pivots below are
// in that range: of a finite T none is smaller than its pivmin (1e-306 at least) or larger than 1e300.
__device__ __forceinline__ double recip(double q) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(q));
  const double e = fma(-q, r, 1.0);
  return fma(r, fma(e, e, e), r);
}
// ... for any q: zero, a subnormal, one above 2^1022, an infinity or a NaN goes to the division (which
// costs the loops of the counts and factorisations 1 % where it is not needed)
__device__ __forceinline__ double recip_any(double q) {
  const unsigned ex = ((unsigned)__double2hiint(q) >> 20) & 0x7ffu;
  return ex - 1u < 2044u ? recip(q) : 1.0 / q;
}

// a pivot of the Sturm count: tiny ones become -pivmin (their high words compared); the sign adds
// to the count
__device__ __forceinline__ double sturm_pivot(double q, double pivmin, int& cnt) {
  if (mag_hi(q) < mag_hi(pivmin)) q = -pivmin;
  cnt += (unsigned)__double2hiint(q) >> 31;
  return q;
}

// number of eigenvalues < sigma (LDL^T pivots of T - sigma I, leaves first); T's entries with the
// couplings squared: leaves d, b2, hub and path a, e2
__device__ inline int sturm_count(const double* d, const double* b2, int h, const double* a, const double* e2, int nq,
                           double sigma, double pivmin) {
  int cnt = 0;
  double s = 0.0;
  for (int i = 0; i < h; ++i) s = fma(b2[i], recip(sturm_pivot(d[i] - sigma, pivmin, cnt)), s);
  double q = sturm_pivot(a[0] - sigma - s, pivmin, cnt);
  for (int t = 1; t < nq; ++t) q = sturm_pivot(fma(-e2[t - 1], recip(q), a[t] - sigma), pivmin, cnt);
  return cnt;
}

// ---- the same count in double-FP32 arithmetic: numbers (hi, lo), about 2^-45 relative each step
__device__ __forceinline__ float2 f2_sub(float2 x, float2 y) {       // TwoSum of the high parts
  const float s = __fsub_rn(x.x, y.x), t = __fsub_rn(s, x.x);
  const float e = __fadd_rn(__fsub_rn(x.x, __fsub_rn(s, t)), -__fadd_rn(y.x, t));
  const float l = __fadd_rn(e, __fsub_rn(x.y, y.y));
  const float h = __fadd_rn(s, l);
  return make_float2(h, __fsub_rn(l, __fsub_rn(h, s)));
}
__device__ __forceinline__ float2 f2_div(float2 x, float2 y) {       // q = x / y with one correction
  const float r = __frcp_rn(y.x);
  const float q = __fmul_rn(x.x, r);
  float e = __fmaf_rn(-q, y.x, x.x);
  e = __fadd_rn(e, __fmaf_rn(-q, y.y, x.y));
  const float l = __fmul_rn(e, r);
  const float h = __fadd_rn(q, l);
  return make_float2(h, __fsub_rn(l, __fsub_rn(h, q)));
}
__device__ __forceinline__ float2 f2_pivot(float2 q, float pivmin, int& cnt) {
  if (fabsf(q.x) < pivmin) q = make_float2(-pivmin, 0.f);
  cnt += q.x < 0.f;
  return q;
}
__device__ inline int sturm_count32(const float2* d, const float2* b2, int h, const float2* a, const float2* e2, int nq,
                             float2 sigma, float pivmin) {
  int cnt = 0;
  float2 s = make_float2(0.f, 0.f);                                  // minus the leaves' sum
#pragma unroll 2
  for (int i = 0; i < h; ++i) s = f2_sub(s, f2_div(b2[i], f2_pivot(f2_sub(d[i], sigma), pivmin, cnt)));
  s.x = -s.x;
  s.y = -s.y;
  float2 q = f2_pivot(f2_sub(f2_sub(a[0], sigma), s), pivmin, cnt);
  for (int t = 1; t < nq; ++t)
    q = f2_pivot(f2_sub(f2_sub(a[t], sigma), f2_div(e2[t - 1], q)), pivmin, cnt);
  return cnt;
}

__device__ __forceinline__ float2 f2_split(double v) {
  const float f = (float)v;
  return make_float2(f, (float)(v - (double)f));
}

// the power of two that brings the norm to at most 1
__device__ __forceinline__ double tree_scale(double tnorm) { return tnorm > 0.0 ? exp2(-ceil(log2(tnorm))) : 1.0; }

// The eigenvalue of index idx (ascending) by a CTA of RV_THREADS threads, one shift each: diagonal
// x[0, n) (leaves, then hub and path), squared couplings c, both also in double-FP32 times tree_scale
// (its square for the couplings); [lo, hi] holds the spectrum; s_sig and s_cnt are shared memory.
constexpr int RV_THREADS = 128;

__device__ __forceinline__ double tree_eigenvalue(const double* x, const double* c, const float2* xf, const float2* cf,
                                                  int h, int nq, int idx, double lo, double hi, double tnorm, double sc,
                                                  double* s_sig, int* s_cnt) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // one round of the multisection: the shifts' counts give the interval [s_{L-1}, s_L] that holds
  // the wanted index, L the number of shifts with count <= idx
  auto narrow = [&](double sig, int cnt) {
    s_sig[tid] = sig;
    const unsigned below = __ballot_sync(0xffffffffu, cnt <= idx);
    if (lane == 0) s_cnt[warp] = __popc(below);
    __syncthreads();
    const int L = s_cnt[0] + s_cnt[1] + s_cnt[2] + s_cnt[3];
    if (L > 0) lo = s_sig[L - 1];
    if (L < RV_THREADS) hi = s_sig[L];
    __syncthreads();
    return L;
  };
  const double lo0 = lo, hi0 = hi;
  const double margin = ldexp(tnorm, -41);
  bool known = true;                       // count(lo) <= idx < count(hi) holds by FP64 counts
  if (sc > 1e-250 && sc < 1e250) {
    for (int it = 0; it < 10 && hi - lo > 2.0 * margin; ++it) {
      const double sig = lo + (hi - lo) * (double)(tid + 1) * (1.0 / (RV_THREADS + 1));
      narrow(sig, sturm_count32(xf, cf, h, xf + h, cf + h, nq, f2_split(sig * sc), 1e-30f));
      known = false;
    }
    if (!known) {                          // 2^-41 ||T|| on both sides covers the FP32 counts' error
      lo = fmax(lo0, lo - margin);
      hi = fmin(hi0, hi + margin);
    }
  }
  const double pivmin = 1e-290 * fmax(1.0, tnorm * tnorm);
  const double eps = 2.220446049250313e-16;
  for (int it = 0; it < 100; ++it) {
    const double width = hi - lo;
    if (known && width <= 2.0 * eps * fmax(fabs(lo), fabs(hi)) + 4.0 * pivmin) break;
    // until the ends are known to hold the index they are shifts themselves
    const double sig = known ? lo + width * (double)(tid + 1) * (1.0 / (RV_THREADS + 1))
                             : (tid == RV_THREADS - 1 ? hi : lo + width * (double)tid * (1.0 / (RV_THREADS - 1)));
    const int L = narrow(sig, sturm_count(x, c, h, x + h, c + h, nq, sig, pivmin));
    if (!known && (L == 0 || L == RV_THREADS)) { lo = lo0; hi = hi0; }   // the bracket missed it
    known = true;
  }
  return 0.5 * (lo + hi);
}

// ---------------------------------------------------------------- inverse iteration
struct Fact {      // factorisation of T - lambda I (shared memory)
  double* invd;    // 1 / delta_i of the leaves, then 1 / pivot of the path (U's diagonal)
  double* dl;      // path GEPP: multipliers
  double* du;      // path GEPP: U first super-diagonal
  double* du2;     // path GEPP: U second super-diagonal
  unsigned char* piv;
};

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int m = 16; m >= 1; m >>= 1) v += __shfl_xor_sync(0xffffffffu, v, m);
  return v;
}

// |a| >= |b| as integers (no NaN)
__device__ __forceinline__ bool abs_ge(double a, double b) {
  return (__double_as_longlong(a) & 0x7fffffffffffffffll) >= (__double_as_longlong(b) & 0x7fffffffffffffffll);
}

// Factor T - lambda I (a warp): leaves eliminated into the hub, lane by lane, then Gaussian
// elimination with partial pivoting on the tridiagonal hub + path block, which every lane runs with
// the current row in registers (one of them stores).  Pivots below pivmin become pivmin, so their
// reciprocals exist.
__device__ inline void factor_tree(const TV& T, double lam, double pivmin, Fact& F, int lane) {
  const int h = T.h, q = T.n - h;
  double s = 0.0;
  for (int i = lane; i < h; i += 32) {
    double di = T.d[i] - lam;
    if (!abs_ge(di, pivmin)) di = di < 0.0 ? -pivmin : pivmin;
    const double r = recip(di), b = T.b[i];
    F.invd[i] = r;
    s = fma(b * b, r, s);
  }
  s = warp_sum(s);
  double* rp = F.invd + h;
  double d = T.a[0] - lam - s, du = q > 1 ? T.e[0] : 0.0;      // row t: d, du (and 0)
  for (int t = 0; t + 1 < q; ++t) {
    const double e = T.e[t], dn = T.a[t + 1] - lam, un = t + 2 < q ? T.e[t + 1] : 0.0;
    double pu, pu2, f, r, d2, u2;
    const bool keep = abs_ge(d, e);
    if (keep) {                          // row t is the pivot row
      if (!abs_ge(d, pivmin)) d = d < 0.0 ? -pivmin : pivmin;
      r = recip(d);
      f = e * r;
      pu = du; pu2 = 0.0;
      d2 = fma(-f, du, dn);
      u2 = un;
    } else {                             // row t + 1: (e, dn, un)
      r = recip(abs_ge(e, pivmin) ? e : pivmin);
      f = d * r;
      pu = dn; pu2 = un;
      d2 = fma(-f, dn, du);
      u2 = -f * un;
    }
    if (lane == 0) {
      F.piv[t] = keep ? 0 : 1;
      F.du[t] = pu; F.du2[t] = pu2; F.dl[t] = f;
      rp[t] = r;
    }
    d = d2;
    du = u2;
  }
  if (!abs_ge(d, pivmin)) d = d < 0.0 ? -pivmin : pivmin;
  const double r = recip(d);
  if (lane == 0) rp[q - 1] = r;
  __syncwarp();
}

// Solve (T - lambda I) x = r in place (a warp; x holds r on entry), x has n entries in shared memory.
__device__ inline void solve_tree(const TV& T, const Fact& F, double* x, int lane) {
  const int h = T.h, q = T.n - h;
  const double* rp = F.invd + h;
  double* y = x + h;   // hub + path part
  double s = 0.0;
  for (int i = lane; i < h; i += 32) s = fma(T.b[i] * x[i], F.invd[i], s);
  s = warp_sum(s);
  // every lane runs the recurrence, one of them stores: each entry is read by all before it is rewritten
  double cur = y[0] - s;
  for (int t = 0; t + 1 < q; ++t) {
    const double nx = y[t + 1];
    __syncwarp();
    if (F.piv[t] == 0) {
      if (lane == 0) y[t] = cur;
      cur = fma(-F.dl[t], cur, nx);
    } else {
      if (lane == 0) y[t] = nx;
      cur = fma(-F.dl[t], nx, cur);
    }
  }
  __syncwarp();
  double x1 = cur * rp[q - 1], x2 = 0.0;
  if (lane == 0) y[q - 1] = x1;
  for (int t = q - 2; t >= 0; --t) {
    const double v = fma(-F.du2[t], x2, fma(-F.du[t], x1, y[t])) * rp[t];
    __syncwarp();
    if (lane == 0) y[t] = v;
    x2 = x1;
    x1 = v;
  }
  __syncwarp();
  for (int i = lane; i < h; i += 32) x[i] = fma(-T.b[i], x1, x[i]) * F.invd[i];
  __syncwarp();
}

__host__ __device__ __forceinline__ uint64_t mix64(uint64_t x) {
  x += 0x9e3779b97f4a7c15ull;
  x = (x ^ (x >> 30)) * 0xbf58476d1ce4e5b9ull;
  x = (x ^ (x >> 27)) * 0x94d049bb133111ebull;
  return x ^ (x >> 31);
}

}  // namespace bse
