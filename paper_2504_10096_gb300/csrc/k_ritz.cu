// Projected eigenproblem and restart decision of the thick-restart Lanczos
// iteration (Sec. 2.2.1: the problem is projected onto a small structured
// problem; a thick restart keeps Ritz vectors without destroying structure).
//
// After a restart the projected matrix of the active (unlocked) block is
//     [ diag(theta_kept)   b          0   ]
//     [ b^T                alpha_l   beta ]
//     [ 0                  beta      tridiagonal ...]
// i.e. an arrowhead glued to a tridiagonal: its graph is a star (the kept
// Ritz vectors) attached to a path (the new Lanczos vectors).  Gaussian
// elimination from the leaves of that tree has no fill-in, so
//   * the inertia of T - sigma I (a Sturm count) costs O(n): used for
//     multisection of every wanted eigenvalue, four warps per eigenvalue;
//   * (T - lambda I) x = r costs O(n): used for inverse iteration, one warp
//     per cluster of close eigenvalues, Gram-Schmidt inside a cluster.
//
// What bounds them is latency: a warp-wide FP64 instruction holds its scheduler's FP64 pipe for 64
// clocks whatever its active lanes, and a division is some nine of them (measured: 570 clocks), so
// a Sturm count with one division per row took 860 clocks a row.  Therefore
//   * the multisection narrows each eigenvalue to about 2^-40 of ||T|| with counts in double-FP32
//     arithmetic (FP32 pipes), and FP64 counts take over from there: they check that the bracket
//     holds the wanted index (else they start from the whole interval) and finish to FP64
//     accuracy, so the result does not rest on the FP32 counts;
//   * reciprocals are the hardware's 20-bit one and one cubic Newton step, r (1 + e + e^2) with
//     e = 1 - q r (three FMAs), signs and magnitudes are compared as integers;
//   * in the factorisation and the solves the leaves go over the lanes, and only the path part
//     (the new Lanczos vectors of the cycle) is sequential, with the pivots' reciprocals kept.
// Measured per restart, 46 wanted of order 62 (PH N = 3000): values 342 -> 70 us, vectors 79
// -> 29 us (and the lock decision by a warp instead of a thread 19 -> 4 us).
//
// Gruning variant: the projected matrix is H's own, the symmetric matrix with
// zero diagonal that couples u_j -- w_j (alpha_j) and w_j -- u_{j+1} (beta_j);
// after a restart each kept Ritz pair (u~_i, w~_i) is coupled by sigma_i and
// w~_i to the hub u_l by rho_i.  Rotating each kept pair to (u~ +- w~)/sqrt 2
// gives leaves +sigma_i and -sigma_i with couplings +-rho_i / sqrt 2 to the hub,
// followed by the path u_l, w_l, u_{l+1}, ..., w_{m-1}: the same star-plus-path
// tree, of order 2 (m - k), whose spectrum is +-sigma.  The wanted values are
// the indices m - k, m - k + 1, ... of its ascending spectrum (bisection as
// above), and each eigenvector splits into even-side (V) and odd-side (W)
// coefficients of norm 1 / sqrt 2 each.
#include "bse_internal.cuh"

namespace bse {

struct TV {        // view of the active projected matrix of one problem
  const double* d; // leaves' diagonal (theta[k..l))
  const double* b; // leaves' couplings to the hub (barrow[k..l))
  int h;           // number of leaves
  const double* a; // hub and tail diagonal (alpha[l..m))
  const double* e; // tail off-diagonal: e[t] couples a[t] and a[t+1]
  int n;           // order = h + (m - l)
};

__device__ __forceinline__ bool is_gk(const Prob& p) { return p.ph && p.variant == VAR_GRUNING; }

__device__ __forceinline__ TV make_tv(const Prob& p, const KState* st) {
  TV t;
  if (is_gk(p)) {
    const int ld = p.jwld;
    t.d = p.jw;
    t.b = p.jw + ld;
    t.h = 2 * (st->l - st->k);
    t.a = p.jw + 2 * ld;
    t.e = p.jw + 3 * ld;
    t.n = 2 * (st->m - st->k);
    return t;
  }
  t.d = p.theta + st->k;
  t.b = p.barrow + st->k;
  t.h = st->l - st->k;
  t.a = p.alpha + st->l;
  t.e = p.beta + st->l;
  t.n = st->m - st->k;
  return t;
}

// column i of the projected problem's Ritz vectors (the tree's, on the Gruning path)
__device__ __forceinline__ double* ritz_vec(const Prob& p, int i) {
  return is_gk(p) ? p.jw + 4 * (int64_t)p.jwld + (int64_t)i * p.jwld : p.S + (int64_t)i * p.ncv;
}

// Gruning path: the tree arrays of the active block (one thread per problem)
__global__ void k_gk_form(const Prob* __restrict__ probs, int nprob) {
  const int ip = blockIdx.x * blockDim.x + threadIdx.x;
  if (ip >= nprob) return;
  const Prob& p = probs[ip];
  const KState* st = p.st;
  if (!restart_ready(st)) return;
  const int k = st->k, l = st->l, m = st->m, h = l - k, ld = p.jwld;
  double* d = p.jw;
  double* b = p.jw + ld;
  double* a = p.jw + 2 * ld;
  double* e = p.jw + 3 * ld;
  const double r2 = 0.70710678118654752440;
  for (int i = 0; i < h; ++i) {
    d[i] = p.theta[k + i];
    d[h + i] = -p.theta[k + i];
    b[i] = p.barrow[k + i] * r2;
    b[h + i] = -p.barrow[k + i] * r2;
  }
  for (int t = 0; t < 2 * (m - l); ++t) a[t] = 0.0;
  for (int t = 0; t < m - l; ++t) {
    e[2 * t] = p.alpha[l + t];
    if (t + 1 < m - l) e[2 * t + 1] = p.beta[l + t];
  }
}

__device__ __forceinline__ int nwanted(const KState* st) {
  const int n = st->m - st->k;
  const int w = st->r_pkeep - st->k;
  return w < n ? w : n;
}

__device__ __forceinline__ int hi_abs(double v) { return __double2hiint(v) & 0x7fffffff; }

// 1 / q to FP64 rounding for a normal q: the hardware's approximation and one cubic Newton step
__device__ __forceinline__ double recip(double q) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(q));
  const double e = fma(-q, r, 1.0);
  return fma(r, fma(e, e, e), r);
}

// a pivot of the Sturm count: tiny ones become -pivmin (their high words compared); the sign adds
// to the count
__device__ __forceinline__ double sturm_pivot(double q, double pivmin, int& cnt) {
  if (hi_abs(q) < hi_abs(pivmin)) q = -pivmin;
  cnt += (unsigned)__double2hiint(q) >> 31;
  return q;
}

// number of eigenvalues < sigma (LDL^T pivots of T - sigma I, leaves first); T's entries with the
// couplings squared: leaves d, b2, hub and path a, e2
__device__ int sturm_count(const double* d, const double* b2, int h, const double* a, const double* e2, int nq,
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
__device__ int sturm_count32(const float2* d, const float2* b2, int h, const float2* a, const float2* e2, int nq,
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

__device__ void gersh(const TV& T, double& lo, double& hi, double& tnorm, int lane) {
  double glo = 1e300, ghi = -1e300, sb = 0.0, mx = 0.0;
  for (int i = lane; i < T.h; i += 32) {
    glo = fmin(glo, T.d[i] - fabs(T.b[i]));
    ghi = fmax(ghi, T.d[i] + fabs(T.b[i]));
    sb += fabs(T.b[i]);
  }
  const int q_n = T.n - T.h;
  for (int t = lane; t < q_n; t += 32) {
    double r = (t > 0 ? fabs(T.e[t - 1]) : 0.0) + (t + 1 < q_n ? fabs(T.e[t]) : 0.0);
    if (t == 0) r += 0.0;  // the leaves' couplings are added below
    glo = fmin(glo, T.a[t] - r);
    ghi = fmax(ghi, T.a[t] + r);
  }
#pragma unroll
  for (int m = 16; m >= 1; m >>= 1) {
    glo = fmin(glo, __shfl_xor_sync(0xffffffffu, glo, m));
    ghi = fmax(ghi, __shfl_xor_sync(0xffffffffu, ghi, m));
    sb += __shfl_xor_sync(0xffffffffu, sb, m);
  }
  // hub row also carries sum |b_i|
  const double r0 = sb + (q_n > 1 ? fabs(T.e[0]) : 0.0);
  glo = fmin(glo, T.a[0] - r0);
  ghi = fmax(ghi, T.a[0] + r0);
  mx = fmax(fabs(glo), fabs(ghi));
  const double pad = 2.2e-16 * 8.0 * mx + 1e-300;
  lo = glo - pad;
  hi = ghi + pad;
  tnorm = mx;
}

// four warps (128 shifts) per wanted eigenvalue; grid (ncv, nprob); dynamic shared memory: the
// tree's entries in FP64 and in double-FP32 (scaled by a power of two to norm 1)
constexpr int RV_THREADS = 128;

__global__ void __launch_bounds__(RV_THREADS) k_ritz_values(const Prob* __restrict__ probs) {
  extern __shared__ double sm[];
  __shared__ double s_g[3];
  __shared__ double s_sig[RV_THREADS];
  __shared__ int s_cnt[RV_THREADS / 32];
  const Prob& p = probs[blockIdx.y];
  const KState* st = p.st;
  if (!restart_ready(st)) return;
  const int i = blockIdx.x;
  if (i >= nwanted(st)) return;
  const TV T = make_tv(p, st);
  const int idx = is_gk(p) ? (st->m - st->k) + i : i;   // position in the ascending spectrum
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n = T.n, h = T.h, nq = n - h;
  if (warp == 0) {
    double lo, hi, tnorm;
    gersh(T, lo, hi, tnorm, lane);
    if (lane == 0) { s_g[0] = lo; s_g[1] = hi; s_g[2] = tnorm; }
  }
  __syncthreads();
  double lo = s_g[0], hi = s_g[1];
  const double tnorm = s_g[2];
  // entries: diagonal x[0, n) (leaves, then hub and path), squared couplings c[0, n - 1)
  double* x = sm;
  double* c = sm + n;
  float2* xf = reinterpret_cast<float2*>(c + n);
  float2* cf = xf + n;
  const double sc = tnorm > 0.0 ? exp2(-ceil(log2(tnorm))) : 1.0;
  auto split = [](double v) {
    const float f = (float)v;
    return make_float2(f, (float)(v - (double)f));
  };
  for (int t = tid; t < n; t += RV_THREADS) {
    const double xv = t < h ? T.d[t] : T.a[t - h];
    const double cv = t < h ? T.b[t] : (t + 1 < n ? T.e[t - h] : 0.0);
    x[t] = xv;
    c[t] = cv * cv;
    xf[t] = split(xv * sc);
    cf[t] = split((cv * sc) * (cv * sc));
  }
  __syncthreads();
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
      narrow(sig, sturm_count32(xf, cf, h, xf + h, cf + h, nq, split(sig * sc), 1e-30f));
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
  if (tid == 0) p.ritz[i] = 0.5 * (lo + hi);
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
__device__ void factor_tree(const TV& T, double lam, double pivmin, Fact& F, int lane) {
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
__device__ void solve_tree(const TV& T, const Fact& F, double* x, int lane) {
  const int h = T.h, q = T.n - h;
  const double* rp = F.invd + h;
  double* y = x + h;   // hub + path part
  double s = 0.0;
  for (int i = lane; i < h; i += 32) s = fma(T.b[i] * x[i], F.invd[i], s);
  s = warp_sum(s);
  double cur = y[0] - s;
  for (int t = 0; t + 1 < q; ++t) {
    const double nx = y[t + 1];
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

// one warp per cluster leader; grid (ncv, nprob), block 32, dynamic smem.
__global__ void __launch_bounds__(32) k_ritz_vectors(const Prob* __restrict__ probs) {
  extern __shared__ double sm[];
  const Prob& p = probs[blockIdx.y];
  const KState* st = p.st;
  if (!restart_ready(st)) return;
  const int nw = nwanted(st);
  const int i0 = blockIdx.x;
  if (i0 >= nw) return;
  const TV T = make_tv(p, st);
  const int n = T.n, lane = threadIdx.x;
  double lo, hi, tnorm;
  gersh(T, lo, hi, tnorm, lane);
  const double eps = 2.220446049250313e-16;
  const double ctol = 1e-7 * tnorm;             // cluster threshold
  const double* rz = p.ritz;
  if (i0 > 0 && rz[i0] - rz[i0 - 1] < ctol) return;   // not a cluster leader
  int i1 = i0 + 1;
  while (i1 < nw && rz[i1] - rz[i1 - 1] < ctol) ++i1;
  const int M = is_gk(p) ? p.jwld : p.ncv;    // scratch stride
  Fact F;
  F.invd = sm;
  F.dl = sm + M;
  F.du = sm + 2 * M;
  F.du2 = sm + 3 * M;
  double* x = sm + 4 * M;
  F.piv = (unsigned char*)(sm + 5 * M);
  // pivot guard of the inverse iteration: a shift equal to a leaf value (a
  // converged kept Ritz value with a negligible coupling) must give a large
  // but finite growth, so tiny pivots are replaced by eps * ||T||
  const double pivmin = eps * fmax(tnorm, 1e-300);
  const double pert = 10.0 * eps * tnorm;
  double lam_prev = -1e300;
  for (int i = i0; i < i1; ++i) {
    double lam = rz[i];
    if (i > i0 && lam - lam_prev < pert) lam = lam_prev + pert;
    lam_prev = lam;
    factor_tree(T, lam, pivmin, F, lane);
    // deterministic start vector
    for (int t = lane; t < n; t += 32) {
      const uint64_t hsh = mix64((uint64_t)(i + 1) * 0x100000001b3ull + (uint64_t)t);
      x[t] = (double)(hsh >> 11) * (1.0 / 9007199254740992.0) - 0.5;
    }
    __syncwarp();
    for (int it = 0; it < 4; ++it) {
      // orthogonalise against the cluster's earlier vectors (twice), normalise
      for (int rep = 0; rep < 2; ++rep) {
        for (int c = i0; c < i; ++c) {
          const double* sc = ritz_vec(p, c);
          double dot = 0.0;
          for (int t = lane; t < n; t += 32) dot += sc[t] * x[t];
          dot = warp_sum(dot);
          for (int t = lane; t < n; t += 32) x[t] -= dot * sc[t];
          __syncwarp();
        }
      }
      double nr = 0.0;
      for (int t = lane; t < n; t += 32) nr += x[t] * x[t];
      nr = warp_sum(nr);
      const double inv = nr > 0.0 ? rsqrt(nr) : 0.0;
      for (int t = lane; t < n; t += 32) x[t] *= inv;
      __syncwarp();
      if (it == 3) break;
      solve_tree(T, F, x, lane);
    }
    double* out = ritz_vec(p, i);
    for (int t = lane; t < n; t += 32) out[t] = x[t];
    if (is_gk(p)) {
      // even-side (u~_k.., hub, u_{l+1}..) and odd-side (w~_k.., w_l..) coefficients, each
      // of norm 1 after the factor sqrt 2
      const int h = st->l - st->k, nt = st->m - st->l;
      const double s2 = 1.41421356237309504880;
      double* Se = p.S + (int64_t)i * p.ncv;
      double* So = p.S2 + (int64_t)i * p.ncv;
      for (int c = lane; c < h; c += 32) {
        Se[c] = x[c] + x[h + c];
        So[c] = x[c] - x[h + c];
      }
      for (int t = lane; t < nt; t += 32) {
        So[h + t] = s2 * x[2 * h + 1 + 2 * t];
        Se[h + t] = s2 * x[2 * h + 2 * t];
      }
      if (lane == 0) p.rest[i] = fabs(p.beta[st->m - 1] * s2 * x[n - 1]);
    } else if (lane == 0) {
      p.rest[i] = fabs(p.beta[st->m - 1] * x[n - 1]);
    }
    __syncwarp();
  }
}

// Lock the leading converged Ritz pairs, choose what to keep, and write the
// restarted arrow (theta, b).  One warp per problem.
__global__ void __launch_bounds__(32) k_lock_decide(const Prob* __restrict__ probs, int ph) {
  const Prob& p = probs[blockIdx.x];
  KState* st = p.st;
  if (!restart_ready(st)) return;
  const int lane = threadIdx.x;
  const int k = st->k, m = st->m, n = m - k, nev = st->nev;
  const int nw = nwanted(st);
  const double lock_tol = st->lock_tol;
  const bool notpd = ph && p.ritz[0] <= 0.0;
  // leading pairs within the tolerance, 32 at a time
  int nl = 0;
  for (;;) {
    const int i = nl + lane;
    const bool ok = i < nw && k + i < nev && p.rest[i] <= lock_tol * fabs(p.ritz[i]);
    const int run = __ffs(~__ballot_sync(0xffffffffu, ok)) - 1;      // -1: all 32
    nl += run < 0 ? 32 : run;
    if (run >= 0) break;
  }
  int nkeep;
  if (k + nl >= nev) {
    nkeep = nl;
  } else {
    nkeep = st->r_pkeep - k;
    if (nkeep < nl + 1) nkeep = nl + 1;
    if (nkeep > nw) nkeep = nw;
  }
  const double bl = p.beta[m - 1];
  __syncwarp();                                    // the state has been read by every lane
  if (notpd) {
    if (lane == 0) st->status = ST_NOTPD;
    return;
  }
  const double* Sl = is_gk(p) ? p.S2 : p.S;        // the last basis vector's side
  for (int i = lane; i < nkeep; i += 32) {
    p.theta[k + i] = p.ritz[i];
    p.barrow[k + i] = i < nl ? 0.0 : bl * Sl[(int64_t)i * p.ncv + (n - 1)];
  }
  if (lane == 0) {
    st->beta_last = bl;
    st->r_k0 = k;
    st->r_nl = nl;
    st->r_nkeep = nkeep;
    st->r_go = 1;
  }
}

void launch_ritz(const Prob* dprobs, int nprob, int ncv, bool gruning, cudaStream_t s) {
  if (gruning) {
    count_launch();
    k_gk_form<<<(nprob + 127) / 128, 128, 0, s>>>(dprobs, nprob);
  }
  count_launch(2);
  const size_t M = gruning ? (size_t)(2 * ncv + 2) : (size_t)ncv;
  const size_t sv = M * 2 * (sizeof(double) + sizeof(float2)), sm = M * 5 * sizeof(double) + M + 16;
  if (sv > 48 * 1024) cudaFuncSetAttribute(k_ritz_values, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sv);
  if (sm > 48 * 1024) cudaFuncSetAttribute(k_ritz_vectors, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  k_ritz_values<<<dim3(ncv, nprob), RV_THREADS, sv, s>>>(dprobs);
  k_ritz_vectors<<<dim3(ncv, nprob), 32, sm, s>>>(dprobs);
}

void launch_lock_decide_form(const Prob* dprobs, int nprob, int ph, cudaStream_t s) {
  count_launch();
  k_lock_decide<<<nprob, 32, 0, s>>>(dprobs, ph);
}

}  // namespace bse
