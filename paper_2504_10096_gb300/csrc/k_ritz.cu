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
// (tree_solve.cuh has both and what bounds them).  Measured per restart, 46 wanted of order 62 (PH
// N = 3000): values 342 -> 70 us, vectors 79 -> 29 us, the lock decision by a warp instead of a thread
// 19 -> 4 us.
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
#include "tree_solve.cuh"

namespace bse {

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
  dep_begin();
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
__global__ void __launch_bounds__(RV_THREADS) k_ritz_values(const Prob* __restrict__ probs) {
  dep_begin();
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
  const double lo = s_g[0], hi = s_g[1], tnorm = s_g[2];
  // entries: diagonal x[0, n) (leaves, then hub and path), squared couplings c[0, n - 1)
  double* x = sm;
  double* c = sm + n;
  float2* xf = reinterpret_cast<float2*>(c + n);
  float2* cf = xf + n;
  const double sc = tree_scale(tnorm);
  for (int t = tid; t < n; t += RV_THREADS) {
    const double xv = t < h ? T.d[t] : T.a[t - h];
    const double cv = t < h ? T.b[t] : (t + 1 < n ? T.e[t - h] : 0.0);
    x[t] = xv;
    c[t] = cv * cv;
    xf[t] = f2_split(xv * sc);
    cf[t] = f2_split((cv * sc) * (cv * sc));
  }
  __syncthreads();
  const double v = tree_eigenvalue(x, c, xf, cf, h, nq, idx, lo, hi, tnorm, sc, s_sig, s_cnt);
  if (tid == 0) p.ritz[i] = v;
}

// ---------------------------------------------------------------- inverse iteration
// one warp per cluster leader; grid (ncv, nprob), block 32, dynamic smem.
__global__ void __launch_bounds__(32) k_ritz_vectors(const Prob* __restrict__ probs) {
  dep_begin();
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
  const double pivmin = eps * fmax(tnorm, 1e-290);    // normal, and its reciprocal too
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
  dep_begin();
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
    launch_dep(k_gk_form, (nprob + 127) / 128, 128, 0, s, dprobs, nprob);
  }
  count_launch(2);
  const size_t M = gruning ? (size_t)(2 * ncv + 2) : (size_t)ncv;
  auto values_bytes = [](size_t m) { return m * 2 * (sizeof(double) + sizeof(float2)); };
  auto vectors_bytes = [](size_t m) { return m * 5 * sizeof(double) + m + 16; };
  const size_t sv = values_bytes(M), sm = vectors_bytes(M);
  // opt in to what the largest subspace takes: the 48 KiB without it include the static arrays, and
  // another thread's launch may need more than this one
  static PerDevice<bool> opt_in;
  opt_in.get(current_device(), [&] {
    const size_t top = 2 * MAXM + 2;
    cudaFuncSetAttribute(k_ritz_values, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)values_bytes(top));
    cudaFuncSetAttribute(k_ritz_vectors, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)vectors_bytes(top));
    return true;
  });
  launch_dep(k_ritz_values, dim3(ncv, nprob), RV_THREADS, sv, s, dprobs);
  launch_dep(k_ritz_vectors, dim3(ncv, nprob), 32, sm, s, dprobs);
}

void launch_lock_decide_form(const Prob* dprobs, int nprob, int ph, cudaStream_t s) {
  count_launch();
  launch_dep(k_lock_decide, nprob, 32, 0, s, dprobs, ph);
}

}  // namespace bse
