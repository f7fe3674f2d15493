// Phase bodies of the Krylov step, shared by the one-kernel-per-phase launches (k_product.cu,
// k_krylov.cu: the kernels there are thin wrappers that map blockIdx onto a body's unit
// arguments and declare its shared memory) and the persistent step kernel (k_persist.cu: one
// cooperative launch runs whole Krylov steps, every phase a loop of its CTAs over the units,
// the phases separated by a grid barrier).  A body computes the same bits in either setting:
// it takes its work unit and shared memory as arguments and keeps the summation order of the
// unit fixed.  Loads of data that a persistent launch rewrites between its phases (the Krylov
// basis, the work vectors, the partial sums) go through ldv<COH>: L2 loads (ordered by
// the barrier's fences, and never served from a stale L1 line) when COH.
#pragma once

#include <type_traits>

#include "bse_internal.cuh"

namespace bse {

template <bool COH, typename T>
__device__ __forceinline__ T ldv(const T* p) {
  if constexpr (COH) return __ldcg(p);
  else return *p;
}
template <typename R> struct Acc;
template <> struct Acc<float> { using T = float2; };
template <> struct Acc<double> { using T = double2; };

template <typename T>
__device__ __forceinline__ T shfl_xor_c(T v, int m) {
  v.x = __shfl_xor_sync(0xffffffffu, v.x, m);
  v.y = __shfl_xor_sync(0xffffffffu, v.y, m);
  return v;
}

template <typename ST> struct RealOf;
template <> struct RealOf<float2> { using T = float; };
template <> struct RealOf<double2> { using T = double; };

__device__ __forceinline__ bool kactive(const KState* st) {
  return !st->done && st->status == ST_OK && !st->breakdown && st->j < st->m;
}
// problems that need a fresh basis vector: the very first one (j < 0) or a
// replacement after an invariant subspace was found (breakdown)
__device__ __forceinline__ bool kfresh(const KState* st) {
  return !st->done && st->status == ST_OK && (st->j < 0 || st->breakdown);
}
__device__ __forceinline__ bool kphase(const KState* st, int fresh) {
  return fresh ? kfresh(st) : kactive(st);
}

__device__ __forceinline__ double2 dshfl(double2 v, int m) {
  v.x = __shfl_xor_sync(0xffffffffu, v.x, m);
  v.y = __shfl_xor_sync(0xffffffffu, v.y, m);
  return v;
}

// ---------------------------------------------------------------- CGS2 sets
// The vectors of one Gram-Schmidt pass: x -= Um Re(Dm^H x) + i Ut Im(Dt^H x) on the PH
// paths (real coefficients), x -= Um (Um^H x) on the TDA path (complex ones).  The
// set entries are c < nm (main) and nm <= c < nm + nt (twins).  The input x of the first
// pass of a Gruning half is a basis column (p_j, z_j); the result always goes to w.
struct CgsSet {
  const void* dm; const void* dt;   // dot sources
  const void* um; const void* ut;   // update bases (the twins enter as i * Ut)
  int nm, nt;
};

__device__ __forceinline__ CgsSet cgs_set(const Prob& p, const KState* st, int ph, int half) {
  const int j = st->j;
  CgsSet c;
  if (!ph) {
    c.dm = c.um = p.V; c.dt = c.ut = nullptr; c.nm = j + 1; c.nt = 0;
  } else if (half == 0) {
    c.dm = p.P; c.dt = p.V; c.um = p.V; c.ut = p.P; c.nm = c.nt = j + 1;
  } else if (half == 1) {
    c.dm = p.Z; c.dt = p.P; c.um = p.W; c.ut = p.V; c.nm = j; c.nt = j + 1;
  } else {
    c.dm = p.P; c.dt = p.Z; c.um = p.V; c.ut = p.W; c.nm = c.nt = j + 1;
  }
  return c;
}

// the input of the first pass of a Gruning half (a basis column), else w
template <typename ST>
__device__ __forceinline__ const ST* cgs_src(const Prob& p, const KState* st, int half, int pass, int newvec) {
  if (pass == 0 && !newvec) {
    if (half == 1) return (const ST*)p.P + (int64_t)st->j * p.Npad;
    if (half == 2) return (const ST*)p.Z + (int64_t)st->j * p.Npad;
  }
  return (const ST*)p.w;
}

// Resolve the input / output vectors of a product for problem p.
// Returns false if the problem takes no part in this launch.
template <typename ST, typename R>
__device__ __forceinline__ bool prod_operands(const Prob& p, int mode, const GenericIO& io,
                                              const ST*& x, ST*& y, R& sB) {
  const KState* st = p.st;
  if (mode == PM_GENERIC) {
    x = (const ST*)io.xa; y = (ST*)io.y; sB = (R)io.sB; return true;
  }
  if (st->done || st->status != ST_OK) return false;
  const int j = st->j;
  const bool fresh = j < 0 || st->breakdown;
  switch (mode) {
    case PM_STEP_MMINUS:
      if (fresh || j >= p.ncv) return false;
      x = (const ST*)p.P + (int64_t)j * p.Npad; y = (ST*)p.w; sB = (R)-1; return true;
    case PM_STEP_MPLUS:
      if (fresh || j >= p.ncv) return false;
      x = (const ST*)p.w; y = (ST*)p.pw; sB = (R)1; return true;
    case PM_STEP_A:
      if (fresh || j >= p.ncv) return false;
      x = (const ST*)p.V + (int64_t)j * p.Npad; y = (ST*)p.w; sB = (R)0; return true;
    case PM_START_MPLUS:
      if (!fresh) return false;
      x = (const ST*)p.w; y = (ST*)p.pw; sB = (R)1; return true;
    case PM_STEP_MMINUS_W:
      if (fresh || j >= p.ncv) return false;
      x = (const ST*)p.w; y = (ST*)p.pw; sB = (R)-1; return true;
  }
  return false;
}

// A CTA walks the global job list either as one contiguous run or with stride
// gridDim.x (ProdShape).  Registers allow one FP64 CTA per SM (FP64-pipe
// bound) and two FP32 ones, so that twice as many tile loads are in flight
// (the FP32 product is HBM-latency bound).
// The tile walk of CTA bid of nblk; shared memory: xc, xr (column block J and row block I of
// x, TS entries each) and red (8 x TS, the column reduction across warps).
template <typename ST, typename R, bool HASB, bool COH = false>
__device__ __forceinline__ void prod_tiles_body(const Prob* __restrict__ probs, const TileJob* __restrict__ jobs,
                                                int njobs, int mode, const GenericIO& io, int strided, int bid,
                                                int nblk, typename Acc<R>::T* xc, typename Acc<R>::T* xr,
                                                typename Acc<R>::T (*red)[TS]) {
  using CT = typename Acc<R>::T;
  // complex128 PH tiles hold P = A + B and Q = A - B; complex64 PH tiles hold A and B
  constexpr bool PQ = HASB && std::is_same<ST, double2>::value;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int lane = tid & 31, warp = tid >> 5;
  const int per = strided ? 1 : (njobs + nblk - 1) / nblk;
  const int t0 = strided ? bid : bid * per;
  const int t1 = strided ? njobs : min(njobs, t0 + per);
  const int dt = strided ? nblk : 1;
  for (int t = t0; t < t1; t += dt) {
    const TileJob jb = jobs[t];
    const Prob& p = probs[jb.prob];
    const ST* x; ST* yout; R sB;
    if (!prod_operands<ST, R>(p, mode, io, x, yout, sB)) continue;   // uniform per CTA
    const bool diag = (jb.I == jb.J);
    __syncthreads();                       // smem of the previous tile is free
    if (tid < TS) xc[tid] = ccvt<CT>(ldv<COH>(x + (int64_t)jb.J * TS + tid));
    else xr[tid - TS] = ccvt<CT>(ldv<COH>(x + (int64_t)jb.I * TS + tid - TS));
    __syncthreads();
    // PH: M_s u = A u + s B conj(u) is real-linear; in (Re, Im) form its block
    // row is [[U_re, -V_im], [U_im, V_re]] with U = A + s B, V = A - s B (the
    // real matrix M_r of Eq. 5 for s = +1), and the transpose use of the same
    // tile is [[U_re, U_im], [-V_im, V_re]].  That is 8 real FMAs per stored
    // element pair instead of the 16 of A u + s B conj(u) as two complex
    // products.  Complex128 tiles store P = A + B and Q = A - B, so U, V are
    // P, Q (s = +1) or Q, P (s = -1); complex64 tiles keep A and B exact and
    // form U, V in registers.
    const bool pos = sB > (R)0;
    const ST* At = (const ST*)(PQ && !pos ? p.B : p.A) + (int64_t)jb.t * (TS * TS);
    const ST* Bt = HASB ? (const ST*)(PQ && !pos ? p.A : p.B) + (int64_t)jb.t * (TS * TS) : nullptr;
    CT racc[8], cacc[8];
#pragma unroll
    for (int b = 0; b < 8; ++b) cacc[b] = czero<CT>();
#pragma unroll
    for (int a = 0; a < 8; ++a) {
      const int r = ty + 16 * a;
      ST av[8], bv[8];
#pragma unroll
      for (int b = 0; b < 8; ++b) {
        av[b] = __ldg(At + r * TS + tx + 16 * b);
        if (HASB) bv[b] = __ldg(Bt + r * TS + tx + 16 * b);
      }
      CT ra = czero<CT>();
      const CT y = xr[r];
#pragma unroll
      for (int b = 0; b < 8; ++b) {
        const int c = tx + 16 * b;
        const CT xv = xc[c];
        if (HASB) {
          CT u, v;
          if constexpr (PQ) {
            u = ccvt<CT>(av[b]);
            v = ccvt<CT>(bv[b]);
          } else {
            const CT a0 = ccvt<CT>(av[b]), b0 = ccvt<CT>(bv[b]);
            u.x = fma(sB, b0.x, a0.x); u.y = fma(sB, b0.y, a0.y);
            v.x = fma(-sB, b0.x, a0.x); v.y = fma(-sB, b0.y, a0.y);
          }
          ra.x = fma(u.x, xv.x, ra.x); ra.x = fma(-v.y, xv.y, ra.x);    // (M_s x_J)_r
          ra.y = fma(u.y, xv.x, ra.y); ra.y = fma(v.x, xv.y, ra.y);
          if (!diag) {                                                  // (M_s^T x_I)_c
            cacc[b].x = fma(u.x, y.x, cacc[b].x); cacc[b].x = fma(u.y, y.y, cacc[b].x);
            cacc[b].y = fma(v.x, y.y, cacc[b].y); cacc[b].y = fma(-v.y, y.x, cacc[b].y);
          }
        } else {
          const CT A = ccvt<CT>(av[b]);
          cfma(ra, A, xv);                      // (A_IJ x_J)_r
          if (!diag) cfmac(cacc[b], A, y);      // (A_IJ^H x_I)_c
        }
      }
      racc[a] = ra;
    }
    // ---- row sums: reduce-scatter over the 16 tx lanes (xor 8, 4, 2, 1)
    {
      const bool u8 = tx & 8;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        CT send = u8 ? racc[q] : racc[q + 4];
        CT keep = u8 ? racc[q + 4] : racc[q];
        racc[q] = cadd(keep, shfl_xor_c(send, 8));
      }
      const bool u4 = tx & 4;
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        CT send = u4 ? racc[q] : racc[q + 2];
        CT keep = u4 ? racc[q + 2] : racc[q];
        racc[q] = cadd(keep, shfl_xor_c(send, 4));
      }
      const bool u2 = tx & 2;
      {
        CT send = u2 ? racc[0] : racc[1];
        CT keep = u2 ? racc[1] : racc[0];
        racc[0] = cadd(keep, shfl_xor_c(send, 2));
      }
      racc[0] = cadd(racc[0], shfl_xor_c(racc[0], 1));
      if ((tx & 1) == 0) {
        const int a = (tx >> 1) & 7;
        const int r = ty + 16 * a;
        CT* part = (CT*)p.part;
        part[((int64_t)jb.I * p.nT + jb.J) * TS + r] = racc[0];
      }
    }
    if (!diag) {
      // ---- column sums: pair the two ty of a warp (xor 16), then across warps
      const bool up = lane & 16;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        CT send = up ? cacc[q] : cacc[q + 4];
        CT keep = up ? cacc[q + 4] : cacc[q];
        cacc[q] = cadd(keep, shfl_xor_c(send, 16));
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) red[warp][tx + 16 * (q + (up ? 4 : 0))] = cacc[q];
      __syncthreads();
      if (tid < TS) {
        CT s = red[0][tid];
#pragma unroll
        for (int w = 1; w < 8; ++w) s = cadd(s, red[w][tid]);
        CT* part = (CT*)p.part;
        part[((int64_t)jb.J * p.nT + jb.I) * TS + tid] = s;
      }
    }
  }
}

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int m = 16; m >= 1; m >>= 1) v += __shfl_xor_sync(0xffffffffu, v, m);
  return v;
}

// The products whose result closes a Krylov vector: their reduction leaves the partial sums of the
// squared norm Re(w^H M w) (one per 32 rows), so that the normalisation needs no pass of its own.
__device__ __forceinline__ bool prod_is_norm(int mode) {
  return mode == PM_STEP_MPLUS || mode == PM_START_MPLUS || mode == PM_STEP_MMINUS_W;
}
template <typename ST>
__device__ __forceinline__ double norm_term(ST a, ST b) {
  return (double)a.x * (double)b.x + (double)a.y * (double)b.y;
}

// y[I*TS + r] = sum_J part[I][J][r].  A unit is 32 rows of a block row: 8 warps, lane = row, warp
// g sums the slots J = g, g + 8, ... in order, and the eight group sums are added in group order
// (a fixed rounding order).  FP64 adds cost 64 clocks per warp and scheduler on this GPU, so the
// rows are spread over four times as many CTAs as there are block rows.
constexpr int REDUCE_GROUPS = 8;
constexpr int REDUCE_ROWS = 32;
constexpr int REDUCE_UNITS = TS / REDUCE_ROWS;       // units of a block row

// One unit: rows 32 (u % 4) ... of block row u / 4 of problem ip; grp: REDUCE_GROUPS x 32 entries
// of shared memory.
template <typename ST, typename R, bool COH = false>
__device__ __forceinline__ void prod_reduce_body(const Prob* __restrict__ probs, int mode, const GenericIO& io,
                                                 int u, int ip, typename Acc<R>::T (*grp)[REDUCE_ROWS]) {
  using CT = typename Acc<R>::T;
  const Prob& p = probs[ip];
  const int I = u / REDUCE_UNITS;
  if (I >= p.nT) return;
  const ST* x; ST* y; R sB;
  if (!prod_operands<ST, R>(p, mode, io, x, y, sB)) return;
  const int lane = threadIdx.x & 31, g = threadIdx.x >> 5;
  const int r = (u % REDUCE_UNITS) * REDUCE_ROWS + lane;
  const CT* part = (const CT*)p.part + (int64_t)I * p.nT * TS;
  CT acc = czero<CT>();
  int J = g;
  for (; J + 3 * REDUCE_GROUPS < p.nT; J += 4 * REDUCE_GROUPS) {   // four loads in flight, then the sums
    CT v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = ldv<COH>(part + (int64_t)(J + k * REDUCE_GROUPS) * TS + r);
#pragma unroll
    for (int k = 0; k < 4; ++k) acc = cadd(acc, v[k]);
  }
  for (; J < p.nT; J += REDUCE_GROUPS) acc = cadd(acc, ldv<COH>(part + (int64_t)J * TS + r));
  if constexpr (std::is_same<CT, double2>::value) {
    // fixed-point tiles: the column sums of a tile's further bands, planes 1 ... nq - 1
    const int nb = p.nq - 1;
    for (int k = g; k < nb * I; k += REDUCE_GROUPS) {
      const int q = 1 + k / I, Jq = k - (q - 1) * I;
      if (p.texp[(int64_t)Jq * p.nT - (int64_t)Jq * (Jq - 1) / 2 + (I - Jq)] < 0) continue;
      acc = cadd(acc, ldv<COH>(part + ((int64_t)q * p.nT * p.nT + Jq) * TS + r));
    }
  }
  grp[g][lane] = acc;
  __syncthreads();
  if (g == 0) {
#pragma unroll
    for (int q = 1; q < REDUCE_GROUPS; ++q) acc = cadd(acc, grp[q][lane]);
    const int64_t row = (int64_t)I * TS + r;
    if constexpr (std::is_same<CT, double2>::value) {
      // ... and the diagonal entry, which a fixed-point diagonal tile leaves out
      const int64_t t = (int64_t)I * p.nT - (int64_t)I * (I - 1) / 2;
      if (p.nq > 0 && p.texp[t] >= 0) {
        const int64_t d = t * (TS * TS) + r * (TS + 1);
        const CT xv = ldv<COH>((const CT*)x + row);
        const CT u = ((const CT*)(p.ph && sB < (R)0 ? p.B : p.A))[d];
        const CT v = p.ph ? ((const CT*)(sB < (R)0 ? p.A : p.B))[d] : u;
        acc.x = fma(u.x, xv.x, acc.x); acc.x = fma(-v.y, xv.y, acc.x);
        acc.y = fma(u.y, xv.x, acc.y); acc.y = fma(v.x, xv.y, acc.y);
      }
    }
    const ST yv = ccvt<ST>(acc);
    y[row] = yv;
    if (prod_is_norm(mode)) {          // the squared norm's partial sum Re(w^H M w)
      const double s = norm_term(ldv<COH>(x + row), yv);
      const double t = warp_sum_d(s);
      if (lane == 0) p.npart[u] = t;
    }
  }
  __syncthreads();                     // grp is rewritten by the next unit
}

// ---------------------------------------------------------------- CGS2 dots
// PH: cpart[k][c] = sum_{rows in chunk k} Re(conj(Dm[row, c]) x[row]) for c < nm and
// Im(conj(Dt[row, c']) x[row]) for c = nm + c' (the twin coefficients), nm + nt in all;
// TDA: the complex conj(V[row, c]) x[row], c <= j.  A warp-wide FP64 instruction takes 64 clocks
// of its scheduler, so the work is cut into one-warp tasks (a column on a chunk of rows) that
// spread evenly over all schedulers of the GPU; at most DOT_CHUNKS chunks, whole tiles each.  A lane's
// FP32 sums go to FP64 every DOT_RUN rounds of four rows, so their rounding does not grow with N.
constexpr int DOT_RUN = 4;
__host__ __device__ __forceinline__ int dot_chunk_tiles(int nT) { return (nT + DOT_CHUNKS - 1) / DOT_CHUNKS; }
__host__ __device__ __forceinline__ int dot_chunks(int nT) {
  return (nT + dot_chunk_tiles(nT) - 1) / dot_chunk_tiles(nT);
}

// One task (a warp): column c of the set, chunk k.
template <typename ST, bool COH>
__device__ __forceinline__ void cgs_dot_task(const Prob& p, const KState* st, const CgsSet& cs, int ph, int newvec,
                                             int half, int pass, int c, int k) {
  using R = typename RealOf<ST>::T;
  const int lane = threadIdx.x & 31;
  const bool twin = c >= cs.nm;                         // warp-uniform
  const int col = twin ? c - cs.nm : c;
  const int64_t rows = (int64_t)dot_chunk_tiles(p.nT) * TS;
  const int64_t r0 = k * rows, r1 = min(p.Npad, r0 + rows);
  const ST* Q = (const ST*)(twin ? cs.dt : cs.dm) + (int64_t)col * p.Npad;
  const ST* w = cgs_src<ST>(p, st, half, pass, newvec);
  int64_t r = r0 + lane;
  if (ph) {   // real coefficients: Re(conj(q) x), or Im(conj(q) x) = Re(conj(q) (-i x)) for twins
    R a1 = 0, a2 = 0;   // two chains (x and y products)
    double s = 0.0;
    for (int n = 1; r < r1; r += 4 * 32, ++n) {                       // whole tiles: four rows per lane and round
      ST q[4], x[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        q[u] = ldv<COH>(Q + r + 32 * u);
        x[u] = ldv<COH>(w + r + 32 * u);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        a1 = fma(q[u].x, twin ? x[u].y : x[u].x, a1);
        a2 = fma(q[u].y, twin ? -x[u].x : x[u].y, a2);
      }
      if (sizeof(R) == 4 && n % DOT_RUN == 0) {
        s += (double)a1 + (double)a2;
        a1 = a2 = 0;
      }
    }
    const double t = warp_sum_d(sizeof(R) == 4 ? s + ((double)a1 + (double)a2) : (double)a1 + (double)a2);
    if (lane == 0) p.cpart[(int64_t)k * p.ncol + c] = t;
  } else {
    ST acc = czero<ST>();
    double2 a = mk(0.0, 0.0);
    for (int n = 1; r < r1; r += 4 * 32, ++n) {
      ST q[4], x[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        q[u] = ldv<COH>(Q + r + 32 * u);
        x[u] = ldv<COH>(w + r + 32 * u);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) cfmac(acc, q[u], x[u]);
      if (sizeof(R) == 4 && n % DOT_RUN == 0) {
        a = cadd(a, mk((double)acc.x, (double)acc.y));
        acc = czero<ST>();
      }
    }
    a = sizeof(R) == 4 ? cadd(a, mk((double)acc.x, (double)acc.y)) : mk((double)acc.x, (double)acc.y);
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1) a = cadd(a, dshfl(a, m));
    if (lane == 0) ((double2*)p.cpart)[(int64_t)k * p.ncol + c] = a;
  }
}

// ---------------------------------------------------------------- CGS2 updates
// w[row] = x[row] - sum_{c < nm} Um[row, c] coef[pass][c] (- i sum_{c'} Ut[row, c'] coef[pass][nm+c']
// on the PH paths: the twin projection).  A unit is a slab of 8, 16 or 32 rows (Prob::slab: the
// smallest that does not give more units than there are SMs; every unit sums the dots'
// partial sums itself, so more of them cost more than they spread): a thread owns one row and every (256 / rows)-th
// column of the set, and the partial sums meet in shared memory.
// the sum of column c's partial dots over the chunks, in chunk order
template <bool COH>
__device__ __forceinline__ double2 cgs_coef(const Prob& p, int ph, int c, int nch) {
  double2 sc = mk(0.0, 0.0);
  if (ph) {
    double v[DOT_CHUNKS];
#pragma unroll
    for (int k = 0; k < DOT_CHUNKS; ++k) v[k] = k < nch ? ldv<COH>(p.cpart + (int64_t)k * p.ncol + c) : 0.0;
    sc.x = v[0];
    for (int k = 1; k < nch; ++k) sc.x += v[k];
  } else {
    const double2* cp = (const double2*)p.cpart;
    for (int k = 0; k < nch; ++k) sc = cadd(sc, ldv<COH>(cp + (int64_t)k * p.ncol + c));
  }
  return sc;
}

// One unit: slab bx of problem ip; cf: 2 MAXM + 2 entries and red: 8 x 32 entries of shared memory.
template <typename ST, bool COH, int RS>
__device__ __forceinline__ void cgs_update_slab(const Prob& p, const KState* st, int ph, int pass, int newvec, int half,
                                                int bx, ST* cf, ST (*red)[32]) {
  using R = typename RealOf<ST>::T;
  constexpr int G = 256 / RS;                 // column groups
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const CgsSet cs = cgs_set(p, st, ph, half);
  const int nm = cs.nm;
  const int nset = nm + cs.nt;
  const int nch = dot_chunks(p.nT);
  const int64_t row = (int64_t)bx * RS + (tid & (RS - 1));
  const ST* vb = (const ST*)cs.um + row;
  const ST* pb = ph ? (const ST*)cs.ut + row : nullptr;
  // Loads in flight per thread, the first of them beside the sums of the coefficients.  A TDA cycle at
  // N = 2000 took 31.2 ms of steps and restarts with 4, 32.4 with 6, 33.1 with 8 (32.5 with the loads
  // behind the coefficients); a pseudo-Hermitian one at 3000 243.7, 246.6, 247.2 (251).
  // FP32 has a sum for each of eight loads: one sum alone would be a chain of nset / 8 roundings.
  constexpr int U = sizeof(R) == 4 ? 8 : 4, NA = sizeof(R) == 4 ? U : 1;
  const int64_t ld = p.Npad;
  // entry cc of the set: Um[:, cc] for cc < nm, else the twin's Ut[:, cc - nm]
  auto load = [&](int cc) -> ST { return ldv<COH>(cc < nm ? vb + (int64_t)cc * ld : pb + (int64_t)(cc - nm) * ld); };
  const int c0 = tid / RS;
  ST v[U];
#pragma unroll
  for (int u = 0; u < U; ++u)                 // the first round does not wait for the coefficients
    if (c0 + G * u < nset) v[u] = load(c0 + G * u);
  // coefficients; the first slab also stores them for the step's end
  double2* coef = (double2*)p.coef + (int64_t)(pass & 1) * p.ncol;
  for (int c = tid; c < nset; c += 256) {
    const double2 sc = cgs_coef<COH>(p, ph, c, nch);
    cf[c] = ccvt<ST>(sc);
    if (bx == 0) coef[c] = sc;
  }
  __syncthreads();
  ST acc[NA];
#pragma unroll
  for (int u = 0; u < NA; ++u) acc[u] = czero<ST>();
  for (int c = c0; c < nset; c += G * U) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int cc = c + G * u;
      if (cc >= nset) continue;
      ST& part = acc[u % NA];
      if (ph) {                               // real coefficients; the twin i t = (-t.y, t.x)
        const R f = cf[cc].x;
        const bool tw = cc >= nm;
        part.x = fma(tw ? -v[u].y : v[u].x, f, part.x);
        part.y = fma(tw ? v[u].x : v[u].y, f, part.y);
      } else {
        cfma(part, v[u], cf[cc]);
      }
    }
    if (c + G * U < nset) {
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (c + G * (U + u) < nset) v[u] = load(c + G * (U + u));
    }
  }
  ST part = acc[0];
#pragma unroll
  for (int u = 1; u < NA; ++u) part = cadd(part, acc[u]);
#pragma unroll
  for (int m = RS; m < 32; m <<= 1) part = cadd(part, shfl_xor_c(part, m));   // the warp's groups
  if (lane < RS) red[warp][lane] = part;
  __syncthreads();
  // eight sums per row and component: a lane per sum
  const ST* x = cgs_src<ST>(p, st, half, pass, newvec);
  ST* w = (ST*)p.w;
  double nrm = 0.0;
#pragma unroll
  for (int v = tid; v < RS * 16; v += 256) {
    const int r = v >> 4, comp = (v >> 3) & 1;
    const R* e = reinterpret_cast<const R*>(&red[v & 7][r]);
    R t = e[comp];
#pragma unroll
    for (int m = 1; m < 8; m <<= 1) t += __shfl_xor_sync(0xffffffffu, t, m);
    if ((v & 7) == 0) {
      const int64_t o = ((int64_t)bx * RS + r) * 2 + comp;
      const R nw = ldv<COH>((const R*)x + o) - t;
      ((R*)w)[o] = nw;
      nrm += (double)nw * (double)nw;
    }
  }
  if (!ph && (pass & 1)) {                  // TDA: the squared norm's partial sum of the slab
    nrm = warp_sum_d(nrm);
    __syncthreads();
    double* rd = reinterpret_cast<double*>(red);
    if (lane == 0) rd[warp] = nrm;
    __syncthreads();
    if (tid == 0) {
      double t = rd[0];
      for (int q = 1; q < (RS * 16 < 256 ? RS * 16 / 32 : 8); ++q) t += rd[q];
      p.npart[bx] = t;
    }
  }
}

template <typename ST, bool COH>
__device__ __forceinline__ void cgs_update_unit(const Prob& p, const KState* st, int ph, int pass, int newvec, int half,
                                                int bx, ST* cf, ST (*red)[32]) {
  switch (p.slab) {
    case 8: return cgs_update_slab<ST, COH, 8>(p, st, ph, pass, newvec, half, bx, cf, red);
    case 16: return cgs_update_slab<ST, COH, 16>(p, st, ph, pass, newvec, half, bx, cf, red);
    default: return cgs_update_slab<ST, COH, 32>(p, st, ph, pass, newvec, half, bx, cf, red);
  }
}

// ---------------------------------------------------------------- norms
// Partial sums of a new vector's squared norm: per 32 rows on the PH paths (the reduction of the
// closing product), per slab of the last Gram-Schmidt update on the TDA path.
__device__ __forceinline__ int norm_parts(const Prob& p, int ph) {
  return (int)(p.Npad / (ph ? REDUCE_ROWS : p.slab));
}

// their sum in every lane of a warp, in a fixed order
template <bool COH>
__device__ __forceinline__ double norm_sum(const Prob& p, int ph) {
  const int n = norm_parts(p, ph);
  double s = 0.0;
  for (int i = threadIdx.x & 31; i < n; i += 32) s += ldv<COH>(p.npart + i);
  return warp_sum_d(s);
}

// Where a normalised vector goes: V[:, j+1] (and P) for the folded / TDA step and the even
// half of a Gruning step, W[:, j] (and Z) for the odd half.
template <typename ST>
__device__ __forceinline__ void norm_dest(const Prob& p, const KState* st, int half, ST*& X, ST*& Y) {
  if (half == 1) {
    X = (ST*)p.W + (int64_t)st->j * p.Npad;
    Y = (ST*)p.Z + (int64_t)st->j * p.Npad;
  } else {
    X = (ST*)p.V + (int64_t)(st->j + 1) * p.Npad;
    Y = p.ph ? (ST*)p.P + (int64_t)(st->j + 1) * p.Npad : nullptr;
  }
}

// The double-FP32 shadows of a new V (and P) column, where the problem keeps them.
template <typename ST>
__device__ __forceinline__ void shadow_store(const Prob& p, const KState* st, int half, int64_t row, ST xv, ST yv) {
  if constexpr (std::is_same<ST, double2>::value) {
    if (p.Vs && half != 1) {
      const int64_t o = (int64_t)(st->j + 1) * p.Npad + row;
      p.Vs[o] = dsplit(xv);
      if (p.ph) p.Ps[o] = dsplit(yv);
    }
  }
}

// X = w / beta, Y = pw / beta (norm_dest) for one row, beta^2 = b2 > 0 and finite
template <typename ST, bool COH>
__device__ __forceinline__ void normalize_row(const Prob& p, const KState* st, int ph, int half, int64_t row,
                                              typename RealOf<ST>::T inv) {
  ST *X, *Y;
  norm_dest<ST>(p, st, half, X, Y);
  const ST xv = cscale(ldv<COH>((const ST*)p.w + row), inv);
  X[row] = xv;
  ST yv = czero<ST>();
  if (ph) Y[row] = yv = cscale(ldv<COH>((const ST*)p.pw + row), inv);
  shadow_store<ST>(p, st, half, row, xv, yv);
}

// Record alpha_j, beta_j, advance j, given beta^2 = b2 of the new vector.  fresh = 0:
// regular step; fresh = 1: a first or replacement vector was just normalised.
// p.st is a copy of the state that is not yet in use (k_normalize) or each CTA's own (k_persist.cu);
// one of the CTAs (`writer`) also stores alpha and beta.
template <bool COH>
__device__ __forceinline__ void step_finish_one(const Prob& p, int ph, int fresh, double b2, bool writer) {
  KState* st = p.st;
  const int j = st->j;
  if (!fresh) {
    const double2* coef = (const double2*)p.coef;
    const double a = ldv<COH>(&coef[j].x) + ldv<COH>(&coef[p.ncol + j].x);
    if (!isfinite(a) || !isfinite(b2)) { st->status = ST_NOTFINITE; return; }
    if (writer) p.alpha[j] = a;
    st->passes += ph ? 2 : 1;
    st->steps += 1;
    // scale of the projected matrix for the breakdown test
    double scale = fabs(a);
    scale = fmax(scale, st->theta_scale);   // max |theta| of the kept Ritz values
    if (j > 0) scale = fmax(scale, fabs(ldv<COH>(p.beta + j - 1)));
    const double tiny = 1e-26 * scale * scale + 1e-300;
    if (ph && b2 < -1e6 * tiny) { st->status = ST_NOTPD; return; }
    if (b2 <= tiny) {                 // invariant subspace: the chain restarts
      if (writer) p.beta[j] = 0.0;    // with a fresh vector (host-driven), unless the subspace is full
      if (j + 1 < st->m) st->breakdown = 1;     // (then its Ritz pairs are exact and all lock; a fresh
      else st->j = j + 1;                       // vector may not even exist: m = N)
      return;
    }
    if (writer) p.beta[j] = sqrt(b2);
    st->j = j + 1;
  } else {
    if (!isfinite(b2)) { st->status = ST_NOTFINITE; return; }
    if (!(b2 > 0.0)) { st->status = ph ? ST_NOTPD : ST_NOTFINITE; return; }
    st->breakdown = 0;
    st->passes += ph ? 1 : 0;
    st->j = j + 1;
  }
  if (st->steps >= st->maxit && !st->done) { st->done = 1; st->status = ST_NOCONV; }
}

// Gruning step: record alpha_j (odd half) or beta_j and advance j (even half), given the
// squared M-norm b2 of the new vector; fresh = 1: a first or replacement even vector.
// An odd vector cannot vanish when M+ is positive definite (M+ maps the j + 1 even
// vectors onto j + 1 independent odd ones), so a vanishing alpha means not definite.
__device__ __forceinline__ void gk_finish_one(const Prob& p, int half, int fresh, double b2, bool writer) {
  KState* st = p.st;
  const int j = st->j;
  if (!isfinite(b2)) { st->status = ST_NOTFINITE; return; }
  if (fresh) {
    if (!(b2 > 0.0)) { st->status = ST_NOTPD; return; }
    st->breakdown = 0;
    st->passes += 1;
    st->j = j + 1;
  } else {
    double scale = 0.0;
    scale = fmax(scale, st->theta_scale);   // max |theta| of the kept Ritz values
    if (j > 0) scale = fmax(scale, p.beta[j - 1]);
    if (half == 2) scale = fmax(scale, p.alpha[j]);
    const double tiny = 1e-26 * scale * scale + 1e-300;
    if (b2 < -1e6 * tiny) { st->status = ST_NOTPD; return; }
    if (half == 1) {
      if (b2 <= tiny) { st->status = ST_NOTPD; return; }
      if (writer) p.alpha[j] = sqrt(b2);
      return;                           // the even half follows in the same step
    }
    st->passes += 2;
    st->steps += 1;
    if (b2 <= tiny) {                   // invariant subspace: the chain restarts
      if (writer) p.beta[j] = 0.0;      // with a fresh vector (host-driven), unless the subspace is full
      if (j + 1 < st->m) st->breakdown = 1;
      else st->j = j + 1;
      return;
    }
    if (writer) p.beta[j] = sqrt(b2);
    st->j = j + 1;
  }
  if (st->steps >= st->maxit && !st->done) { st->done = 1; st->status = ST_NOCONV; }
}

template <bool COH>
__device__ __forceinline__ void finish_one(const Prob& p, int ph, int fresh, int half, double b2, bool writer) {
  if (half) gk_finish_one(p, half, fresh, b2, writer);
  else step_finish_one<COH>(p, ph, fresh, b2, writer);
}


}  // namespace bse
