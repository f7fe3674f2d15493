// Y = A XA + B XB for blocks of columns in FP64 accuracy on the integer pipe: the residual
// products H z of every returned pair, and bse_apply on blocks of complex128 vectors.
//
// The FP64 row-block kernel (k_prod_rowblock) is bound by the two-lane FP64 pipe and, at the orders
// where a solve takes a fraction of a second, by its few CTAs (one per block row and 16 columns).
// Here a real FMA is three integer multiply-adds (fx_phases.cuh: 30-bit limbs under a scale per
// tile and per 128-entry chunk of a column), the block columns J are split over CTAs as well, and
// the partial sums of the splits meet in FP64 in a fixed order.
//
// In real arithmetic one stored element pair has four real coefficients (p, q, r, t) and adds
//     y += p z0 + q z1 + r z2 + t z3,    z complex
// to an output: for complex128 PH tiles (P = A + B, Q = A - B, s = (XA + XB) / 2, d = (XA - XB) / 2)
//     P s + Q d                        (z = s, i s, d, i d)      tile (I, J), J >= I
//     P_re s - i P_im d + Q_re d - i Q_im s                      tile (J, I), A = A^H, B = B^T
// and for complex64 tiles (A, B) the same with z = XA, +-i XA, XB, i XB; A alone has two terms.  So
// the inner loop is one for all, and the forms differ in how a chunk of X is staged.
//
// Unit: 64 rows x 16 columns, 256 threads of 2 x 2 outputs; 8 steps of q staged at a time.  Every
// two (hl) or four (hh) q a sum's bits above 2^38 move to a 32-bit counter, so it stays exact over a whole tile; then
// it becomes one FP64 number (integer instructions; formed again in FP64 where it is too small for the error
// of its scales, fx_weak) and is added.  Measured against
// k_prod_rowblock: H on 20 vectors at N = 1500, complex128, 6.8 -> 0.50 ms a call; the residuals of 32
// pairs at N = 5000, complex64 storage, 42.7 -> 6.4 ms; of 20 pairs at N = 2000, TDA, 4.3 -> 0.28 ms.
#include <algorithm>

#include "fx_phases.cuh"

namespace bse {
namespace {

constexpr int BR = 64;       // rows of a unit
constexpr int BC = 16;       // columns of a unit
constexpr int BQ = 8;        // inner indices staged at a time
constexpr int BRP = BR + 1;  // padded row stride of the staged tile (conflict-free both ways)

// limbs of a block of columns: F0 (s or XA) and F1 (d or XB), column c at c Npad, and the scale
// exponent of chunk I (and its strong entries, as in texp) at E[c nT + I]; grid (nT, K), TS threads
template <bool HASB, bool PQ>
__global__ void __launch_bounds__(TS)
k_block_stage(const double2* __restrict__ xa, const double2* __restrict__ xb, int64_t ldx, double sB, int64_t Npad,
              int nT, int4* __restrict__ F0, int4* __restrict__ F1, int* __restrict__ E) {
  __shared__ unsigned int smx[TS / 32];
  __shared__ int sst[TS / 32];
  const int c = blockIdx.y, tid = threadIdx.x;
  const int64_t r = (int64_t)blockIdx.x * TS + tid;
  double2 a = xa[c * ldx + r], b = make_double2(0.0, 0.0);
  if (HASB) {
    b = xb ? xb[c * ldx + r] : conjc(a);
    b = cscale(b, sB);
    if (PQ) {
      a = cscale(a, 0.5);                // halves first: the sum of two large entries stays finite
      b = cscale(b, 0.5);
      const double2 s = cadd(a, b), d = csub(a, b);
      a = s;
      b = d;
    }
  }
  unsigned int m = max(hi_abs(a.x), hi_abs(a.y));
  if (HASB) m = max(m, max(hi_abs(b.x), hi_abs(b.y)));
  m = __reduce_max_sync(0xffffffffu, m);
  if ((tid & 31) == 0) smx[tid >> 5] = m;
  __syncthreads();
  m = max(max(smx[0], smx[1]), max(smx[2], smx[3]));
  const int e = max(1, (int)(m >> 20));
  F0[c * Npad + r] = fx_entry(a, e);
  if (HASB) F1[c * Npad + r] = fx_entry(b, e);
  // strong entries: both vectors' (a sum P s + Q d is only as large as its smaller pairing)
  unsigned int h = max(hi_abs(a.x), hi_abs(a.y));
  if (HASB) h = min(h, max(hi_abs(b.x), hi_abs(b.y)));
  const unsigned int st = __ballot_sync(0xffffffffu, h + (FX_STRONG << 20) >= m);
  if ((tid & 31) == 0) sst[tid >> 5] = __popc(st);
  __syncthreads();
  if (tid == 0) E[(int64_t)c * nT + blockIdx.x] = e | ((sst[0] + sst[1] + sst[2] + sst[3]) << FX_EBITS);
}

// scales of complex64 tiles, -1 for those a fixed-point product must not take (as k_fx_pack)
template <bool HASB>
__global__ void __launch_bounds__(256)
k_block_scale64(const float2* __restrict__ A, const float2* __restrict__ B, int64_t N, int nT, int* __restrict__ texp) {
  const int I = blockIdx.y, J = blockIdx.x;
  if (J < I) return;
  const int64_t t = (int64_t)I * nT - (int64_t)I * (I - 1) / 2 + (J - I);
  __shared__ float smx[8], smn[8];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nr = (int)min((int64_t)TS, N - (int64_t)I * TS), nc = (int)min((int64_t)TS, N - (int64_t)J * TS);
  float m = 0.f, mn = INFINITY;
  bool bad = false;
  for (int e = tid; e < TS * TS; e += 256) {
    const float2 a = A[t * (TS * TS) + e], b = HASB ? B[t * (TS * TS) + e] : make_float2(0.f, 0.f);
    const float v = fmaxf(fmaxf(fabsf(a.x), fabsf(a.y)), fmaxf(fabsf(b.x), fabsf(b.y)));
    if ((e >> 7) < nr && (e & (TS - 1)) < nc) mn = fminf(mn, v);
    if (I == J && (e >> 7) == (e & (TS - 1))) continue;
    m = fmaxf(m, v);
    bad |= !(isfinite(a.x) && isfinite(a.y) && isfinite(b.x) && isfinite(b.y));
  }
#pragma unroll
  for (int k = 16; k >= 1; k >>= 1) {
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, k));
    mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, k));
  }
  if (lane == 0) { smx[warp] = m; smn[warp] = mn; }
  const bool any_bad = __syncthreads_or(bad ? 1 : 0);
  if (tid == 0) {
    for (int w = 1; w < 8; ++w) { m = fmaxf(m, smx[w]); mn = fminf(mn, smn[w]); }
    const int ex = (int)((__float_as_uint(m) >> 23) & 0xffu) + 896;      // FP64 bias
    // (entries far below 2^-100 would leave the FP32 range of the limbs' conversion)
    const bool ok = !any_bad && (m == 0.f || (m > 1e-25f && m < 1e25f && m <= (float)(1 << FX_SPREAD) * mn));
    texp[t] = !ok ? -1 : (m == 0.f ? 1 : ex);
  }
}

// limbs of a float under the scale 2^(e - 1022) (exact down to 2^-59 of it)
__device__ __forceinline__ void fx_limbs32(float v, int e, int& hi, int& lo) {
  const unsigned int b = __float_as_uint(v);
  const int d = e - ((int)((b >> 23) & 0xffu) + 896);
  unsigned long long m = (b & 0x7f800000u) ? (unsigned long long)((b & 0x7fffffu) | 0x800000u) << 35 : 0ull;
  m = d > 0 ? ((m >> (min(d, 63) - 1)) + 1) >> 1 : m;
  const long long f = d < 62 ? ((int)b < 0 ? -(long long)m : (long long)m) : 0ll;
  fx_limbs(f, hi, lo);
}

// (A, B) of a packed element
template <int MODE>
__device__ __forceinline__ void block_element(const void* A, const void* B, int64_t o, double2& a, double2& b) {
  if (MODE & 1) {
    a = ccvt<double2>(((const float2*)A)[o]);
    if (MODE < 2) b = ccvt<double2>(((const float2*)B)[o]);
  } else {
    a = ((const double2*)A)[o];
    if (MODE < 2) {                      // stored P = A + B, Q = A - B
      const double2 p = a, q = ((const double2*)B)[o];
      a = cscale(cadd(p, q), 0.5);
      b = cscale(csub(p, q), 0.5);
    }
  }
}

// an exact sum over a tile: value = (x 2^38 + v), |v| < 2^63
struct FxAcc {
  long long v;
  int x;
};
__device__ __forceinline__ void fx_carry(FxAcc& a) {
  a.x += (int)(a.v >> 38);
  a.v &= (1ll << 38) - 1;
}

// (hh 2^30 + hl) 2^(eu + ex - 2044 - 88) as a double
__device__ __forceinline__ double fx_acc_double(const FxAcc& hh, const FxAcc& hl, int eu, int ex) {
  const __int128 t = ((((__int128)hh.x << 38) + hh.v) << 30) + (((__int128)hl.x << 38) + hl.v);
  return fx_pack_double((long long)(t >> 68), (unsigned long long)(t >> 16) & 0xfffffffffffffull, eu, ex);
}

// what the sums in FP64 read (A null: none are formed)
struct BlockExact {
  const void* A;
  const void* B;
  const double2* xa;
  const double2* xb;
  int64_t ldx, N;
  double sB;
};

// One output of a tile in FP64, by a warp (in every lane): row r of block row I times chunk J of a column;
// A, B, xa, xb as for k_block_sum, the matrix diagonal left out
template <int MODE>
__device__ __noinline__ double2 block_exact(const void* A, const void* B, int64_t t, bool upper, bool diag, int r,
                                            const double2* xa, const double2* xb, double sB) {
  constexpr bool HASB = MODE < 2;
  double2 y = make_double2(0.0, 0.0);
  for (int q = threadIdx.x & 31; q < TS; q += 32) {
    if (diag && q == r) continue;
    const int64_t o = t * (TS * TS) + (upper ? r * TS + q : q * TS + r);
    double2 a, b = make_double2(0.0, 0.0);
    block_element<MODE>(A, B, o, a, b);
    cfma(y, upper ? a : conjc(a), xa[q]);
    if (HASB) cfma(y, b, cscale(xb ? xb[q] : conjc(xa[q]), sB));
  }
  return make_double2(warp_sum_d(y.x), warp_sum_d(y.y));
}

// MODE 0: complex128 PH (P, Q limbs); 1: complex64 PH (A, B); 2: complex128 TDA (A limbs);
// 3: complex64 TDA.  grid (2 nT, ceil(K / BC), splits); part: splits x K x Npad
template <int MODE>
__global__ void __launch_bounds__(256, 2)
k_block_fx(const void* __restrict__ M0, const void* __restrict__ M1, const int* __restrict__ texp, int nT, int64_t Npad,
           const int4* __restrict__ F0, const int4* __restrict__ F1, const int* __restrict__ E, int K,
           double2* __restrict__ part, const BlockExact ax) {
  constexpr bool HASB = MODE < 2, F32 = MODE & 1;
  constexpr int NZ = HASB ? 4 : 2;
  __shared__ int4 sm0[BQ * BRP];
  __shared__ int4 sm1[HASB ? BQ * BRP : 1];
  __shared__ int4 sz[BQ][NZ][BC];
  const int I = blockIdx.x >> 1, rh = (blockIdx.x & 1) * BR;
  const int c0 = blockIdx.y * BC;
  const int tid = threadIdx.x, rp = tid & 31, cp = tid >> 5;
  const int per = (nT + gridDim.z - 1) / gridDim.z;
  const int J0 = blockIdx.z * per, J1 = min(nT, J0 + per);
  double2 y[2][2];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) y[i][j] = make_double2(0.0, 0.0);
  for (int J = J0; J < J1; ++J) {
    const bool upper = J >= I;
    const int ti = upper ? I : J, tj = upper ? J : I;
    const int64_t t = (int64_t)ti * nT - (int64_t)ti * (ti - 1) / 2 + (tj - ti);
    const int te = texp[t], eu = te & FX_EMASK;
    FxAcc hh[2][2][2], hl[2][2][2];      // [row][column][re, im]
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int k = 0; k < 2; ++k) hh[i][j][k] = hl[i][j][k] = FxAcc{0, 0};
    for (int q0 = 0; q0 < TS; q0 += BQ) {
      __syncthreads();
      // BQ x BR entries of the tile, q along the rows of the product
      for (int e = tid; e < BQ * BR; e += 256) {
        const int q = upper ? e % BQ : e / BR, r = upper ? e / BQ : e % BR;
        const int64_t off = t * (TS * TS) + (upper ? (rh + r) * TS + q0 + q : (q0 + q) * TS + rh + r);
        const bool dg = I == J && rh + r == q0 + q;       // the diagonal is added in FP64
        int4 u, w = make_int4(0, 0, 0, 0);
        if (F32) {
          const float2 a = __ldg((const float2*)M0 + off);
          fx_limbs32(a.x, eu, u.x, u.y);
          fx_limbs32(a.y, eu, u.z, u.w);
          if (HASB) {
            const float2 b = __ldg((const float2*)M1 + off);
            fx_limbs32(b.x, eu, w.x, w.y);
            fx_limbs32(b.y, eu, w.z, w.w);
          }
          if (dg) u = w = make_int4(0, 0, 0, 0);
        } else {
          u = __ldg((const int4*)M0 + off);
          if (HASB) w = __ldg((const int4*)M1 + off);
        }
        sm0[q * BRP + r] = u;
        if (HASB) sm1[q * BRP + r] = w;
      }
      if (tid < BQ * BC) {
        const int q = tid % BQ, c = tid / BQ;
        int4 a = make_int4(0, 0, 0, 0), b = a;
        if (c0 + c < K) {
          const int64_t o = (int64_t)(c0 + c) * Npad + (int64_t)J * TS + q0 + q;
          a = F0[o];
          if (HASB) b = F1[o];
        }
        // i z = (-z_im, z_re), -i z = (z_im, -z_re)
        auto ipos = [](int4 z) { return make_int4(-z.z, -z.w, z.x, z.y); };
        auto ineg = [](int4 z) { return make_int4(z.z, z.w, -z.x, -z.y); };
        sz[q][0][c] = a;
        sz[q][1][c] = upper ? ipos(a) : (MODE == 0 ? ineg(b) : ineg(a));
        if (HASB) {
          sz[q][2][c] = b;
          sz[q][3][c] = MODE == 0 ? (upper ? ipos(b) : ineg(a)) : ipos(b);
        }
      }
      __syncthreads();
#pragma unroll 1
      for (int q2 = 0; q2 < BQ; q2 += 2) {
#pragma unroll
        for (int q = q2; q < q2 + 2; ++q) {
          int4 u[2], w[2];
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            u[i] = sm0[q * BRP + rp + 32 * i];
            if (HASB) w[i] = sm1[q * BRP + rp + 32 * i];
          }
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            const int4 z0 = sz[q][0][2 * cp + j], z1 = sz[q][1][2 * cp + j];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              fx_mac(hh[i][j][0].v, hl[i][j][0].v, u[i].x, u[i].y, z0.x, z0.y);
              fx_mac(hh[i][j][1].v, hl[i][j][1].v, u[i].x, u[i].y, z0.z, z0.w);
              fx_mac(hh[i][j][0].v, hl[i][j][0].v, u[i].z, u[i].w, z1.x, z1.y);
              fx_mac(hh[i][j][1].v, hl[i][j][1].v, u[i].z, u[i].w, z1.z, z1.w);
            }
            if (HASB) {
              const int4 z2 = sz[q][NZ - 2][2 * cp + j], z3 = sz[q][NZ - 1][2 * cp + j];
#pragma unroll
              for (int i = 0; i < 2; ++i) {
                fx_mac(hh[i][j][0].v, hl[i][j][0].v, w[i].x, w[i].y, z2.x, z2.y);
                fx_mac(hh[i][j][1].v, hl[i][j][1].v, w[i].x, w[i].y, z2.z, z2.w);
                fx_mac(hh[i][j][0].v, hl[i][j][0].v, w[i].z, w[i].w, z3.x, z3.y);
                fx_mac(hh[i][j][1].v, hl[i][j][1].v, w[i].z, w[i].w, z3.z, z3.w);
              }
            }
          }
        }
        // after 16 products of two limbs (2^58 each at most; hl takes eight per q, hh four) a sum is below
        // 2^63 with the 2^38 left before
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
          for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int k = 0; k < 2; ++k) {
              fx_carry(hl[i][j][k]);
              if (q2 & 2) fx_carry(hh[i][j][k]);
            }
      }
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int c = c0 + 2 * cp + j;
      const int xe = c < K ? E[(int64_t)c * nT + J] : 64, ex = xe & FX_EMASK;
      // sums that nothing answers for are formed again in FP64, the warp's rows one by one (its columns are the
      // same); not for the residuals (ax.A null), which are a norm
      const bool check = !F32 && ax.A && c < K && ((xe >> FX_EBITS) < ((te >> FX_WEAK2) & FX_WMASK) + FX_MASS || ex == 2047);
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        double2 v = make_double2(fx_acc_double(hh[i][j][0], hl[i][j][0], eu, ex),
                                 fx_acc_double(hh[i][j][1], hl[i][j][1], eu, ex));
        if (check) {
          const bool weak = (int64_t)I * TS + rh + rp + 32 * i < ax.N && fx_weak(max(hi_abs(v.x), hi_abs(v.y)), eu, ex, (int)min((int64_t)TS, ax.N - (int64_t)J * TS));
          for (unsigned int todo = __ballot_sync(0xffffffffu, weak); todo; todo &= todo - 1) {
            const int l = __ffs(todo) - 1;
            const int64_t o = c * ax.ldx + (int64_t)J * TS;
            const double2 e = block_exact<MODE>(ax.A, ax.B, t, upper, I == J, rh + l + 32 * i, ax.xa + o,
                                                ax.xb ? ax.xb + o : nullptr, ax.sB);
            if (rp == l) v = e;
          }
        }
        y[i][j] = cadd(y[i][j], v);
      }
    }
  }
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const int c = c0 + 2 * cp + j;
    if (c >= K) continue;
#pragma unroll
    for (int i = 0; i < 2; ++i)
      part[((int64_t)blockIdx.z * K + c) * Npad + (int64_t)I * TS + rh + rp + 32 * i] = y[i][j];
  }
}

// Y = sum of the splits + the diagonal's part, in FP64; grid (Npad / 256, K)
template <int MODE>
__global__ void __launch_bounds__(256)
k_block_sum(const double2* __restrict__ part, int nsplit, const void* __restrict__ A, const void* __restrict__ B,
            int nT, int64_t Npad, const double2* __restrict__ xa, const double2* __restrict__ xb, int64_t ldx, double sB,
            int K, double2* __restrict__ Y, int64_t ldy) {
  constexpr bool HASB = MODE < 2;
  const int c = blockIdx.y;
  const int64_t r = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (r >= Npad) return;
  double2 y = part[(int64_t)c * Npad + r];
  for (int s = 1; s < nsplit; ++s) y = cadd(y, part[((int64_t)s * K + c) * Npad + r]);
  const int I = (int)(r / TS), d = (int)(r % TS);
  const int64_t o = ((int64_t)I * nT - (int64_t)I * (I - 1) / 2) * (TS * TS) + (int64_t)d * (TS + 1);
  const double2 va = xa[c * ldx + r];
  double2 a, b = make_double2(0.0, 0.0);
  block_element<MODE>(A, B, o, a, b);
  cfma(y, a, va);
  if (HASB) cfma(y, b, cscale(xb ? xb[c * ldx + r] : conjc(va), sB));
  Y[c * ldy + r] = y;
}

template <int MODE>
void run_block(const BlockFx& q, const double2* xa, const double2* xb, int64_t ldx, double sB, double2* y, int64_t ldy,
               int K, void* work, cudaStream_t s) {
  const int nT = q.nT;
  const int64_t Npad = (int64_t)nT * TS;
  int4* F0 = (int4*)work;
  int4* F1 = F0 + (size_t)K * Npad;
  double2* part = (double2*)(F1 + (MODE < 2 ? (size_t)K * Npad : 0));
  const int ns = block_fx_splits(nT, K);
  int* E = (int*)(part + (size_t)ns * K * Npad);
  count_launch(3);
  k_block_stage<(MODE < 2), MODE == 0><<<dim3(nT, K), TS, 0, s>>>(xa, xb, ldx, sB, Npad, nT, F0, F1, E);
  k_block_fx<MODE><<<dim3(2 * nT, (K + BC - 1) / BC, ns), 256, 0, s>>>(q.M0, q.M1, q.texp, nT, Npad, F0, F1, E, K, part,
                                                                 BlockExact{q.each ? q.A : nullptr, q.B, xa, xb, ldx, q.N, sB});
  k_block_sum<MODE><<<dim3((unsigned)((Npad + 255) / 256), K), 256, 0, s>>>(part, ns, q.A, q.B, nT, Npad, xa, xb, ldx,
                                                                            sB, K, y, ldy);
}

}  // namespace

// Splits of the block columns: about three waves of two CTAs per SM, so that the last one's idle
// share stays small, but whole tiles each.
int block_fx_splits(int nT, int K) {
  const int64_t units = 2ll * nT * ((K + BC - 1) / BC);
  const int64_t want = (6ll * num_sms() + units - 1) / units;
  const int per = (int)std::max<int64_t>(1, nT / std::max<int64_t>(1, std::min<int64_t>(want, nT)));
  return (nT + per - 1) / per;
}

size_t block_fx_bytes(int nT, int K, bool hasB) {
  const size_t col = (size_t)K * nT * TS * 16;
  return col * (hasB ? 2 : 1) + col * block_fx_splits(nT, K) + sizeof(int) * (size_t)K * nT;
}

void launch_block_fx(const BlockFx& q, bool hasB, bool tiles64, const double2* xa, const double2* xb, int64_t ldx,
                     double sB, double2* y, int64_t ldy, int K, void* work, cudaStream_t s) {
  if (hasB) {
    if (tiles64) run_block<1>(q, xa, xb, ldx, sB, y, ldy, K, work, s);
    else run_block<0>(q, xa, xb, ldx, sB, y, ldy, K, work, s);
  } else {
    if (tiles64) run_block<3>(q, xa, xb, ldx, sB, y, ldy, K, work, s);
    else run_block<2>(q, xa, xb, ldx, sB, y, ldy, K, work, s);
  }
}

void launch_block_scale64(const float2* A, const float2* B, int64_t N, int nT, int* texp, cudaStream_t s) {
  count_launch();
  if (B) k_block_scale64<true><<<dim3(nT, nT), 256, 0, s>>>(A, B, N, nT, texp);
  else k_block_scale64<false><<<dim3(nT, nT), 256, 0, s>>>(A, nullptr, N, nT, texp);
}

}  // namespace bse
