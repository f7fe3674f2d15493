// FP64-accurate structured product on the integer pipe (complex128 handles).
//
// GB300 runs two FP64 FMAs per SM and clock (a warp-wide FP64 instruction holds its scheduler's
// FP64 pipe for 64 clocks, whatever its active lanes), but about 27 32 x 32 + 64-bit integer
// multiply-adds (measured, IMAD.WIDE in a loop).  So the streaming product of complex128 tiles
// is done in fixed point: an entry u of a tile is stored as round(u 2^59 / 2^E), 2^E the power
// of two above the tile's largest component, split into two signed 30-bit limbs (uh, ul); the
// vector is split the same way per 128-entry chunk.  A real multiply-add is three integer
// multiply-adds
//     hh += uh xh          (unit 2^60)
//     hl += uh xl + ul xh  (unit 2^30; the dropped ul xl is 2^-60 of the largest product)
// into 64-bit sums that cannot overflow over the 16 terms a thread adds between two flushes, so
// the sums are exact and do not depend on the order.  The sums of a row or column travel as three
// 26-bit words (unit 2^-72 of 2^(E_u + E_x)) through integer reductions, and become one FP64
// value per tile, row and column, built with integer instructions.
//
// Accuracy.  Each entry of U and of x is off by at most 2^-60 of its tile's or chunk's 2^E, each
// product by 2^-60 (the dropped term); the sums add nothing.  An FP64 dot product rounds every
// partial sum at 2^-53, so the fixed-point one is the more accurate of the two as long as the
// tile's largest entry is not far above its typical one.  Where it is -- peak^2 above
// FX_PEAK^2 mean square, an infinity, a NaN, or exponents near the ends of the FP64 range -- the
// tile stays on the FP64 kernel (k_fx_pack writes the decision).  The diagonal of the matrix,
// which holds the transition energies far above everything else in its tiles, is left out of the
// tiles (zeros there) and added in FP64 by the block-row reduction.
//
// Bounds: 3 integer multiply-adds per real FMA instead of one FMA of a two-lane FP64 pipe; 32
// bytes per element pair either way, so the large products meet HBM instead of the FP64 pipe.
// Measured, folded product: N = 8000 503 -> 228 us (HBM floor 154), N = 3000 75 -> 36 us,
// N = 900 38 -> 6.7 us (36 tiles in bands).  Against extended precision, N = 127 ... 2500: 0.3 to
// 1.2 units of 2^-53 normwise, the FP64 kernel 0.8 to 5.5.
#pragma once

#include "bse_phases.cuh"

namespace bse {

constexpr int FX_THREADS = 256;
constexpr int FX_WARPS = FX_THREADS / 32;
constexpr float FX_PEAK = 64.f;

// shared memory of one unit
struct FxShared {
  int4 x[2][TS];                       // limbs of the column chunk J and the row chunk I
  int rows[TS][6];                     // three words of (re, im) per row of the unit
  int cols[FX_WARPS][6][TS];           // ... per column, one partial sum per warp
  unsigned int mx[2][TS / 32];
};

__device__ __forceinline__ unsigned int hi_abs(double v) { return (unsigned int)__double2hiint(v) & 0x7fffffffu; }

// round(v 2^59 / 2^(e - 1022)): v's magnitude is below 2^(e - 1022), e a biased exponent >= 64
__device__ __forceinline__ long long fx_fixed(double v, int e) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  const int ev = (int)(b >> 52) & 0x7ff;
  const int d = e - ev;
  unsigned long long m = ((b & 0xfffffffffffffull) | 0x10000000000000ull) << 6;
  m = d > 0 ? ((m >> (min(d, 63) - 1)) + 1) >> 1 : m;
  const long long f = d < 62 ? (long long)m : 0ll;
  return (long long)b < 0 ? -f : f;
}
// signed 30-bit limbs: f = hi 2^30 + lo
__device__ __forceinline__ void fx_limbs(long long f, int& hi, int& lo) {
  lo = (int)((unsigned int)f << 2) >> 2;
  hi = (int)((f - lo) >> 30);
}
__device__ __forceinline__ int4 fx_entry(double2 v, int e) {
  int4 r;
  fx_limbs(fx_fixed(v.x, e), r.x, r.y);
  fx_limbs(fx_fixed(v.y, e), r.z, r.w);
  return r;
}

__device__ __forceinline__ void fx_mac(long long& hh, long long& hl, int uh, int ul, int xh, int xl) {
  hh += (long long)uh * xh;
  hl += (long long)uh * xl;
  hl += (long long)ul * xh;
}

// (hh, hl) as three words: w0 2^52 + w1 2^26 + w2 in units of 2^-14 of hh's (w1, w2 in [0, 2^26))
__device__ __forceinline__ void fx_words(long long hh, long long hl, int& w0, int& w1, int& w2) {
  const long long v = hh + (hl >> 30);
  const unsigned int lo = (unsigned int)hl & 0x3fffffffu;
  w0 = (int)(v >> 38);
  w1 = (int)((unsigned int)(v >> 12) & 0x3ffffffu);
  w2 = (int)((((unsigned int)v & 0xfffu) << 14) | (lo >> 16));
}

// (w0 2^52 + w1 2^26 + w2) 2^(eu + ex - 2044 - 72) as a double (sums of words: w1, w2 unsigned);
// eu, ex: biased exponents of the scales, 2047 (an infinity or a NaN in the chunk) gives a NaN
__device__ __forceinline__ double fx_double(int w0, unsigned int w1, unsigned int w2, int eu, int ex) {
  const unsigned long long l0 = ((unsigned long long)w1 << 26) + w2;
  long long h = (long long)w0 + (long long)(l0 >> 52);
  unsigned long long l = l0 & 0xfffffffffffffull;
  const bool neg = h < 0;
  if (neg) {
    h = -h - (l ? 1 : 0);
    l = l ? 0x10000000000000ull - l : 0ull;
  }
  // 64 leading bits m of h 2^52 + l = m 2^q (h < 2^33)
  unsigned long long m;
  int q;
  if (h) {
    const int n = 64 - __clzll(h);
    m = ((unsigned long long)h << (64 - n)) | ((l << 12) >> n);
    q = n - 12;
  } else {
    const int n = l ? __clzll(l) : 0;
    m = l << n;
    q = -n;
  }
  const unsigned long long r = (m >> 11) + ((m >> 10) & 1);      // 53 bits, rounded
  const int e = q + 63 + (eu + ex - 2044 - 72) + 1023;
  unsigned long long b = ((unsigned long long)(e - 1) << 52) + r;
  if (e < 1 || m == 0) b = 0;
  if (e > 2046) b = 0x7ff0000000000000ull;
  if (ex == 2047) b = 0x7ff8000000000000ull;
  return __longlong_as_double((long long)(b | (neg ? 0x8000000000000000ull : 0ull)));
}

// Units of the fixed-point product: a tile, or a band of TS / nq of its rows.  A band's row sums
// are whole rows of slot (I, J); its column sums go to plane q of the slots, which the reduction
// adds.  Bands exist so that a problem of few tiles still occupies every SM.
// One unit: job t, band q; `sh` is rewritten by the next unit.
template <bool HASB, bool COH>
__device__ __forceinline__ void fx_tile_unit(const Prob& p, const TileJob jb, const double2* x, bool pos, int q, int nq,
                                             FxShared& sh) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool diag = jb.I == jb.J;
  const int nrow = TS / nq, row0 = q * nrow;
  const int4* At = (const int4*)(HASB && !pos ? p.Bfx : p.Afx) + (int64_t)jb.t * (TS * TS);
  const int4* Bt = HASB ? (const int4*)(pos ? p.Bfx : p.Afx) + (int64_t)jb.t * (TS * TS) : nullptr;
  __syncthreads();                       // shared memory of the previous unit is free
  const double2 xv = ldp<COH>(x + (int64_t)(tid < TS ? jb.J : jb.I) * TS + (tid & (TS - 1)));
  {
    const unsigned int m = __reduce_max_sync(0xffffffffu, max(hi_abs(xv.x), hi_abs(xv.y)));
    if (lane == 0) sh.mx[warp >> 2][warp & 3] = m;
  }
  for (int e = tid; e < FX_WARPS * 6 * TS / 4; e += FX_THREADS)
    reinterpret_cast<int4*>(sh.cols)[e] = make_int4(0, 0, 0, 0);
  __syncthreads();
  auto chunk_exp = [&](int k) {
    const unsigned int m = max(max(sh.mx[k][0], sh.mx[k][1]), max(sh.mx[k][2], sh.mx[k][3]));
    return max(64, (int)(m >> 20));
  };
  const int ec = chunk_exp(0), er = chunk_exp(1);
  sh.x[tid >> 7][tid & (TS - 1)] = fx_entry(xv, tid < TS ? ec : er);
  __syncthreads();
  int4 xc[4];
#pragma unroll
  for (int b = 0; b < 4; ++b) xc[b] = sh.x[0][lane + 32 * b];
  const int4* ar = At + (int64_t)(row0 + warp) * TS + lane;
  const int4* br = HASB ? Bt + (int64_t)(row0 + warp) * TS + lane : nullptr;
  const int npr = nrow / FX_WARPS;       // rows of this warp: row0 + warp + 8 a
  int4 un[4], vn[4];
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    un[b] = __ldg(ar + 32 * b);
    if (HASB) vn[b] = __ldg(br + 32 * b);
  }
  for (int a0 = 0; a0 < npr; a0 += 8) {
    const int a1 = min(npr, a0 + 8);     // a flush every eight rows: 16 terms per column sum
    long long chh[4][2], chl[4][2];
#pragma unroll
    for (int b = 0; b < 4; ++b) chh[b][0] = chh[b][1] = chl[b][0] = chl[b][1] = 0;
#pragma unroll 1
    for (int a = a0; a < a1; ++a) {
      int4 u[4], v[4];
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        u[b] = un[b];
        v[b] = HASB ? vn[b] : un[b];
      }
      if (a + 1 < npr) {                 // the next row's loads run under this row's arithmetic
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          un[b] = __ldg(ar + (int64_t)(a + 1) * FX_WARPS * TS + 32 * b);
          if (HASB) vn[b] = __ldg(br + (int64_t)(a + 1) * FX_WARPS * TS + 32 * b);
        }
      }
      const int r = row0 + warp + FX_WARPS * a;
      const int4 y = sh.x[1][r];
      const int4 yn = make_int4(-y.x, -y.y, -y.z, -y.w);
      // row (M_s x_J)_r: re = U_re x_re - V_im x_im, im = U_im x_re + V_re x_im
      long long s1h = 0, s1l = 0, s2h = 0, s2l = 0, s3h = 0, s3l = 0;
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        fx_mac(s1h, s1l, u[b].x, u[b].y, xc[b].x, xc[b].y);
        fx_mac(s2h, s2l, v[b].z, v[b].w, xc[b].z, xc[b].w);
        fx_mac(s3h, s3l, u[b].z, u[b].w, xc[b].x, xc[b].y);
        fx_mac(s3h, s3l, v[b].x, v[b].y, xc[b].z, xc[b].w);
      }
      if (!diag) {
        // column (M_s^T x_I)_c: re = U_re y_re + U_im y_im, im = V_re y_im - V_im y_re
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          fx_mac(chh[b][0], chl[b][0], u[b].x, u[b].y, y.x, y.y);
          fx_mac(chh[b][0], chl[b][0], u[b].z, u[b].w, y.z, y.w);
          fx_mac(chh[b][1], chl[b][1], v[b].x, v[b].y, y.z, y.w);
          fx_mac(chh[b][1], chl[b][1], v[b].z, v[b].w, yn.x, yn.y);
        }
      }
      int w[6];
      fx_words(s1h - s2h, s1l - s2l, w[0], w[1], w[2]);
      fx_words(s3h, s3l, w[3], w[4], w[5]);
#pragma unroll
      for (int k = 0; k < 6; ++k) w[k] = __reduce_add_sync(0xffffffffu, w[k]);
      if (lane == 0) {
#pragma unroll
        for (int k = 0; k < 6; ++k) sh.rows[r - row0][k] = w[k];
      }
    }
    if (!diag) {
#pragma unroll
      for (int b = 0; b < 4; ++b)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          int w[3];
          fx_words(chh[b][c], chl[b][c], w[0], w[1], w[2]);
#pragma unroll
          for (int k = 0; k < 3; ++k) sh.cols[warp][3 * c + k][lane + 32 * b] += w[k];
        }
    }
  }
  __syncthreads();
  const int eu = p.texp[jb.t];
  double* part = (double*)p.part;
  const int i = tid >> 1, c = tid & 1;
  if (i < nrow) {
    const int* w = sh.rows[i] + 3 * c;
    part[(((int64_t)jb.I * p.nT + jb.J) * TS + row0 + i) * 2 + c] = fx_double(w[0], w[1], w[2], eu, ec);
  }
  if (!diag) {
    int w[3] = {0, 0, 0};
#pragma unroll
    for (int wp = 0; wp < FX_WARPS; ++wp)
#pragma unroll
      for (int k = 0; k < 3; ++k) w[k] += sh.cols[wp][3 * c + k][i];
    part[(((int64_t)q * p.nT * p.nT + (int64_t)jb.J * p.nT + jb.I) * TS + i) * 2 + c] =
        fx_double(w[0], w[1], w[2], eu, er);
  }
}

// the unit walk of CTA bid of nblk over njobs * nq units
template <bool HASB, bool COH>
__device__ __forceinline__ void fx_tiles_body(const Prob* __restrict__ probs, const TileJob* __restrict__ jobs,
                                              int njobs, int nq, int mode, const GenericIO& io, int strided, int bid,
                                              int nblk, FxShared& sh) {
  const int nunit = njobs * nq;
  const int per = strided ? 1 : (nunit + nblk - 1) / nblk;
  const int u0 = strided ? bid : bid * per;
  const int u1 = strided ? nunit : min(nunit, u0 + per);
  const int du = strided ? nblk : 1;
  for (int u = u0; u < u1; u += du) {
    const TileJob jb = jobs[u / nq];
    const Prob& p = probs[jb.prob];
    const double2* x;
    double2* y;
    double sB;
    if (!prod_operands<double2, double>(p, mode, io, x, y, sB)) continue;   // uniform per CTA
    fx_tile_unit<HASB, COH>(p, jb, x, sB > 0.0, u % nq, nq, sh);
  }
}

}  // namespace bse
