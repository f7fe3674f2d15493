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
// product by 2^-60 (the dropped term); the sums add nothing.  So a sum over a tile is off by some
// 2^-57.6 of 2^(E_u + E_x) (root mean square over its 256 multiply-adds; 2^-59 where one entry of x is far
// above the others), where an FP64 one is off by 2^-53 of its own sum of magnitudes |U||x|.  So a sum is
// good to a few tens of 2^-53 |U||x| if |U||x| is at least 2^-10 or 2^-11 of 2^(E_u + E_x).  That is sure when
//   * the chunk has FX_MASS strong entries more than any row (column) of the tile has weak ones: FX_MASS pairs
//     of 2^-2 FX_STRONG max|U| max|x| each.  Almost every sum is certified that way, before it is formed; or
//   * the sum itself is that large (2^-FX_SURE; less for the few terms of the matrix's last rows and columns).
// Any other sum -- x with a few entries far above the rest of its chunk, mostly -- is formed again in FP64 by
// a warp.  For these to be rare a tile runs in fixed point only when every entry of the matrix in
// it is within 2^FX_SPREAD of its largest (k_fx_pack; in the diagonal tiles the diagonal counts as one
// of the entries).  Sparse tiles, graded rows or columns, a peak, an infinity, a NaN, or exponents near the ends of the
// FP64 range keep a tile on the FP64 kernel.  Why 2^16: 16384 entries without structure spread by
// themselves (2^5 to 2^10 for a complex pair A, B; 2^8 to 2^14 for a complex A alone, one tile in 600
// above that and about one in 50000 above 2^16), and a tile left over costs a persistent step 20 us.
// (Without the count, sums that are small by cancellation were formed again too: N = 900, PH, 53 ms a solve
// and its gradients instead of 42.)
// x may have any exponent, subnormals included.  The diagonal of the matrix,
// which holds the transition energies far above everything else in its tiles, is left out of the
// tiles (zeros there) and added in FP64 by the block-row reduction.
//
// Bounds: 3 integer multiply-adds per real FMA instead of one FMA of a two-lane FP64 pipe; 32
// bytes per element pair either way, so the large products meet HBM instead of the FP64 pipe.
// Measured, folded product: N = 8000 503 -> 171 us (6.05 TB/s), N = 3000 75 -> 28.5 us, N = 900
// 38 -> 7.1 us (36 tiles in bands).  Sixteen warps per SM matter: the integer multiply-adds wait
// on one another, and eight warps ran N = 8000 in 229 us.  Against extended precision, N = 127 ... 2500: 0.3 to
// 1.2 units of 2^-53 normwise, the FP64 kernel 0.8 to 5.5.
#pragma once

#include "bse_phases.cuh"

namespace bse {

constexpr int FX_THREADS = 256;
constexpr int FX_WARPS = FX_THREADS / 32;
constexpr int FX_SPREAD = 16;        // largest over smallest entry of a fixed-point tile, log2
// What tells whether a sum's own magnitude |U||x| may be far below its scales (see above).  An entry of a
// tile or a chunk is strong when it is within 2^-FX_STRONG of the largest.  texp[t] holds the tile's scale
// exponent, then the largest number of entries in one of its rows or columns that are not strong: those
// where neither matrix has a strong element, and those where one of the two has not.
constexpr int FX_STRONG = 6, FX_EBITS = 11, FX_EMASK = (1 << FX_EBITS) - 1;
constexpr int FX_WEAK = FX_EBITS, FX_WEAK2 = FX_EBITS + 8, FX_WMASK = 0xff;
constexpr int FX_MASS = 16;          // strong pairs that make a sum sure
constexpr int FX_SURE = 11;          // a sum of 128 terms is sure above 2^-FX_SURE of its scales, too

constexpr long long FX_SPIN = 1ll << 24;      // polls of one wait for a row

// Shared memory of a CTA.  Each warp streams its own rows of the tiles through a ring of row
// buffers (a row of A and of B, 4 KiB, or of A alone, 2 KiB) with bulk asynchronous copies that
// complete on the warp's own barriers, several rows ahead and across the units'
// boundaries: 128 KiB in flight per SM and no block barrier in the row loop.
template <int RING>                    // bytes of a warp's ring
struct FxShared {
  unsigned char ring[FX_WARPS][RING];
  unsigned long long bar[FX_WARPS][8];
  int4 x[2][TS];                       // limbs of the column chunk J and the row chunk I
  int rows[TS][6];                     // three words of (re, im) per row of the unit
  int cols[FX_WARPS][6][TS];           // ... per column, one partial sum per warp
  unsigned int mx[2][TS / 32];
  int4 strong[2];                      // strong entries of the two chunks, by warp
};

__device__ __forceinline__ uint32_t fx_s32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// once per launch, before the first unit (all threads; the caller synchronises the block)
template <int RING>
__device__ __forceinline__ void fx_init(FxShared<RING>& sh) {
  if (threadIdx.x < FX_WARPS * 8)
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(fx_s32(&sh.bar[0][0] + threadIdx.x)) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ bool fx_wait(uint32_t bar, uint32_t parity) {
  for (long long i = 0; i < FX_SPIN; ++i) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  return false;
}

__device__ __forceinline__ void fx_copy(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "l"(src),
      "r"(bytes), "r"(bar)
      : "memory");
}

__device__ __forceinline__ unsigned int hi_abs(double v) { return (unsigned int)__double2hiint(v) & 0x7fffffffu; }

// round(v 2^59 / 2^(e - 1022)): v's magnitude is below 2^(e - 1022), e a biased exponent >= 1
__device__ __forceinline__ long long fx_fixed(double v, int e) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  const int ev = (int)(b >> 52) & 0x7ff;
  const int d = e - max(ev, 1);
  unsigned long long m = ((b & 0xfffffffffffffull) | (ev ? 0x10000000000000ull : 0ull)) << 6;
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

// (h 2^52 + l) 2^(eu + ex - 2044 - 72) as a double, |h| < 2^33 and 0 <= l < 2^52; eu, ex: biased
// exponents of the scales, ex = 2047 (an infinity or a NaN in the chunk) gives a NaN
__device__ __forceinline__ double fx_pack_double(long long h, unsigned long long l, int eu, int ex) {
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
  const int e = q + 63 + (eu + ex - 2044 - 72) + 1023;
  const int sub = max(0, min(1 - e, 52));                        // bits a subnormal result loses
  const unsigned long long r = (m >> (11 + sub)) + ((m >> (10 + sub)) & 1);      // 53 bits or fewer, rounded
  unsigned long long b = ((unsigned long long)(max(e, 1) - 1) << 52) + r;
  if (m == 0 || e < -52) b = 0;
  if (e > 2046) b = 0x7ff0000000000000ull;
  if (ex == 2047) b = 0x7ff8000000000000ull;
  return __longlong_as_double((long long)(b | (neg ? 0x8000000000000000ull : 0ull)));
}
// ... of words or sums of words: w0 2^52 + w1 2^26 + w2 (w1, w2 unsigned)
__device__ __forceinline__ double fx_double(int w0, unsigned int w1, unsigned int w2, int eu, int ex) {
  const unsigned long long l = ((unsigned long long)w1 << 26) + w2;
  return fx_pack_double((long long)w0 + (long long)(l >> 52), l & 0xfffffffffffffull, eu, ex);
}

// A warp's place in its stream of rows; it outlives one walk over the units (the barriers' phases
// go on), so a kernel keeps one per warp for its whole life.
struct FxPipe {
  unsigned int issued = 0, used = 0;     // rows copied, rows consumed
  bool ok = true;                        // no wait has expired
};

// A sum of n terms, its larger component's high word h, under the scales eu and ex (1: a tile or a chunk of
// zeros) that has to be formed again in FP64; an infinity or a NaN in the chunk (ex = 2047) asks for it too.
// (Its error goes with the square root of the terms.)
__device__ __forceinline__ bool fx_weak(unsigned int h, int eu, int ex, int n) {
  const int sure = FX_SURE + ((__clz(n) - 24) >> 1);
  return eu > 1 && ex > 1 && ((int)(h >> 20) < eu + ex - 1021 - sure || ex == 2047);
}

// One sum of a unit in FP64, by a warp (in every lane): row idx of the tile times x_J, or its rows
// [r0, r0 + n) of column idx times x_I; the matrix diagonal left out.  U, V: the tile's elements.
template <bool HASB, bool COH>
__device__ __forceinline__ double2 fx_exact(const double2* U, const double2* V, const double2* x, int idx, int r0, int n,
                                         bool col, bool diag) {
  const int lane = threadIdx.x & 31;
  double re = 0.0, im = 0.0;
  for (int k = r0 + lane; k < r0 + n; k += 32) {
    if (diag && k == idx) continue;
    const int e = col ? k * TS + idx : idx * TS + k;
    const double2 u = U[e], v = HASB ? V[e] : u, z = ldv<COH>(x + k);
    if (col) {
      re = fma(u.x, z.x, fma(u.y, z.y, re));
      im = fma(v.x, z.y, fma(-v.y, z.x, im));
    } else {
      re = fma(u.x, z.x, fma(-v.y, z.y, re));
      im = fma(u.y, z.x, fma(v.x, z.y, im));
    }
  }
  return make_double2(warp_sum_d(re), warp_sum_d(im));
}

// The row sums (or the column sums) of a unit that nothing answers for, again in FP64: those of the mask
// `todo` (a warp's lanes; sum threadIdx.x / 2 goes to the thread's `out`).  Out of line: it is rare.
template <bool HASB, bool COH>
__device__ __noinline__ void fx_settle(const Prob& p, int I, int J, int t, int mode, const void* io_x, double io_sB,
                                       double* out, unsigned int todo, int row0, int nrow, bool col) {
  const int tid = threadIdx.x, lane = tid & 31;
  const double2* x;
  double2* y;
  double sB;
  GenericIO io{};
  io.xa = io_x;
  io.sB = io_sB;
  prod_operands<double2, double>(p, mode, io, x, y, sB);
  const double2* U = (const double2*)(HASB && !(sB > 0.0) ? p.B : p.A) + (int64_t)t * (TS * TS);
  const double2* V = HASB ? (const double2*)(sB > 0.0 ? p.B : p.A) + (int64_t)t * (TS * TS) : nullptr;
  x += (int64_t)(col ? I : J) * TS;
  while (todo) {
    const int l = __ffs(todo) - 1, i = (tid - lane + l) >> 1;
    todo &= ~(3u << l);
    const double2 s = col ? fx_exact<HASB, COH>(U, V, x, i, row0, nrow, true, I == J)
                          : fx_exact<HASB, COH>(U, V, x, row0 + i, 0, TS, false, I == J);
    if ((lane >> 1) == (l >> 1)) *out = tid & 1 ? s.y : s.x;
  }
}

// Units of the fixed-point product: a tile, or a band of TS / nq of its rows.  A band's row sums
// are whole rows of slot (I, J); its column sums go to plane q of the slots, which the reduction
// adds.  Bands exist so that a problem of few tiles still occupies every SM.
// The walk of CTA bid of nblk over njobs * nq units.  A wait that expires raises *err; the warp
// then goes on without waiting (its reads stay inside the ring) and issues no further copy.
template <bool HASB, bool COH, int RING>
__device__ __forceinline__ void fx_tiles_body(const Prob* __restrict__ probs, const TileJob* __restrict__ jobs,
                                              int njobs, int nq, int mode, const GenericIO& io, int strided, int bid,
                                              int nblk, FxShared<RING>& sh, FxPipe& pipe, int* err) {
  constexpr unsigned int ROWB = TS * sizeof(int4);                     // bytes of one matrix's row
  constexpr unsigned int DEPTH = RING / (HASB ? 2 * ROWB : ROWB);   // rows in the ring
  const int lq = 31 - __clz(nq), nunit = njobs << lq;                  // nq is a power of two
  const int per = strided ? 1 : (nunit + nblk - 1) / nblk;
  const int u0 = strided ? bid : bid * per;
  const int u1 = strided ? nunit : min(nunit, u0 + per);
  const int du = strided ? nblk : 1;
  // Unit of position u.  The plus halves of a chain take a CTA's units in the opposite order: what it
  // read last is then what it wants first, while it may still be in the L2 (60 Haydock steps at
  // N = 8000: 23.4 ms against 23.8; nothing in the persistent kernel, whose problems nearly fit).
  const bool turned = !COH && (mode == PM_STEP_MPLUS || (mode == PM_GENERIC && io.sB > 0.0));
  const int usum = 2 * u0 + (u1 > u0 ? (u1 - 1 - u0) / du * du : 0);
  auto unit = [&](int u) { return turned ? usum - u : u; };
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nrow = TS >> lq, npr = nrow / FX_WARPS;   // rows of a unit and of a warp: row0 + warp + 8 a
  const uint32_t ring = fx_s32(sh.ring[warp]), bars = fx_s32(sh.bar[warp]);
  const double2* x;
  double2* y;
  double sB = 0.0;
  // the next unit from u on whose problem takes part, and its operand
  auto next_unit = [&](int u, TileJob& jb) {
    for (; u < u1; u += du) {
      jb = jobs[unit(u) >> lq];
      if (prod_operands<double2, double>(probs[jb.prob], mode, io, x, y, sB)) break;
    }
    return u;
  };
  auto x_value = [&](const TileJob& jb) {
    return ldv<COH>(x + (int64_t)(tid < TS ? jb.J : jb.I) * TS + (tid & (TS - 1)));
  };
  TileJob jb{}, jn{}, jp{};
  int un = next_unit(u0, jn);
  double2 xn = make_double2(0.0, 0.0);
  if (un < u1) xn = x_value(jn);
  // producer: `left` rows of unit pu to copy, the next ones at srcA, srcB
  int pu = un, left = 0;
  const int4 *srcA = nullptr, *srcB = nullptr;
  jp = jn;
  auto source = [&]() {
    if (pu >= u1) return;
    const Prob& p = probs[jp.prob];
    const int64_t off = (int64_t)jp.t * (TS * TS) + ((unit(pu) & (nq - 1)) * nrow + warp) * TS;
    const bool pos = sB > 0.0;           // U, V = P, Q for the plus half, Q, P for the minus half
    srcA = (HASB && !pos ? p.Bfx : p.Afx) + off;
    if (HASB) srcB = (pos ? p.Bfx : p.Afx) + off;
    left = pipe.ok ? npr : 0;
  };
  source();
  auto produce = [&]() {
    if (left == 0) return;
    if (lane == 0) {
      const unsigned int s = pipe.issued % DEPTH;
      const uint32_t dst = ring + s * (RING / DEPTH), bar = bars + 8 * s;
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar),
                   "r"(HASB ? 2 * ROWB : ROWB)
                   : "memory");
      fx_copy(dst, srcA, ROWB, bar);
      if (HASB) fx_copy(dst + ROWB, srcB, ROWB, bar);
    }
    srcA += FX_WARPS * TS;
    if (HASB) srcB += FX_WARPS * TS;
    ++pipe.issued;
    if (--left == 0) {
      const double2* xs = x;             // the consumer's operand stays
      pu = next_unit(pu + du, jp);
      source();
      x = xs;
    }
  };
  for (unsigned int k = 0; k < DEPTH; ++k) produce();
  while (un < u1) {
    const int u = un;
    jb = jn;
    const Prob& p = probs[jb.prob];
    const bool diag = jb.I == jb.J;
    const int q = unit(u) & (nq - 1), row0 = q * nrow;
    const double2 xv = xn;
    un = next_unit(u + du, jn);
    if (un < u1) xn = x_value(jn);       // arrives under this unit's arithmetic
    __syncthreads();                     // the shared sums of the previous unit have been read
    {
      const unsigned int m = __reduce_max_sync(0xffffffffu, max(hi_abs(xv.x), hi_abs(xv.y)));
      if (lane == 0) sh.mx[warp >> 2][warp & 3] = m;
    }
    __syncthreads();
    auto chunk_exp = [&](int k) {
      const unsigned int m = max(max(sh.mx[k][0], sh.mx[k][1]), max(sh.mx[k][2], sh.mx[k][3]));
      return max(1, (int)(m >> 20));
    };
    const int ec = chunk_exp(0), er = chunk_exp(1);
    {
      const unsigned int m = max(max(sh.mx[warp >> 2][0], sh.mx[warp >> 2][1]), max(sh.mx[warp >> 2][2], sh.mx[warp >> 2][3]));
      const unsigned int b = __ballot_sync(0xffffffffu, max(hi_abs(xv.x), hi_abs(xv.y)) + (FX_STRONG << 20) >= m);
      if (lane == 0) reinterpret_cast<int*>(sh.strong)[warp] = __popc(b);
    }
    sh.x[tid >> 7][tid & (TS - 1)] = fx_entry(xv, tid < TS ? ec : er);
    __syncthreads();
    int4 xc[4];
#pragma unroll
    for (int b = 0; b < 4; ++b) xc[b] = sh.x[0][lane + 32 * b];
    for (int a0 = 0; a0 < npr; a0 += 8) {
      const int a1 = min(npr, a0 + 8);   // a flush every eight rows: 16 terms per column sum
      long long chh[4][2], chl[4][2];
#pragma unroll
      for (int b = 0; b < 4; ++b) chh[b][0] = chh[b][1] = chl[b][0] = chl[b][1] = 0;
#pragma unroll 1
      for (int a = a0; a < a1; ++a) {
        const unsigned int s = pipe.used % DEPTH;
        if (pipe.ok && __any_sync(0xffffffffu, !fx_wait(bars + 8 * s, (pipe.used / DEPTH) & 1))) {
          if (lane == 0) atomicExch(err, 1);
          pipe.ok = false;
          left = 0;
        }
        const int4* rp = reinterpret_cast<const int4*>(sh.ring[warp] + s * (RING / DEPTH)) + lane;
        int4 uu[4], vv[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          uu[b] = rp[32 * b];
          vv[b] = HASB ? rp[TS + 32 * b] : uu[b];
        }
        ++pipe.used;
        __syncwarp();                    // the row is in registers: its buffer may be refilled
        produce();
        const int r = row0 + warp + FX_WARPS * a;
        const int4 y4 = sh.x[1][r];
        const int ynh = -y4.x, ynl = -y4.y;
        // row (M_s x_J)_r: re = U_re x_re - V_im x_im, im = U_im x_re + V_re x_im
        long long s1h = 0, s1l = 0, s2h = 0, s2l = 0, s3h = 0, s3l = 0;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          fx_mac(s1h, s1l, uu[b].x, uu[b].y, xc[b].x, xc[b].y);
          fx_mac(s2h, s2l, vv[b].z, vv[b].w, xc[b].z, xc[b].w);
          fx_mac(s3h, s3l, uu[b].z, uu[b].w, xc[b].x, xc[b].y);
          fx_mac(s3h, s3l, vv[b].x, vv[b].y, xc[b].z, xc[b].w);
        }
        if (!diag) {
          // column (M_s^T x_I)_c: re = U_re y_re + U_im y_im, im = V_re y_im - V_im y_re
#pragma unroll
          for (int b = 0; b < 4; ++b) {
            fx_mac(chh[b][0], chl[b][0], uu[b].x, uu[b].y, y4.x, y4.y);
            fx_mac(chh[b][0], chl[b][0], uu[b].z, uu[b].w, y4.z, y4.w);
            fx_mac(chh[b][1], chl[b][1], vv[b].x, vv[b].y, y4.z, y4.w);
            fx_mac(chh[b][1], chl[b][1], vv[b].z, vv[b].w, ynh, ynl);
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
            for (int k = 0; k < 3; ++k) {
              int& d = sh.cols[warp][3 * c + k][lane + 32 * b];
              d = a0 == 0 ? w[k] : d + w[k];
            }
          }
      }
    }
    __syncthreads();
    const int te = p.texp[jb.t], eu = te & FX_EMASK;
    double* part = (double*)p.part;
    const int i = tid >> 1, c = tid & 1;
    auto settle = [&](double v, double* out, bool live, int k, int ex) {
      const int4 ns = sh.strong[k];
      if (ns.x + ns.y + ns.z + ns.w >= ((te >> FX_WEAK) & FX_WMASK) + FX_MASS && ex != 2047) return;
      unsigned int h = hi_abs(v);
      h = max(h, __shfl_xor_sync(0xffffffffu, h, 1));
      const int n = (int)min((int64_t)TS, p.N - (int64_t)(k ? jb.I : jb.J) * TS);
      const unsigned int todo = __ballot_sync(0xffffffffu, live && fx_weak(h, eu, ex, n));
      if (todo) fx_settle<HASB, COH>(p, jb.I, jb.J, jb.t, mode, io.xa, io.sB, out, todo, row0, nrow, k != 0);
    };
    double v = 0.0;
    double* out = part + (((int64_t)jb.I * p.nT + jb.J) * TS + row0 + i) * 2 + c;
    if (i < nrow) {
      const int* w = sh.rows[i] + 3 * c;
      v = fx_double(w[0], w[1], w[2], eu, ec);
      *out = v;
    }
    settle(v, out, i < nrow && (int64_t)jb.I * TS + row0 + i < p.N, 0, ec);
    if (!diag) {
      int w[3] = {0, 0, 0};
#pragma unroll
      for (int wp = 0; wp < FX_WARPS; ++wp)
#pragma unroll
        for (int k = 0; k < 3; ++k) w[k] += sh.cols[wp][3 * c + k][i];
      out = part + (((int64_t)q * p.nT * p.nT + (int64_t)jb.J * p.nT + jb.I) * TS + i) * 2 + c;
      v = fx_double(w[0], w[1], w[2], eu, er);
      *out = v;
      settle(v, out, (int64_t)jb.J * TS + i < p.N, 1, er);
    }
  }
  if (!pipe.ok && lane == 0)             // leave no copy in flight
    for (unsigned int k = pipe.issued > DEPTH ? pipe.issued - DEPTH : 0; k < pipe.issued; ++k)
      fx_wait(bars + 8 * (k % DEPTH), (k / DEPTH) & 1);
}

}  // namespace bse
