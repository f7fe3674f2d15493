"""Rounding of the complex64 Gram-Schmidt passes (bse_phases.cuh) at large N and many columns, the code
run on the host.  All terms of a sum are equal, so the roundings of a chain add up instead of averaging
out: a chain of n FP32 terms may be off by n 2^-24 of the sum of magnitudes.  A lane's chain in the dots
has 16 terms per component, then FP64 goes on; a thread's chain in the update has nset / 64 terms, then
eight sums of its own and eight of the warps."""
import numpy as np
import pytest

from tests.simt import cut, run

SRC = r"""
#include "simt.h"
#define __restrict__
template <typename T> T __ldcg(const T* p) { return *p; }
namespace bse {
constexpr int TS = 128, DOT_CHUNKS = 8, MAXM = 1024;
inline double2 mk(double x, double y) { return make_double2(x, y); }
template <typename T> T czero() { return T{0, 0}; }
template <typename T> T ccvt(double2 v) { T r; r.x = v.x; r.y = v.y; return r; }
template <typename T> T cadd(T a, T b) { a.x += b.x; a.y += b.y; return a; }
template <typename T> void cfma(T& y, T a, T x) {
  y.x = fma(a.x, x.x, y.x); y.x = fma(-a.y, x.y, y.x);
  y.y = fma(a.x, x.y, y.y); y.y = fma(a.y, x.x, y.y);
}
template <typename T> void cfmac(T& y, T a, T x) {
  y.x = fma(a.x, x.x, y.x); y.x = fma(a.y, x.y, y.x);
  y.y = fma(a.x, x.y, y.y); y.y = fma(-a.y, x.x, y.y);
}
enum { ST_OK = 0 };
struct KState { int j, m, done, status, breakdown; };
struct Prob {
  int nT; int64_t Npad; int slab, ncol; const void *V, *P, *Z, *W; void* w; double *cpart, *coef, *npart; KState* st;
};
%s
%s
}
using namespace bse;
int main(int, char** argv) {
  const int ph = atoi(argv[1]), nT = atoi(argv[2]), nj = atoi(argv[3]);
  const float c = atof(argv[4]);
  Prob p{};
  KState st{nj - 1, nj + 1, 0, 0, 0};
  p.nT = nT;
  p.Npad = nT * TS;
  p.slab = 32;
  p.ncol = 2 * nj + 1;
  p.st = &st;
  std::vector<float2> v(p.Npad * nj, make_float2(c, 0.f)), w(p.Npad, make_float2(c, 0.f));
  std::vector<double> cp(2 * DOT_CHUNKS * p.ncol, 0.0), coef(4 * p.ncol), np(p.Npad);
  p.V = p.P = v.data();
  p.w = w.data();
  p.cpart = cp.data();
  p.coef = coef.data();
  p.npart = np.data();
  const CgsSet cs = cgs_set(p, &st, ph, 0);
  double s = 0.0;
  for (int k = 0; k < dot_chunks(nT); ++k) {
    if (!simt::run_block(32, false, [&] { cgs_dot_task<float2, false>(p, &st, cs, ph, 0, 0, 0, 0, k); })) return 1;
    s += ph ? cp[k * p.ncol] : cp[2 * k * p.ncol];
  }
  printf("%%.17g %%.17g\n", s, (double)c * c * p.Npad);
  // one row slab of the update: every coefficient one
  for (auto& t : cp) t = 0.0;
  for (int q = 0; q < p.ncol; ++q) cp[ph ? q : 2 * q] = 1.0;
  std::vector<float2> cf(2 * MAXM + 2);
  static float2 red[8][32];
  if (!simt::run_block(256, false, [&] { cgs_update_unit<float2, false>(p, &st, ph, 0, 0, 0, 0, cf.data(), red); })) return 1;
  printf("%%.17g %%.17g\n", (double)w[0].x, c - (double)nj * c);
}
"""


@pytest.mark.parametrize("ph", [0, 1])
def test_chains_do_not_grow_with_n(tmp_path, ph):
    a = cut("bse_phases.cuh", "template <bool COH, typename T>", "// Resolve the input / output")
    b = cut("bse_phases.cuh", "// ---------------------------------------------------------------- CGS2 dots",
            "// ---------------------------------------------------------------- norms")
    src = SRC % (a, "__device__ __forceinline__ double warp_sum_d(double v) {\n"
                    "  for (int m = 16; m >= 1; m >>= 1) v += __shfl_xor_sync(0xffffffffu, v, m);\n  return v;\n}\n" + b)
    worst = np.zeros(2)
    for c in np.float32([0.3, 0.57, 0.71, 1.01, 1.37, 1.79]):
        nj = 700
        (s, sref), (w, wref) = run(tmp_path, src, ph, 391, nj, repr(float(c)))       # N = 50000
        worst = np.maximum(worst, [abs(s - sref) / sref, abs(w - wref) / abs(wref)])
    assert worst[0] <= 17 * 2.0 ** -24                      # 16 terms, and one for the constant's square
    assert worst[1] <= (-(-(1 + ph) * nj // 64) + 8 + 8 + 2) * 2.0 ** -24
