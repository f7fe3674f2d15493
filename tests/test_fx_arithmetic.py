"""The fixed-point product's arithmetic (fx_phases.cuh) and its choice of tiles (k_fx_pack), run on the
host: one 128 x 128 tile times a vector, element by element against |U||x|, and which tiles are left to
the FP64 kernel.

Bound.  u and x are off by at most 2^-60 of 2^E (twice the largest component at most), the dropped
product by 2^-60: 3 2^-58 max|u| max|x| per real multiply-add.  A row has two per entry; their signs are
as good as random, so a sum over 128 entries is within 6 sigma of sqrt(2 128) times a third of that:
96 2^-58 max|u| max|x| < 2^-51 max|u| max|x|, and 2^-53 of the result.  In a tile that qualifies max|u| is
at most 2^14 times any entry, so this is at most 2^-37 |U||x|, whatever x; for x without
outliers, |U||x| is some 128 / 8 max|u| max|x|, and the bound 2^-53 |U||x| holds."""
import numpy as np
import pytest

from tests.simt import cut, run

SRC = r"""
#include "simt.h"
#define __restrict__
namespace bse {
constexpr int TS = 128;
%s
%s
%s
}
using namespace bse;
int main(int, char** argv) {
  const int N = atoi(argv[3]), I = atoi(argv[4]), J = atoi(argv[5]), nT = 2;
  const int t = I * nT - I * (I - 1) / 2 + (J - I);
  std::vector<double2> A(3 * TS * TS), x(TS);
  FILE* f = fopen(argv[1], "rb");
  fread(A.data() + t * TS * TS, 16, TS * TS, f);
  f = fopen(argv[2], "rb");
  fread(x.data(), 16, TS, f);
  std::vector<int4> Af(3 * TS * TS);
  int texp[3] = {0, 0, 0};
  blockIdx.x = J;
  blockIdx.y = I;
  if (!simt::run_block(256, false, [&] { k_fx_pack<false>(A.data(), nullptr, N, nT, Af.data(), nullptr, texp); })) return 1;
  printf("%%d\n", texp[t]);
  const int eu = texp[t] < 0 ? 1 : texp[t];
  unsigned m = 0;
  for (auto v : x) m = max(m, max(hi_abs(v.x), hi_abs(v.y)));
  const int ex = max(1, (int)(m >> 20));
  for (int r = 0; r < TS; ++r) {
    int w[6] = {0, 0, 0, 0, 0, 0};
    for (int lane = 0; lane < 32; ++lane) {
      long long s1h = 0, s1l = 0, s2h = 0, s2l = 0, s3h = 0, s3l = 0;
      for (int b = 0; b < 4; ++b) {
        const int4 u = Af[t * TS * TS + r * TS + lane + 32 * b], c = fx_entry(x[lane + 32 * b], ex);
        fx_mac(s1h, s1l, u.x, u.y, c.x, c.y);
        fx_mac(s2h, s2l, u.z, u.w, c.z, c.w);
        fx_mac(s3h, s3l, u.z, u.w, c.x, c.y);
        fx_mac(s3h, s3l, u.x, u.y, c.z, c.w);
      }
      int k[6];
      fx_words(s1h - s2h, s1l - s2l, k[0], k[1], k[2]);
      fx_words(s3h, s3l, k[3], k[4], k[5]);
      for (int i = 0; i < 6; ++i) w[i] += k[i];
    }
    printf("%%.17g %%.17g\n", fx_double(w[0], w[1], w[2], eu, ex), fx_double(w[3], w[4], w[5], eu, ex));
  }
}
"""


def _product(tmp_path, u, x, n=256, tile=(0, 1)):
    """(tile exponent or -1, U x by the kernel's arithmetic); tile (I, J) of a matrix of order n"""
    a = cut("fx_phases.cuh", "__device__ __forceinline__ unsigned int hi_abs", "// A warp's place")
    k = cut("k_product_fx.cu", "// v / 2", "}  // namespace")
    c = cut("fx_phases.cuh", "constexpr int FX_THREADS", "constexpr long long FX_SPIN")
    fu, fx = tmp_path / "u", tmp_path / "x"
    fu.write_bytes(np.ascontiguousarray(u, np.complex128).tobytes())
    fx.write_bytes(np.ascontiguousarray(x, np.complex128).tobytes())
    out = run(tmp_path, SRC % (c, a, k), fu, fx, n, *tile)
    return int(out[0][0]), np.array([complex(*v) for v in out[1:]])


def _gauss(rng, *shape):
    return rng.standard_normal(shape) + 1j * rng.standard_normal(shape)


def _err(u, x, y):
    ref = (u.astype(np.clongdouble) * x.astype(np.clongdouble)[None, :]).sum(1)
    return np.abs(y - ref).astype(float), (np.abs(u) * np.abs(x)[None, :]).sum(1)


@pytest.mark.parametrize("scale", [1.0, 2.0 ** -900, 2.0 ** -1015, 2.0 ** 900])
def test_vector_of_any_exponent(tmp_path, scale):
    """x of ordinary entries near the ends of the FP64 range: the result to FP64 rounding (2^-1074 at
    its own lower end)."""
    rng = np.random.default_rng(3)
    u, x = _gauss(rng, 128, 128), _gauss(rng, 128)
    big = 1.0 if scale < 1 else 2.0 ** 60       # so that neither factor alone decides
    ex, y = _product(tmp_path, u * big, x * scale)
    err, mag = _err(u, x, y / big / scale if scale >= 2.0 ** -900 else y * 2.0 ** 1015)
    assert ex > 0
    assert np.all(err <= 2.0 ** -53 * mag + (2.0 ** -50 if scale == 2.0 ** -1015 else 0.0))
