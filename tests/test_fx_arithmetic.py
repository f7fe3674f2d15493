"""The fixed-point product's arithmetic (fx_phases.cuh) and its choice of tiles (k_fx_pack), run on the
host: one 128 x 128 tile times a vector, element by element against |U||x|, and which tiles are left to
the FP64 kernel.

Bound.  u and x are off by at most 2^-60 of 2^E (twice the largest component at most), the dropped
product by 2^-60: 3 2^-58 max|u| max|x| per real multiply-add.  A row has two per entry; their signs are
as good as random, so a sum over 128 entries is within 6 sigma of sqrt(2 128) times a third of that:
96 2^-58 max|u| max|x| < 2^-51 max|u| max|x|, and 2^-53 of the result.  In a tile that qualifies max|u| is
at most 2^16 times any entry, so this is at most 2^-35 |U||x|, whatever x; for x without
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
  printf("%%d %%d %%d\n", texp[t] < 0 ? -1 : texp[t] & FX_EMASK, (texp[t] >> FX_WEAK) & FX_WMASK,
         (texp[t] >> FX_WEAK2) & FX_WMASK);
  const int eu = texp[t] < 0 ? 1 : texp[t] & FX_EMASK;
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
    k = cut("k_product_fx.cu", "template <bool HASB>\n__global__ void __launch_bounds__(256)", "}  // namespace")
    c = cut("fx_phases.cuh", "constexpr int FX_THREADS", "constexpr long long FX_SPIN")
    fu, fx = tmp_path / "u", tmp_path / "x"
    fu.write_bytes(np.ascontiguousarray(u, np.complex128).tobytes())
    fx.write_bytes(np.ascontiguousarray(x, np.complex128).tobytes())
    out = run(tmp_path, SRC % (c, a, k), fu, fx, n, *tile)
    _product.weak = out[0][1:]
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


@pytest.mark.parametrize("seed", range(4))
def test_outlier_in_the_vector(tmp_path, seed):
    """An entry of x 1e10 above the others, every row's own magnitude as the measure."""
    rng = np.random.default_rng(seed)
    u, x = _gauss(rng, 128, 128), _gauss(rng, 128)
    x[rng.integers(128)] *= 1e10
    ex, y = _product(tmp_path, u, x)
    err, mag = _err(u, x, y)
    assert ex > 0 and np.all(err <= 64 * 2.0 ** -53 * mag)


def test_unit_vector(tmp_path):
    """x = e_j gives the column of U to the rounding of its entries, 2^-60 of the scale."""
    rng = np.random.default_rng(5)
    u, x = _gauss(rng, 128, 128), np.zeros(128)
    x[17] = 1.0
    ex, y = _product(tmp_path, u, x)
    assert ex > 0 and np.all(np.abs(y - u[:, 17]) <= 2.0 ** -59 * np.maximum(np.abs(u.real), np.abs(u.imag)).max() + 2.0 ** -52 * np.abs(u[:, 17]))


def _tiles():
    rng = np.random.default_rng(7)
    g = _gauss(rng, 128, 128)
    half = np.arange(128) >= 64
    yield "dense", g, True
    yield "zero", 0 * g, True
    yield "two uncoupled blocks", np.where(half[:, None] == half[None, :], g, 0), False
    yield "graded rows", np.where(half[:, None], 1e-10 * g, g), False
    yield "graded columns", np.where(half[None, :], 1e-10 * g, g), False
    one = np.where(np.arange(128)[:, None] == 5, g, 1e-12 * g)
    yield "one large row", one, False
    hole = g.copy()
    hole[100, 3] = 0
    yield "one zero", hole, False
    peak = g.copy()
    peak[4, 99] *= 1e5
    yield "a peak", peak, False
    bad = g.copy()
    bad[9, 9] = np.inf
    yield "an infinity", bad, False
    yield "tiny", g * 2.0 ** -900, False


SRC32 = r"""
#include "simt.h"
#define __restrict__
namespace bse {
constexpr int TS = 128;
%s
%s
}
using namespace bse;
int main(int, char** argv) {
  std::vector<double2> u(TS * TS);
  fread(u.data(), 16, TS * TS, fopen(argv[1], "rb"));
  std::vector<float2> A(3 * TS * TS), B(3 * TS * TS);
  for (int e = 0; e < TS * TS; ++e) {
    A[TS * TS + e] = make_float2((float)u[e].x, 0.f);        // tile (0, 1); the parts over A and B
    B[TS * TS + e] = make_float2(0.f, (float)u[e].y);
  }
  int texp[3] = {0, 0, 0};
  blockIdx.x = 1;
  if (!simt::run_block(256, false, [&] { k_block_scale64<true>(A.data(), B.data(), 256, 2, texp); })) return 1;
  printf("%%d\n", texp[1]);
}
"""


@pytest.mark.parametrize("name,u,fixed", list(_tiles())[:-1], ids=[t[0] for t in list(_tiles())[:-1]])
def test_choice_of_complex64_tiles(tmp_path, name, u, fixed):
    """The same rule for the residual products of complex64 tiles (k_block_scale64)."""
    c = cut("fx_phases.cuh", "constexpr int FX_THREADS", "constexpr long long FX_SPIN")
    k = cut("k_block_fx.cu", "template <bool HASB>\n__global__ void __launch_bounds__(256)", "// limbs of a float")
    (tmp_path / "u").write_bytes(np.ascontiguousarray(u).tobytes())
    assert (run(tmp_path, SRC32 % (c, k), tmp_path / "u")[0][0] >= 0) == fixed


@pytest.mark.parametrize("name,u,fixed", list(_tiles()), ids=[t[0] for t in _tiles()])
def test_choice_of_tiles(tmp_path, name, u, fixed):
    """Tiles in which some row's magnitude may be far below max|u| max|x| stay with the FP64 kernel."""
    ex, _ = _product(tmp_path, u, np.ones(128))
    assert (ex >= 0) == fixed


@pytest.mark.parametrize("n,tile", [(256, (0, 1)), (228, (1, 1)), (133, (0, 1))])
def test_count_of_weak_entries(tmp_path, n, tile):
    """The most entries of a row or column that are not within 2^-6 of the tile's largest (high words, so to
    2^-20); a diagonal tile's diagonal counts as one of them."""
    rng = np.random.default_rng(n)
    nr, nc = min(128, n - 128 * tile[0]), min(128, n - 128 * tile[1])
    u = np.zeros((128, 128), complex)
    u[:nr, :nc] = _gauss(rng, nr, nc)
    u[3, :nc // 2] *= 2.0 ** -4
    if tile[0] == tile[1]:
        u[np.arange(nr), np.arange(nr)] = 5.0
    ex, _ = _product(tmp_path, u, np.ones(128), n, tile)
    m = np.maximum(np.abs(u.real), np.abs(u.imag))[:nr, :nc]
    if tile[0] == tile[1]:
        np.fill_diagonal(m, 0)
    weak = m < 2.0 ** -6 * m.max()
    top = max(weak.sum(0).max(), weak.sum(1).max())
    assert ex > 0 and _product.weak == [top, top]


def test_edges_of_the_matrix(tmp_path):
    """The zeros beyond the order of the matrix do not count, the diagonal does (but not as the scale)."""
    rng = np.random.default_rng(8)
    g = _gauss(rng, 128, 128)
    g = g + g.conj().T
    cutoff = np.where((np.arange(128)[:, None] < 100) & (np.arange(128)[None, :] < 100), g, 0)
    for d, fixed in ((30.0, True), (1e9, True), (1e-9, False)):
        m = cutoff.copy()
        np.fill_diagonal(m[:100, :100], d)
        assert (_product(tmp_path, m, np.ones(128), 228, (1, 1))[0] >= 0) == fixed, d
