"""The reciprocal of the Sturm counts, the inverse iteration and the back substitution (tree_solve.cuh)
against a division, its hardware approximation replaced by one as coarse."""
import os

import numpy as np

from tests.simt import CSRC, run
from tests.test_warp_order import tree_source

MAIN = r"""
using namespace bse;
int main(int, char** argv) {
  FILE* f = fopen(argv[1], "rb");
  double q;
  while (fread(&q, 8, 1, f) == 1) {
    const double r = argv[2][0] == 'a' ? recip_any(q) : recip(q), d = 1.0 / q;
    // distance in ulps of the quotient; the same bits for zeros and infinities
    long long a = __double_as_longlong(r), b = __double_as_longlong(d);
    if (d != d) a = b = (r != r) ? 0 : (b = 1, 0);
    printf("%lld\n", a > b ? a - b : b - a);
  }
}
"""


def _errors(tmp_path, q, which):
    q = np.concatenate([q, -q])
    (tmp_path / "q").write_bytes(q.tobytes())
    err = np.array(run(tmp_path, tree_source() + MAIN, tmp_path / "q", which))[:, 0]
    assert err.size == q.size
    return err


M = np.random.default_rng(1).uniform(1, 2, 20000)


def test_normal_argument(tmp_path):
    """The unguarded form over the pivots' range."""
    q = np.concatenate([M * 2.0 ** np.random.default_rng(2).integers(-1017, 1000, M.size), 1 + 2.0 ** -52 * np.arange(64),
                        2 - 2.0 ** -52 * np.arange(1, 64)])
    assert _errors(tmp_path, q, "n").max() <= 1


def test_any_argument(tmp_path):
    q = np.concatenate([M * 2.0 ** np.random.default_rng(3).integers(-1022, 1024, M.size), M[:2000] * 2.0 ** -1074,
                        M[:500] * 2.0 ** -1040, M[:500] * 2.0 ** 1022,
                        [0.0, np.inf, np.nan, 5e-324, 2.0 ** -1022, 2.0 ** 1023, 1.7976931348623157e308]])
    assert _errors(tmp_path, q, "a").max() <= 1


def test_smallest_pivots(tmp_path):
    """The guard of the factorisation's pivots is a normal number also for a matrix of norm zero."""
    guards = []
    for name in ("k_ritz.cu", "k_dense.cu"):
        guards += open(os.path.join(CSRC, name)).read().split("pivmin = eps * fmax(")[1:]
    assert len(guards) == 2
    for g in guards:
        assert 2.0 ** -52 * float(g.split(",")[1].split(")")[0]) >= 2.0 ** -1021
