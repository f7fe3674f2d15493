"""Fine and coarse tiles of the mixed product in one launch: every split of the tiles between the two
kinds, against the real form of Eq. 5 with the coarse tiles' U and V rounded to FP32."""
import numpy as np
import pytest

from tests.gpu_common import problem, rand_block

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
T = 128


@pytest.mark.parametrize("n,counts", [(300, (1, 2, 3, 5)), (1100, (1, 8, 9, 44))])
def test_any_split_of_fine_and_coarse_tiles(n, counts):
    from paper_2504_10096_gb300 import bse
    A, B = problem(n, "c64", seed=n)
    nt = -(-n // T)
    tiles = [(i, j) for i in range(nt) for j in range(i, nt)]
    cut = lambda m, i, j: m[T * i:T * i + T, T * j:T * j + T]                         # noqa: E731
    top = np.array([max((np.abs(cut(A, i, j).real) + np.abs(cut(B, i, j).real)).max(),
                        (np.abs(cut(A, i, j).imag) + np.abs(cut(B, i, j).imag)).max()) for i, j in tiles])
    s = bse.Solver(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), mixed=True)
    x = rand_block(n, 1, "c128", seed=9)[:, 0]
    xt = torch.from_numpy(x).cuda()
    order = np.sort(top / top.max())[::-1]
    for fine in counts:
        tau = float(np.sqrt(order[fine - 1] * order[fine]))
        for op, sgn in ((bse.BSE_OP_MPLUS, 1.0), (bse.BSE_OP_MMINUS, -1.0)):
            y = torch.full_like(xt, float("nan"))
            assert bse.bse_apply_mixed(s.h, op, tau, xt.data_ptr(), y.data_ptr()) == bse.BSE_OK
            assert (s.stats()["tiles_fine"], s.stats()["tiles_coarse"]) == (fine, len(tiles) - fine)
            rounded = np.zeros((n, n), bool)
            for (i, j), t in zip(tiles, top / top.max()):
                cut(rounded, i, j)[:] = cut(rounded, j, i)[:] = t <= tau
            part = {}
            for name, f in (("re", np.real), ("im", np.imag)):
                a, b = f(A).astype(np.float64), sgn * f(B).astype(np.float64)
                part[name] = [np.where(rounded, (m).astype(np.float32).astype(np.float64), m) for m in (a + b, a - b)]
            (ure, vre), (uim, vim) = part["re"], part["im"]
            emu = (ure @ x.real - vim @ x.imag) + 1j * (uim @ x.real + vre @ x.imag)
            scale = np.max((np.abs(ure) + np.abs(vim) + np.abs(uim) + np.abs(vre)) @ np.abs(x))
            assert np.max(np.abs(y.cpu().numpy() - emu)) <= 2.0 ** -30 * scale, (fine, sgn)
    s.close()
