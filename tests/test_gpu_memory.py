"""A complex128 handle holds a second copy of its tiles only while nothing else needs the memory: what fits
without the copy fits with it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
MB = 1 << 20


def _matrices(n, seed=1):
    g = torch.Generator(device="cuda").manual_seed(seed)
    rnd = lambda: torch.complex(torch.randn(n, n, generator=g, device="cuda", dtype=torch.float64),     # noqa: E731
                                torch.randn(n, n, generator=g, device="cuda", dtype=torch.float64)) * 1e-4
    A, B = rnd(), rnd()
    A = (A + A.mH) / 2 + torch.diag(torch.linspace(1.0, 12.0, n, device="cuda", dtype=torch.float64)).to(A.dtype)
    return A.contiguous(), ((B + B.mT) / 2).contiguous()


class _Filled:
    """Device memory taken until about `left` bytes are free."""

    def __init__(self, left):
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        self.t = []
        for chunk in (8 << 30, 512 * MB, 32 * MB):
            while torch.cuda.mem_get_info()[0] > left + chunk:
                self.t.append(torch.empty(chunk, dtype=torch.uint8, device="cuda"))

    def __enter__(self):
        return torch.cuda.mem_get_info()[0]

    def __exit__(self, *a):
        self.t.clear()
        torch.cuda.empty_cache()


def test_solve_takes_the_memory_of_the_copy():
    """2 x 135 MB of tiles and as much of copies; the solve's buffers need about 330 MB."""
    from paper_2504_10096_gb300 import bse
    A, B = _matrices(4000)
    s = bse.Solver(A, B)
    ref, _, _ = s.solve(6, tol=1e-11, vectors=False)
    s.close()
    s = bse.Solver(A, B)
    x = torch.ones(4000, dtype=A.dtype, device="cuda")
    y = s.apply(bse.BSE_OP_MPLUS, x)
    with _Filled(200 * MB) as free:
        assert free < 260 * MB
        vals, _, nconv = s.solve(6, tol=1e-11, ncv=1000, vectors=False)
        again = s.apply(bse.BSE_OP_MPLUS, x)                    # now in FP64
    assert nconv == 6
    np.testing.assert_allclose(vals, ref, rtol=1e-10, atol=0)
    assert float((again - y).abs().max()) <= 64 * 2.0 ** -53 * float((A.abs() + B.abs()).sum(1).max())
    vals, _, nconv = s.solve(6, tol=1e-11, vectors=False)       # graphs of the kernels that are left
    assert nconv == 6
    np.testing.assert_allclose(vals, ref, rtol=1e-10, atol=0)
    s.close()


def test_new_handle_takes_the_memory_of_an_idle_one():
    from paper_2504_10096_gb300 import bse
    A, B = _matrices(4000)
    first = bse.Solver(A, B)
    r0, _, _ = first.solve(4, tol=1e-11, vectors=False)
    with _Filled(200 * MB):
        second = bse.Solver(A, B)                               # 270 MB of tiles
        r2, _, n2 = second.solve(4, tol=1e-11, vectors=False)
        r1, _, n1 = first.solve(4, tol=1e-11, vectors=False)
    assert n1 == n2 == 4
    np.testing.assert_allclose(r1, r0, rtol=1e-10, atol=0)
    np.testing.assert_allclose(r2, r0, rtol=1e-10, atol=0)
    first.close()
    second.close()


def test_handle_reports_its_arithmetic():
    """How many tiles run in fixed point: all of a dense matrix (3 x 3 blocks); of a graded one only the
    last, whose 44 rows differ by 10^1.7 and its entries by 10^3.5 (the other tiles' by 10^6.9 at least);
    none of a complex64 handle; none after the copy was given up."""
    from paper_2504_10096_gb300 import bse
    A, B = _matrices(300)
    d = torch.logspace(0, -12, 300, dtype=torch.float64, device="cuda").to(A.dtype)
    for a, b, fixed in ((A, B, 6), (A * d[:, None] * d[None, :], B * d[:, None] * d[None, :], 1),
                        (A.to(torch.complex64), B.to(torch.complex64), 0)):
        s = bse.Solver(a, b)
        assert bse.bse_get_fixed_point(s.h) == (fixed, 6)
        s.close()
    A, B = _matrices(4000)
    s = bse.Solver(A, B)
    assert bse.bse_get_fixed_point(s.h) == (528, 528)
    with _Filled(200 * MB):
        s.solve(4, tol=1e-9, ncv=1000, vectors=False)
    assert bse.bse_get_fixed_point(s.h) == (0, 528)
    s.close()
