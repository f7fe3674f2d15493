"""complex128 products on matrices and vectors whose entries differ by many orders of magnitude, element
by element against |M||x|: a product that is accurate only against the largest entry of a tile or of a
chunk of the vector does not pass.  The constant is that of the other product tests (a few tens of
roundings per entry), also where one entry of x is far above the others."""
import numpy as np
import pytest

from tests.gpu_common import UNIT, assert_elementwise, product_bound

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _matrices(rng, n):
    """Dense Hermitian A with a small diagonal, dense symmetric B."""
    g = lambda: rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))        # noqa: E731
    a, b = g(), g()
    return (a + a.conj().T) / 2, (b + b.T) / 4


def _graded(a, b, d):
    return a * d[:, None] * d[None, :], b * d[:, None] * d[None, :]


def _cases(n):
    rng = np.random.default_rng(n)
    a, b = _matrices(rng, n)
    x = rng.standard_normal((n, 1)) + 1j * rng.standard_normal((n, 1))
    half = np.arange(n) % 128 >= 64
    same = half[:, None] == half[None, :]
    yield "two uncoupled blocks, one part of x at 1e-12", a * same, b * same, np.where(half[:, None], 1e-12 * x, x)
    yield "two uncoupled blocks, one part of x at 1e-19", a * same, b * same, np.where(half[:, None], 1e-19 * x, x)
    yield ("graded rows and columns", *_graded(a, b, np.where(half, 1e-10, 1.0)), x)
    yield ("one row far above the others", *_graded(a, b, np.where(np.arange(n) == 5 % n, 1.0, 1e-6)), x)
    out = x.copy()
    out[n // 3] *= 1e10
    yield "an entry of x far above the others", a, b, out
    hole = np.ones((n, n))
    hole[n // 2:, n // 3] = hole[n // 3, n // 2:] = 0
    yield "... that some rows do not see", a * hole, b * hole, out
    peak = np.ones((n, n))
    peak[0, n - 1] = peak[n - 1, 0] = 1e5
    z = x.copy()
    z[[0, n - 1]] = 0
    yield "a peak that x does not see", a * peak, b * peak, z
    yield "x of 1e-300", a, b, 1e-300 * x
    yield "x near the smallest normal number", 2.0 ** 40 * a, 2.0 ** 40 * b, 2.0 ** -1015 * x
    yield "x of 1e300", 2.0 ** -40 * a, 2.0 ** -40 * b, 1e300 * x


NAMES = [c[0] for c in _cases(3)]


@pytest.mark.parametrize("form", ["ph", "tda"])
@pytest.mark.parametrize("n", [96, 300])
@pytest.mark.parametrize("name", NAMES)
def test_every_entry(name, n, form):
    from paper_2504_10096_gb300 import bse
    _, a, b, x = next(c for c in _cases(n) if c[0] == name)
    s = bse.Solver(torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda() if form == "ph" else None)
    L = np.clongdouble
    al, bl, xl = a.astype(L), b.astype(L), x.astype(L)
    ops = [(bse.BSE_OP_A, "a", al @ xl)]
    if form == "ph":
        ops += [(bse.BSE_OP_MPLUS, "mplus", al @ xl + bl @ xl.conj()),
                (bse.BSE_OP_MMINUS, "mminus", al @ xl - bl @ xl.conj())]
    for op, kind, ref in ops:
        # scaled to keep the checks' own squares and sums in range
        f = 2.0 ** np.round(-np.log2(np.abs(ref).max().astype(float)))
        bound = product_bound(a, b, x * f, kind)
        for k in (1, 3):
            y = s.apply(op, torch.from_numpy(np.repeat(x, k, 1)).cuda()).cpu().numpy()
            for c in range(k):
                assert_elementwise(y[:, c:c + 1] * f, (ref * f).astype(complex), bound, UNIT["c128"], 64, f"{name}, {kind}, k = {k}")
    s.close()


@pytest.mark.parametrize("form", ["ph", "tda"])
@pytest.mark.parametrize("n", [100, 300, 1300])
def test_weak_couplings_to_an_outlier(n, form):
    """Entries of size one, some rows coupled by 2^-15 to the one entry of x that counts: every tile is in
    fixed point, and its sums for those rows are far below the scales.  Bands at the smaller orders."""
    from paper_2504_10096_gb300 import bse
    rng = np.random.default_rng(n)
    ph = np.exp(2j * np.pi * rng.random((n, n)))
    a = np.triu(ph, 1)
    a = a + a.conj().T + np.eye(n)
    b = 0.3 * np.exp(2j * np.pi * rng.random((n, n)))
    b = np.triu(b) + np.triu(b, 1).T
    out, weak = n // 3, np.concatenate([np.arange(n // 2, n // 2 + 9), [n - 1]])
    for m in (a, b):
        m[weak, out] *= 2.0 ** -15
        m[out, weak] *= 2.0 ** -15
    x = rng.standard_normal((n, 1)) + 1j * rng.standard_normal((n, 1))
    x[out] *= 1e10
    s = bse.Solver(torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda() if form == "ph" else None)
    nt = -(-n // 128)
    assert bse.bse_get_fixed_point(s.h) == (nt * (nt + 1) // 2,) * 2
    L = np.clongdouble
    al, bl, xl = a.astype(L), b.astype(L), x.astype(L)
    ops = [(bse.BSE_OP_A, "a", al @ xl)]
    if form == "ph":
        ops += [(bse.BSE_OP_MPLUS, "mplus", al @ xl + bl @ xl.conj()), (bse.BSE_OP_MMINUS, "mminus", al @ xl - bl @ xl.conj())]
    for op, kind, ref in ops:
        for k in (1, 3, 17):
            y = s.apply(op, torch.from_numpy(np.repeat(x, k, 1)).cuda()).cpu().numpy()
            for c in (0, k - 1):
                assert_elementwise(y[:, c:c + 1], ref.astype(complex), product_bound(a, b, x, kind), UNIT["c128"], 64, f"{kind}, k = {k}")
    # an infinite entry: what FP64 arithmetic gives, infinities and no NaN (on blocks of the PH form A x and
    # B conj(x) meet with opposite signs, inf - inf)
    x[out] = np.inf
    op = bse.BSE_OP_MPLUS if form == "ph" else bse.BSE_OP_A
    for k in (1, 2) if form == "tda" else (1,):
        y = s.apply(op, torch.from_numpy(np.repeat(x, k, 1)).cuda()).cpu().numpy()
        assert np.isinf(y[:, 0].real).all() and np.isinf(y[:, 0].imag[np.arange(n) != out]).all()
    s.close()


@pytest.mark.parametrize("n,k", [(3, 40000), (1100, 2900)])
def test_more_columns_than_one_launch_takes(n, k):
    """H on blocks that the block kernels take in several groups of columns."""
    from paper_2504_10096_gb300 import bse
    rng = np.random.default_rng(k)
    a, b = _matrices(rng, n)
    X = torch.randn(2 * n, k, dtype=torch.complex128, device="cuda")
    s = bse.Solver(torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda())
    Y = s.apply(bse.BSE_OP_H, X)
    s.close()
    at, bt = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
    ref = torch.cat([at @ X[:n] + bt @ X[n:], -(bt.conj() @ X[:n] + at.conj() @ X[n:])])
    mag = torch.cat([at.abs() @ X[:n].abs() + bt.abs() @ X[n:].abs(), bt.abs() @ X[:n].abs() + at.abs() @ X[n:].abs()])
    assert bool(((Y - ref).abs() <= 64 * UNIT["c128"] * 2 * mag).all())       # both sides are off by as much


@pytest.mark.parametrize("form", ["ph", "tda"])
@pytest.mark.parametrize("n", [140, 520, 1300])
def test_solve_with_tiles_of_both_kinds(n, form):
    """A matrix with holes in every other off-diagonal tile and one graded stripe: the tiles divide between
    fixed point (in bands at these orders) and FP64, in the persistent launch, the replayed graphs and the
    single launches alike."""
    from paper_2504_10096_gb300 import bse
    rng = np.random.default_rng(n)
    a, b = _matrices(rng, n)
    a, b = 1e-3 * a, 1e-3 * b
    for m in (a, b):
        for i in range(0, n, 256):
            if i + 130 < n:
                m[i + 3, i + 130] = m[i + 130, i + 3] = 0
        m[:5] *= 1e-9
        m[:, :5] *= 1e-9
    np.fill_diagonal(a, np.linspace(1.0, 9.0, n))
    s = bse.Solver(torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda() if form == "ph" else None)
    fixed, tiles = bse.bse_get_fixed_point(s.h)
    assert 0 < fixed < tiles
    out = [s.solve(8, tol=1e-12, **kw) for kw in ({}, {"persistent": False}, {"graphs": False})]
    for vals, vecs, nconv in out:
        assert nconv == 8 and s.residuals().max() <= 1e-12
        assert np.array_equal(vals, out[0][0]) and torch.equal(vecs, out[0][1])
    s.close()
    if form == "tda":
        ref = np.linalg.eigvalsh(a)[:8]
    else:
        real = lambda t: np.block([[a.real + t * b.real, -a.imag + t * b.imag], [a.imag + t * b.imag, a.real - t * b.real]])  # noqa: E731
        low = np.linalg.cholesky(real(-1.0))
        ref = np.sqrt(np.linalg.eigvalsh(low.T @ real(1.0) @ low)[:16:2])
    np.testing.assert_allclose(out[0][0], ref, rtol=1e-11, atol=0)
