"""The fixed-point complex128 product (fx_phases.cuh) against extended precision.

Sizes sit at the edges of a tile, at the numbers of tiles where the split into bands changes, and
on both forms; matrices with a peak in one tile, with huge and tiny entries and with a NaN go
(partly) through the FP64 kernel instead.

Bound per row: a term u x is off by at most 3 2^-60 of 2^(E_u + E_x) (the roundings of u and x and
the dropped low product), 256 terms per tile row, 2^E at most twice the largest component: 12 2^-52
max|u| max|x| per tile.  The FP64 sums of the slots and the diagonal add at most one rounding of
the magnitude sum per slot and per diagonal term."""
import numpy as np
import pytest

from tests.gpu_common import problem

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
T = 128


def _product(A, B, x, op):
    from paper_2504_10096_gb300 import bse
    s = bse.Solver(torch.from_numpy(A).cuda(), None if B is None else torch.from_numpy(B).cuda())
    y = s.apply(op, torch.from_numpy(x).cuda()).cpu().numpy()
    s.close()
    return y


def _reference(A, B, x, sign):
    L = np.clongdouble
    y = (A.astype(L) * x.astype(L)[None, :]).sum(1)
    return y + sign * (B.astype(L) * x.conj().astype(L)[None, :]).sum(1) if sign else y


def _bound(A, B, x):
    n = A.shape[0]
    nt = -(-n // T)
    comp = lambda m: np.maximum(np.abs(m.real), np.abs(m.imag))                # noqa: E731
    mag = np.abs(A) if B is None else np.abs(A) + np.abs(B)
    off = comp(A) if B is None else comp(A) + comp(B)
    np.fill_diagonal(off, 0.0)
    out = (8 * nt + 16) * 2.0 ** -53 * (mag @ np.abs(x))
    for i in range(nt):
        for j in range(nt):
            u = off[T * i:T * i + T, T * j:T * j + T].max()
            out[T * i:T * i + T] += 12 * 2.0 ** -52 * u * comp(x[T * j:T * j + T]).max()
    return out


def _check(A, B, x):
    from paper_2504_10096_gb300 import bse
    ops = [(bse.BSE_OP_A, 0)] if B is None else [(bse.BSE_OP_MPLUS, 1), (bse.BSE_OP_MMINUS, -1)]
    for op, sign in ops:
        y = _product(A, B, x, op)
        err = np.abs(y - _reference(A, B, x, sign)).astype(np.float64)
        assert np.all(err <= _bound(A, B, x)), float(np.max(err / _bound(A, B, x)))


@pytest.mark.parametrize("form", ["ph", "tda"])
@pytest.mark.parametrize("n", [1, 2, 127, 128, 129, 385, 700, 1153])
def test_matches_extended_precision(form, n):
    A, B = problem(n, "c128", form=form, seed=n)
    rng = np.random.default_rng(n)
    x = (rng.standard_normal(n) + 1j * rng.standard_normal(n)) * np.exp(2 * rng.standard_normal(n))
    _check(A, B, x)


@pytest.mark.parametrize("scale", [2.0 ** -300, 1.0, 2.0 ** 300])
def test_peaked_tile_and_far_scales(scale):
    """One entry 1e5 times its tile's others (FP64 tile), a zero tile, entries far from one."""
    n = 300
    A, B = problem(n, "c128", seed=4)
    A[3, 200] *= 1e5
    A[200, 3] = A[3, 200].conj()
    B[:128, 256:] = 0
    B[256:, :128] = 0
    A[:128, 256:] = 0
    A[256:, :128] = 0
    rng = np.random.default_rng(1)
    x = rng.standard_normal(n) + 1j * rng.standard_normal(n)
    x[130:250] = 0
    _check(A * scale, B * scale, x / scale)


def test_nan_and_inf_reach_the_result():
    from paper_2504_10096_gb300 import bse
    n = 300
    A, B = problem(n, "c128", seed=4)
    rng = np.random.default_rng(2)
    x = rng.standard_normal(n) + 1j * rng.standard_normal(n)
    for bad in (np.nan, np.inf):
        xb = x.copy()
        xb[7] = bad
        assert not np.isfinite(_product(A, B, xb, bse.BSE_OP_MPLUS)).any()
        Ab = A.copy()
        Ab[5, 140] = bad
        y = _product(Ab, B, x, bse.BSE_OP_MPLUS)
        assert not np.isfinite(y[5]) and not np.isfinite(y[140])


@pytest.mark.parametrize("form,n,k", [("ph", 1, 2), ("ph", 127, 3), ("ph", 129, 16), ("ph", 385, 17), ("ph", 700, 33),
                                      ("tda", 2, 2), ("tda", 128, 15), ("tda", 513, 20)])
def test_blocks_match_extended_precision(form, n, k):
    """bse_apply on k columns (the fixed-point block kernel) at the edges of its 64 x 16 units; the
    columns of very different size.  The PH form multiplies P = A + B and Q = A - B with
    (XA +- XB) / 2, so its bound holds for the larger of the two vectors; one more rounding each for
    P, Q and the half sums."""
    from paper_2504_10096_gb300 import bse
    A, B = problem(n, "c128", form=form, seed=n)
    rng = np.random.default_rng(n)
    rows = 2 * n if form == "ph" else n
    X = (rng.standard_normal((rows, k)) + 1j * rng.standard_normal((rows, k))) * 10.0 ** rng.integers(-6, 7, k)
    s = bse.Solver(torch.from_numpy(A).cuda(), None if B is None else torch.from_numpy(B).cuda())
    L = np.clongdouble
    a, b = A.astype(L), None if B is None else B.astype(L)
    if form == "tda":
        refs = {bse.BSE_OP_A: (X, a @ X.astype(L))}
    else:
        x1, x2 = X[:n].astype(L), X[n:].astype(L)
        refs = {bse.BSE_OP_H: (X, np.vstack([a @ x1 + b @ x2, -(b.conj() @ x1 + a.conj() @ x2)])),
                bse.BSE_OP_MPLUS: (X[:n], a @ x1 + b @ x1.conj()), bse.BSE_OP_A: (X[:n], a @ x1)}
    for op, (V, ref) in refs.items():
        y = s.apply(op, torch.from_numpy(np.ascontiguousarray(V)).cuda()).cpu().numpy()
        for c in range(k):
            big = np.abs(V[:n, c]) + (np.abs(V[n:, c]) if op == bse.BSE_OP_H else 0)
            bnd = _bound(A, B, big.astype(complex)) * (1.0 if form == "tda" else 3.0)
            err = np.abs(y[:, c] - ref[:, c]).astype(np.float64)
            lim = np.concatenate([bnd, bnd]) if op == bse.BSE_OP_H else bnd
            assert np.all(err <= lim), (op, c, float(np.max(err / lim)))
    s.close()
