"""Workloads of the Bethe-Salpeter solver, as a program that uses it would run them.

Each case is a dict of plain values; `prepare` makes its inputs and the handle a program keeps,
`run` takes them once through the public entry points, `work` says what the job cannot do without
and `exact` computes the same outputs with plain torch in 64 bits.

The matrices are seeded stand-ins for a semiconductor's: transition energies on a jittered grid
(what a regular k-mesh gives) on the diagonal of A, plus an exchange term and minus a screened
direct term of 96 plane waves with Coulomb weights; B is the exchange coupling.  Norms as in the
synthetic workloads: 0.3, 0.2 and at most 0.15 eV.
"""
import math

import numpy as np
import torch

from paper_2504_10096_gb300 import bse

N_G = 96


def listed():
    return [
        # the smallest call: one product of a small problem straight from the caller's matrices, inside
        # a latency-bound loop that may not allocate
        {"name": "product-noalloc-600", "kind": "noalloc", "dtype": "c64", "n": 600, "op": "mplus"},
        # H applied to a block of vectors (checking or refining a set of eigenpairs)
        {"name": "apply-h-block-1500", "kind": "block", "dtype": "c128", "n": 1500, "k": 20},
        # one product of a program's own iteration on single-precision matrices, N not a multiple of a tile
        {"name": "product-c64-12001", "kind": "product", "dtype": "c64", "n": 12001, "op": "mplus"},
        # the Lanczos product of the mixed path at the order of the differentiable workload
        {"name": "product-mixed-20000", "kind": "mixed", "dtype": "c64", "n": 20000, "op": "mminus"},
        # absorption spectrum without eigenpairs, FP64: the Lanczos-Haydock recurrence
        {"name": "haydock-c128-8000", "kind": "haydock", "dtype": "c128", "form": "ph", "n": 8000, "m": 60},
        # Tamm-Dancoff eigenpairs, FP64 (the smallest of the standard workloads)
        {"name": "tda-2000", "kind": "solve", "dtype": "c128", "form": "tda", "n": 2000, "nev": 20},
        # the headline's path (pseudo-Hermitian, FP64, tight residuals) at an order a pass of which is short
        {"name": "ph-3000", "kind": "values", "dtype": "c128", "form": "ph", "n": 3000, "nev": 30},
        # the mixed path on single-precision matrices to residual 1e-6
        {"name": "ph-mixed-5000", "kind": "values", "dtype": "mixed", "form": "ph", "n": 5000, "nev": 32},
        # momentum transfers of uneven order solved together on the mixed path
        {"name": "batch-mixed-12", "kind": "batch", "dtype": "mixed", "n": 2400, "count": 12, "nev": 16},
        # one step of a differentiable model: eigenvalues of new matrices, a loss, its gradients
        {"name": "train-900", "kind": "train", "dtype": "c128", "form": "ph", "n": 900, "nev": 16},
        # the adjoint of a single-precision model's solve: dense gradients of the matrices
        {"name": "backward-c64-6000", "kind": "backward", "dtype": "mixed", "n": 6000, "nev": 32},
        # direct diagonalisation where a large share of the spectrum is wanted
        {"name": "dense-300", "kind": "dense", "dtype": "c128", "n": 300, "nev": 60},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["noalloc", "block", "product", "mixed", "haydock", "solve", "values", "batch", "train",
                       "dense", "backward"])
    op = rng.choice(["mplus", "mminus"])
    prec = rng.choice(["c64", "c128"])
    if kind == "noalloc":
        return {"kind": kind, "dtype": prec, "n": _log(rng, 60, 4096), "op": rng.choice([op, "a"])}
    if kind == "block":
        return {"kind": kind, "dtype": prec, "n": _log(rng, 200, 3000), "k": rng.randint(2, 32)}
    if kind == "product":
        return {"kind": kind, "dtype": prec, "n": _log(rng, 500, 16000), "op": op}
    if kind == "mixed":
        return {"kind": kind, "dtype": "c64", "n": _log(rng, 2000, 24000), "op": op}
    if kind == "haydock":
        return {"kind": kind, "dtype": "c128", "form": rng.choice(["ph", "tda"]), "n": _log(rng, 800, 8000),
                "m": rng.randint(20, 60)}
    if kind == "solve":
        return {"kind": kind, "dtype": "c128", "form": rng.choice(["ph", "tda"]), "n": rng.randint(200, 1600),
                "nev": rng.randint(4, 20)}
    if kind == "values":
        # the FP64 path, its double-FP32 products, the mixed path, and the structured variants
        dtype, variant = rng.choice([("c128", "shao"), ("c128", "shao"), ("df", "shao"), ("mixed", "shao"),
                                     ("c128", "gruning"), ("c128", "projected")])
        top = 3000 if variant == "shao" else 1000
        return {"kind": kind, "dtype": dtype, "form": "ph", "n": rng.randint(400, top), "nev": rng.randint(8, 30),
                "variant": variant}
    if kind == "batch":
        return {"kind": kind, "dtype": "mixed", "n": rng.randint(800, 2400), "count": rng.randint(3, 12),
                "nev": rng.randint(6, 16)}
    if kind == "train":
        return {"kind": kind, "dtype": "c128", "form": rng.choice(["ph", "tda"]), "n": rng.randint(100, 900),
                "nev": rng.randint(4, 16)}
    if kind == "dense":
        return {"kind": kind, "dtype": "c128", "n": rng.randint(60, 300), "nev": rng.randint(6, 50)}
    return {"kind": kind, "dtype": "mixed", "n": rng.randint(600, 6000), "nev": rng.randint(8, 32)}


# ---------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _cplx(g, *shape):
    return torch.complex(torch.randn(*shape, generator=g, device="cuda", dtype=torch.float64),
                         torch.randn(*shape, generator=g, device="cuda", dtype=torch.float64)) / math.sqrt(2)


def _matrices(n, dtype, seed, form="ph"):
    """A (Hermitian) and B (symmetric; None for the Tamm-Dancoff form), stored in full."""
    g = _gen(seed)
    # |G|^2 grows like the 2/3 power of the plane wave's rank
    v = 1.0 / ((torch.arange(N_G, device="cuda", dtype=torch.float64) * 0.24) ** (2.0 / 3.0) + 0.1)
    jitter = torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
    energies = 1.5 + 8.5 * (torch.arange(n, device="cuda") + 0.5 * jitter) / n
    f = v.sqrt()[:, None] * _cplx(g, N_G, n)
    fw = v.sqrt()[:, None] * _cplx(g, N_G, n)
    lx, lw = (torch.linalg.eigvalsh(m @ m.mH)[-1] for m in (f, fw))
    cdt = torch.complex128 if dtype in ("c128", "df") else torch.complex64
    left = torch.cat([f * (0.3 / lx), fw * (-0.2 / lw)]).to(cdt)
    right = torch.cat([f, fw]).to(cdt)
    a = left.mH @ right
    a = torch.triu(a, 1)
    a = a + a.mH
    a.diagonal().copy_(energies + (left.conj() * right).sum(0).real)
    if form == "tda":
        return a, None
    b = (f * (0.15 / lx)).to(cdt).mH @ f.to(cdt).conj()
    b = torch.triu(b) + torch.triu(b, 1).mT
    return a, b


def _batch_orders(case):
    """Uneven orders up to n, as different momentum transfers give."""
    c = case["count"]
    return [max(case["nev"] + 40, int(case["n"] * (0.2 + 0.8 * (i + 1) / c)) - 7 * i) for i in range(c)]


def _solver(case, seed):
    a, b = _matrices(case["n"], case["dtype"], seed, case.get("form", "ph"))
    return bse.Solver(a, b, df=case["dtype"] == "df", mixed="mixed" in (case["kind"], case["dtype"]))


OPS = {"a": bse.BSE_OP_A, "mplus": bse.BSE_OP_MPLUS, "mminus": bse.BSE_OP_MMINUS}
VARIANTS = {"shao": bse.BSE_VARIANT_SHAO, "gruning": bse.BSE_VARIANT_GRUNING,
            "projected": bse.BSE_VARIANT_PROJECTED}


def _vector(case, seed):
    x = _cplx(_gen(seed + 1), case["n"])
    return x.to(torch.complex64) if case["dtype"] == "c64" and case["kind"] != "mixed" else x


def _weights(case, seed):
    g = np.random.default_rng([seed, 2])
    return g.uniform(0.0, 1.0, case["nev"]), g.uniform(1.5, 2.0, case["nev"])


def prepare(case, seed):
    bse.load_library()
    kind, n = case["kind"], case["n"]
    st = {"case": case}
    if kind == "noalloc":
        st["A"], st["B"] = _matrices(n, case["dtype"], seed)
        st["x"] = _vector(case, seed)
        st["y"] = torch.empty_like(st["x"])
    elif kind == "train":
        a, b = _matrices(n, case["dtype"], seed, case["form"])
        st["A"] = a.requires_grad_()
        st["B"] = b.requires_grad_() if b is not None else None
        st["w"], st["t"] = (torch.from_numpy(v).cuda() for v in _weights(case, seed))
    elif kind == "batch":
        mats = [_matrices(m, "mixed", seed * 64 + i) for i, m in enumerate(_batch_orders(case))]
        st["solver"] = bse.BatchedSolver([m[0] for m in mats], [m[1] for m in mats], mixed=True)
    else:
        st["solver"] = _solver(case, seed)
        if kind == "block":
            st["X"] = _cplx(_gen(seed + 1), 2 * n, case["k"])
            if case["dtype"] == "c64":
                st["X"] = st["X"].to(torch.complex64)
        elif kind in ("product", "mixed"):
            st["x"] = _vector(case, seed)
            st["y"] = torch.empty_like(st["x"])
        elif kind == "haydock":
            st["d"] = _cplx(_gen(seed + 1), n)
            st["omega"] = np.linspace(1.0, 10.0, 1001)
        elif kind == "backward":
            st["solver"].solve(case["nev"], tol=1e-10)       # tight: the gradient needs the vectors
            st["g"] = _weights(case, seed)[0]
    return st


# ---------------------------------------------------------------- one pass
def _fix_phase(v):
    """Columns with a real positive largest entry (an eigenvector's phase is arbitrary)."""
    top = torch.gather(v, 0, v.abs().argmax(0, keepdim=True))
    return v * (top.conj() / top.abs())


def run(st):
    case = st["case"]
    kind, s = case["kind"], st.get("solver")
    if kind == "noalloc":
        bse._check(bse.bse_apply_noalloc(case["n"], st["A"].data_ptr(), st["B"].data_ptr(),
                                         bse.BSE_C128 if case["dtype"] == "c128" else bse.BSE_C64, OPS[case["op"]],
                                         st["x"].data_ptr(), st["y"].data_ptr(),
                                         torch.cuda.current_stream().cuda_stream), "product")
        return st["y"]
    if kind == "block":
        return s.apply(bse.BSE_OP_H, st["X"])
    if kind == "product":
        return s.apply(OPS[case["op"]], st["x"])
    if kind == "mixed":
        bse._check(bse.bse_apply_mixed(s.h, OPS[case["op"]], 0.0, st["x"].data_ptr(), st["y"].data_ptr()), "product")
        return st["y"]
    if kind == "haydock":
        spectrum, response, coefs, steps = s.haydock(st["d"], case["m"], st["omega"], 0.1)
        return spectrum, response, coefs["alpha"], coefs["beta"], coefs["norm2"], steps
    if kind == "solve":
        vals, vecs, nconv = s.solve(case["nev"], tol=1e-12)
        return vals, _fix_phase(vecs), nconv
    if kind == "values":
        vals, _, nconv = s.solve(case["nev"], tol=1e-6 if case["dtype"] == "mixed" else 1e-12, vectors=False,
                                 variant=VARIANTS[case.get("variant", "shao")])
        return vals, nconv
    if kind == "batch":
        vals, _, nconv = s.solve(case["nev"], tol=1e-6)
        return vals, nconv
    if kind == "train":
        vals = bse.bse_eigenvalues(st["A"], st["B"], case["nev"], tol=1e-12)
        loss = (st["w"] * vals).sum() + ((vals - st["t"]) ** 2).sum()
        wrt = [t for t in (st["A"], st["B"]) if t is not None]
        return [vals.detach(), *torch.autograd.grad(loss, wrt)]
    if kind == "dense":
        vals, vecs, nconv = s.solve_dense(case["nev"])
        return vals, _fix_phase(vecs), nconv
    if kind == "backward":
        return s.backward(st["g"])
    raise ValueError(kind)


# ---------------------------------------------------------------- work and reference values
def work(case):
    kind, n = case["kind"], case["n"]
    e = 16 if case["dtype"] in ("c128", "df") else 8
    mats = 1 if case.get("form") == "tda" or case.get("op") == "a" else 2
    tri = mats * e * n * (n + 1) // 2             # the stored triangles, read once
    nev = case.get("nev", 0)
    if kind in ("noalloc", "product"):
        return {"bytes": tri + 2 * n * e, "flops": 8.0 * n * n}
    if kind == "mixed":
        return {"bytes": tri + 2 * n * 16, "flops": 8.0 * n * n}
    if kind == "block":
        return {"bytes": tri + 4 * n * case["k"] * e, "flops": 32.0 * n * n * case["k"]}
    if kind == "haydock":
        return {"bytes": tri + 16 * n + 8 * 1001 * 4, "flops": 8.0 * n * n * case["m"] * mats}
    if kind == "backward":
        return {"bytes": 2 * n * nev * 16 + 2 * n * n * e, "flops": 16.0 * n * n * nev}
    if kind == "dense":
        return {"bytes": tri + 2 * n * nev * e, "flops": (1 / 3 + 1 + 4 / 3) * (2.0 * n) ** 3}
    # a Krylov space that holds nev vectors took at least nev steps
    if kind == "batch":
        ms = _batch_orders(case)
        return {"bytes": sum(8 * m * (m + 1) for m in ms), "flops": sum(16.0 * m * m * nev for m in ms)}
    flops = 8.0 * n * n * mats * nev
    if kind == "train":
        return {"bytes": tri + mats * n * n * e, "flops": flops + 8.0 * mats * n * n * nev}
    out = (2 if mats == 2 else 1) * n * nev * e if kind == "solve" else 0
    return {"bytes": tri + out, "flops": flops}


def _wide(case, seed):
    a, b = _matrices(case["n"], case["dtype"], seed, case.get("form", "ph"))
    return a.to(torch.complex128), b.to(torch.complex128) if b is not None else None


def _half(a, b, s, x):
    """A x + s B conj(x)."""
    return a @ x + s * (b @ x.conj()) if b is not None and s else a @ x


def _eigenpairs(a, b, nev):
    """Lowest eigenvalues with X, Y (Y None for the Tamm-Dancoff form), Omega-normalised."""
    if b is None:
        w, x = torch.linalg.eigh(a)
        return w[:nev], x[:, :nev], None
    real = lambda s: torch.cat([torch.cat([a.real + s * b.real, -a.imag + s * b.imag], 1),        # noqa: E731
                                torch.cat([a.imag + s * b.imag, a.real - s * b.real], 1)], 0)
    mp, low = real(1.0), torch.linalg.cholesky(real(-1.0))
    w, y = torch.linalg.eigh(low.mT @ mp @ low)
    u = low @ y[:, 0:2 * nev:2]                     # every omega^2 is double
    n = a.shape[0]
    u, om = torch.complex(u[:n], u[n:]), w[0:2 * nev:2].sqrt()
    p = a @ u + b @ u.conj()
    x, yc = om * u + p, (om * u - p).conj()
    x, yc = x.contiguous(), yc.resolve_conj().contiguous()
    nrm = (x.abs().square().sum(0) - yc.abs().square().sum(0)).sqrt()
    return om, x / nrm, yc / nrm


def _gradients(x, y, g):
    g = torch.as_tensor(g, device=x.device).to(x.dtype)
    da = (x * g) @ x.mH
    if y is None:
        return (da,)
    db = (x * g) @ y.mH
    return da + ((y * g) @ y.mH).conj(), db + db.mT


def exact(case, seed):
    kind, n = case["kind"], case["n"]
    if kind == "batch":
        return None
    if kind not in ("noalloc", "block", "product", "mixed", "haydock") and \
            (2 if case.get("form") != "tda" else 1) * n > 3400:
        return None
    a, b = _wide(case, seed)
    if kind in ("noalloc", "product", "mixed"):
        s = {"a": 0.0, "mplus": 1.0, "mminus": -1.0}[case["op"]]
        return _half(a, b, s, _vector(case, seed).to(torch.complex128))
    if kind == "block":
        x = _cplx(_gen(seed + 1), 2 * n, case["k"])
        x = x.to(torch.complex64).to(torch.complex128) if case["dtype"] == "c64" else x
        return torch.cat([a @ x[:n] + b @ x[n:], -(b.conj() @ x[:n] + a.conj() @ x[n:])])
    if kind == "haydock":
        return _haydock(a, b, _cplx(_gen(seed + 1), n), case["m"])
    nev = case["nev"]
    w, x, y = _eigenpairs(a, b, nev)
    if kind == "backward":
        return _gradients(x, y, _weights(case, seed)[0])
    if kind == "train":
        wt, t = (torch.from_numpy(v).cuda() for v in _weights(case, seed))
        return [w, *_gradients(x, y, wt + 2 * (w - t))]
    if kind == "values":
        return w, None
    return w, _fix_phase(x if y is None else torch.cat([x, y])), None


def _haydock(a, b, d, m):
    dot = lambda p, q: float((p.conj() * q).sum().real)                              # noqa: E731
    k = (lambda v: v) if b is None else (lambda v: _half(a, b, -1.0, v))             # inner product
    step = (lambda v: a @ v) if b is None else (lambda v: _half(a, b, 1.0, v))       # the other half, of K q
    kd = k(d)
    norm2 = dot(d, kd)
    q, kq, qp, beta, al, be = d / math.sqrt(norm2), kd / math.sqrt(norm2), torch.zeros_like(d), 0.0, [], []
    for _ in range(m):
        w = step(kq)
        al.append(dot(kq, w))
        r = w - al[-1] * q - beta * qp
        kr = k(r)
        beta = math.sqrt(dot(r, kr))
        be.append(beta)
        qp, q, kq = q, r / beta, kr / beta
    z = np.linspace(1.0, 10.0, 1001) + 0.1j
    zeta = z if b is None else z * z
    cf = np.zeros_like(z)
    for j in reversed(range(m)):
        cf = 1.0 / (zeta - al[j] - (be[j] ** 2 * cf if j + 1 < m else 0.0))
    f = (1.0 if b is None else 2.0) * norm2 * cf
    return -f.imag / math.pi, f, np.array(al), np.array(be[:-1]), np.float64(norm2), None
