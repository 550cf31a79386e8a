"""The work a user of this package has it do, as cases that can be timed.

The products with a polynomial of a sparse matrix (``apply_poly``, ``apply_phi``), the plain product (``spmv``), the
construction of the polynomial (``build_poly``) and the solves around them (``solve``, ``solve_flex``, ``solve_batched``,
``PPGMRESFunction``), over the sizes the package is run at: 2-D grids of 50^2 to 1000^2 nodes, 3-D grids of up to 160^3, FP64
and FP32, matrices with one stencil everywhere, with coefficients that change from node to node, and with rows of
irregular length.

A case is a dict: ``call`` (which entry point), ``matrix`` ("const", "field" or "mesh"), ``nx``, ``ny``, ``nz`` (grid sides;
``nz`` = 1 in two dimensions; a "mesh" has nx * ny rows), ``dtype``, ``d`` (degree), and for solves ``m`` and ``tol``.
"""
import math

import numpy as np
import torch

import paper_1911_07065_gb300 as ppg

DEV = "cuda"
F64 = torch.float64


def listed():
    return [
        # the smallest call: one preconditioner application to a system of a few thousand unknowns, all launch latency
        {"name": "p_2d_50", "call": "p", "matrix": "const", "nx": 50, "ny": 50, "nz": 1, "dtype": "f64", "d": 10},
        # the operator of the outer Arnoldi step on a matrix that fits in L2
        {"name": "phi_2d_1000", "call": "phi", "matrix": "const", "nx": 1000, "ny": 1000, "nz": 1, "dtype": "f64", "d": 40},
        # the FP32 preconditioner of the precision form, on a matrix far larger than L2
        {"name": "p_3d_160_f32", "call": "p", "matrix": "const", "nx": 160, "ny": 160, "nz": 160, "dtype": "f32", "d": 60},
        # the same operator with coefficients of its own in every row and odd grid sides, in FP64
        {"name": "phi_3d_field", "call": "phi", "matrix": "field", "nx": 127, "ny": 131, "nz": 113, "dtype": "f64", "d": 60},
        # a matrix with no grid behind it: rows of 1 to 12 entries and a few of thousands
        {"name": "p_mesh", "call": "p", "matrix": "mesh", "nx": 449, "ny": 443, "nz": 1, "dtype": "f64", "d": 20},
        # one product y = A x, as a caller's own Krylov method or residual check asks for it
        {"name": "spmv_3d_160", "call": "spmv", "matrix": "const", "nx": 160, "ny": 160, "nz": 160, "dtype": "f64", "d": 1},
        # the construction of a polynomial: d Arnoldi steps, orthogonalisation above all
        {"name": "build_3d_101", "call": "build", "matrix": "const", "nx": 101, "ny": 101, "nz": 101, "dtype": "f64", "d": 60},
        # whole calls: construction and solve of a small system and of the workload the benchmark reports
        {"name": "solve_2d_50", "call": "solve", "matrix": "const", "nx": 50, "ny": 50, "nz": 1, "dtype": "f64", "d": 10, "m": 50, "tol": 1e-8},
        {"name": "solve_2d_1000", "call": "solve", "matrix": "const", "nx": 1000, "ny": 1000, "nz": 1, "dtype": "f64", "d": 40, "m": 50, "tol": 1e-10},
        # the precision form: FGMRES in FP64 around the FP32 polynomial
        {"name": "flex_3d_160", "call": "flex", "matrix": "const", "nx": 160, "ny": 160, "nz": 160, "dtype": "f64", "d": 60, "m": 50, "tol": 1e-10},
        # many systems of mixed sizes with four right-hand sides each in one call
        {"name": "batch_64x4", "call": "batch", "matrix": "const", "nx": 64, "ny": 512, "nz": 1, "dtype": "f64", "d": 20, "m": 30, "tol": 1e-10, "nsys": 64, "nrhs": 4},
        # a training step through a solve: x = A(vals)^-1 b and its gradients for b and for the matrix values
        {"name": "adjoint_512", "call": "adjoint", "matrix": "field", "nx": 512, "ny": 512, "nz": 1, "dtype": "f64", "d": 30, "m": 50, "tol": 1e-10},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["p", "p", "phi", "phi", "spmv", "build", "solve", "flex", "batch", "adjoint"])
    matrix = rng.choice(["const", "field", "mesh"]) if call in ("p", "phi", "spmv", "build") else rng.choice(["const", "field"])
    if call == "batch":
        lo = _log_int(rng, 40, 160)
        return {"call": call, "matrix": "const", "nx": lo, "ny": lo + rng.randint(1, 240), "nz": 1, "dtype": "f64", "d": rng.randint(10, 24), "m": 30,
                "tol": 1e-10, "nsys": _log_int(rng, 2, 24), "nrhs": rng.choice([1, 4])}
    three = matrix != "mesh" and call != "adjoint" and rng.random() < (1.0 if call == "flex" else 0.5)
    if three:
        n = _log_int(rng, 3000, 160 ** 3)
        nx = min(400, max(8, int(round(n ** (1 / 3) * rng.uniform(0.7, 1.4)))))
        ny = min(400, max(8, int(round(math.sqrt(n / nx) * rng.uniform(0.8, 1.25)))))
        nz = min(400, max(8, n // (nx * ny)))
    else:
        n = _log_int(rng, 1500, 250000 if matrix == "mesh" else 1000000)
        nx = max(30, int(round(math.sqrt(n) * rng.uniform(0.7, 1.4))))
        ny, nz = max(30, n // nx), 1
    case = {"call": call, "matrix": matrix, "nx": nx, "ny": ny, "nz": nz, "dtype": "f64", "d": rng.randint(8, 60)}
    if call in ("p", "phi", "spmv"):
        case["dtype"] = rng.choice(["f64", "f32"])
    if matrix == "mesh":
        case["d"] = rng.randint(8, 24)
    if call in ("solve", "flex", "adjoint"):
        case["d"] = rng.randint(10, 50)
        case["m"] = 50
        case["tol"] = rng.choice([1e-8, 1e-10])
    return case


# ---------------------------------------------------------------------------
# matrices, in CSR on the GPU
# ---------------------------------------------------------------------------


def _smooth(shape, g, modes=6):
    """A smooth random field on the grid nodes, largest magnitude 1 (``shape``: sides, x first)."""
    f = torch.zeros((), dtype=F64)
    for k in range(modes):
        term = torch.ones((), dtype=F64)
        for axis, n in enumerate(shape):
            phase = 2 * math.pi * float(torch.rand((), generator=g))
            wave = torch.cos(2 * math.pi * float(torch.randint(0, 4, (), generator=g)) * (torch.arange(n, dtype=F64) + 1) / (n + 1) + phase)
            term = term * wave.reshape([n if a == axis else 1 for a in range(len(shape))])
        f = f + float(torch.randn((), generator=g)) / (1 + k) * term
    # rows run with x fastest
    f = f.to(DEV).permute(*reversed(range(len(shape)))).reshape(-1)
    return f / f.abs().max()


def _stencil(shape, cells):
    """-lap u + beta . grad u on a grid (x fastest), scaled by h^2; ``cells``: beta * h per direction, a number or one per node."""
    n = math.prod(shape)
    idx = torch.arange(n, device=DEV)
    stride, lower, upper = 1, [], []
    for axis, side in enumerate(shape):
        c = torch.as_tensor(cells[axis], dtype=F64, device=DEV) / 2
        at = (idx // stride) % side
        lower.append((-stride, at > 0, -1 - c))
        upper.append((stride, at < side - 1, -1 + c))
        stride *= side
    whole = torch.ones(n, dtype=torch.bool, device=DEV)
    entries = lower[::-1] + [(0, whole, torch.tensor(2.0 * len(shape), dtype=F64, device=DEV))] + upper
    valid = torch.stack([v for _, v, _ in entries], 1)
    cols = torch.stack([idx + o for o, _, _ in entries], 1)[valid].to(torch.int32)
    vals = torch.stack([w.expand(n) for _, _, w in entries], 1)[valid]
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    rowptr[1:] = torch.cumsum(valid.sum(1), 0)
    return rowptr.to(torch.int32), cols, vals.contiguous()


def _mesh(n, g):
    """Rows of 1 to 12 entries scattered within some hundred columns of the diagonal, one row in 50,000 with 2,500 anywhere."""
    lens = torch.randint(0, 12, (n,), generator=g)
    lens[:: 50000] = min(2500, n // 2)
    lens = lens.to(DEV)
    row = torch.repeat_interleave(torch.arange(n, device=DEV), lens)
    total = int(lens.sum())
    far = torch.rand(total, generator=g).to(DEV, F64)
    band = 4.0 * math.sqrt(n)
    near = (row + ((far - 0.5) * 2 * band).round().long()).clamp(0, n - 1)
    col = torch.where(lens[row] > 12, (far * n).long().clamp(max=n - 1), near)
    key = torch.unique(torch.cat([row * n + col, torch.arange(n, device=DEV) * (n + 1)]))
    row, col = key // n, key % n
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    rowptr[1:] = torch.cumsum(torch.bincount(row, minlength=n), 0)
    vals = 0.1 * torch.randn(key.numel(), generator=g).to(DEV, F64)
    long = (rowptr[1:] - rowptr[:-1])[row] > 100
    vals = torch.where(long, 0.1 * vals, vals)
    vals[row == col] = 4.0
    return rowptr.to(torch.int32), col.to(torch.int32), vals


def _shape(case):
    return (case["nx"], case["ny"]) if case["nz"] == 1 else (case["nx"], case["ny"], case["nz"])


def _cells(case, shape, g):
    if case["matrix"] == "field":
        return [b * (1 + 0.5 * _smooth(shape, g)) for b in (1.0, 0.4, 0.2)[: len(shape)]]
    return (1.0, 0.0) if len(shape) == 2 else (0.8, 0.4, 0.2)


def _matrix(case, seed, shape=None):
    g = torch.Generator().manual_seed(seed)
    shape = shape or _shape(case)
    if case["matrix"] == "mesh":
        return _mesh(math.prod(shape), g)
    return _stencil(shape, _cells(case, shape, g))


def _csr(case, seed):
    rp, ci, va = _matrix(case, seed)
    return ppg.CSR(rp, ci, va.to(torch.float32) if case["dtype"] == "f32" else va)


def _vector(n, seed, kind, dtype=F64):
    g = torch.Generator(device=DEV).manual_seed(seed)
    v = torch.rand(n, generator=g, device=DEV, dtype=F64) * 2 - 1 if kind == "uniform" else torch.randn(n, generator=g, device=DEV, dtype=F64)
    return v.to(dtype)


# ---------------------------------------------------------------------------
# a polynomial's roots, for the calls that are given one: the harmonic Ritz values of GMRES(d) on a small version of the matrix
# ---------------------------------------------------------------------------


def _dense(rp, ci, va):
    n = rp.numel() - 1
    rp, ci, va = rp.cpu().numpy(), ci.cpu().numpy(), va.cpu().numpy()
    A = np.zeros((n, n))
    A[np.repeat(np.arange(n), np.diff(rp)), ci] = va
    return A


def _leja(t):
    """Modified Leja order: largest modulus first, conjugates side by side."""
    t = [z for z in t if z.imag >= 0]
    order, score = [], [math.log(abs(z)) for z in t]
    while t:
        k = int(np.argmax(score))
        z = t.pop(k)
        score.pop(k)
        if not order:
            score = [0.0] * len(t)
        for w in ([z] if z.imag == 0 else [z, z.conjugate()]):
            order.append(w)
            score = [s + math.log(max(abs(u - w), 1e-300)) for s, u in zip(score, t)]
    return np.array(order, dtype=np.complex128)


def _roots(case, seed):
    shape = _shape(case)
    small = tuple(min(s, 36 if len(shape) == 2 else 12) for s in shape)
    A = _dense(*_matrix(case, seed, small))
    d = case["d"]
    v = np.random.default_rng(seed).standard_normal(A.shape[0])
    V = np.zeros((A.shape[0], d + 1))
    H = np.zeros((d + 1, d))
    V[:, 0] = v / np.linalg.norm(v)
    for j in range(d):
        w = A @ V[:, j]
        for _ in range(2):
            h = V[:, : j + 1].T @ w
            w -= V[:, : j + 1] @ h
            H[: j + 1, j] += h
        H[j + 1, j] = np.linalg.norm(w)
        V[:, j + 1] = w / H[j + 1, j]
    f = np.linalg.solve(H[:d].T, np.eye(d)[:, d - 1])
    M = H[:d].copy()
    M[:, d - 1] += H[d, d - 1] ** 2 * f
    t = np.linalg.eigvals(M)
    t[np.abs(t.imag) < 1e-13 * np.abs(t)] = t[np.abs(t.imag) < 1e-13 * np.abs(t)].real
    return _leja(list(t))


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------


def _batch_specs(case, seed):
    r = np.random.default_rng(seed)
    lo, hi = case["nx"], case["ny"]
    return [(int(r.integers(lo, hi + 1)), float(r.uniform(0.1, 2.0))) for _ in range(case["nsys"])]


def prepare(case, seed):
    call = case["call"]
    if call == "batch":
        As, Bs, v0s = [], [], []
        # the sizes are the workload's own; the seed draws the data
        for i, (side, bh) in enumerate(_batch_specs(case, 104)):
            As.append(ppg.CSR(*_stencil((side, side), (bh, 0.0))))
            Bs.append(_vector(case["nrhs"] * side * side, 1000 * seed + i, "uniform").reshape(case["nrhs"], -1))
            v0s.append(_vector(side * side, 1000 * seed + 500 + i, "normal"))
        return {"case": case, "As": As, "Bs": Bs, "v0s": v0s}
    A = _csr(case, seed)
    s = {"case": case, "A": A}
    if call in ("p", "phi"):
        s["roots"] = ppg.Roots.from_complex(_roots(case, seed))
    if call in ("p", "phi", "spmv"):
        s["v"] = _vector(A.n, seed, "uniform", A.dtype)
    if call in ("build", "solve"):
        s["v0"] = _vector(A.n, seed + 1, "normal")
    if call in ("solve", "flex", "adjoint"):
        s["b"] = _vector(A.n, seed, "uniform")
    if call in ("flex", "adjoint"):
        s["roots"] = ppg.build_poly(A, case["d"], _vector(A.n, seed + 1, "normal"))
    if call == "flex":
        s["A32"] = A.astype(torch.float32)
    if call == "adjoint":
        s["b"].requires_grad_(True)
        s["vals"] = A.vals.clone().requires_grad_(True)
        s["target"] = _vector(A.n, seed + 2, "normal")
    return s


def run(s):
    c = s["case"]
    call = c["call"]
    if call == "p":
        return ppg.apply_poly(s["A"], s["roots"], s["v"])
    if call == "phi":
        return ppg.apply_phi(s["A"], s["roots"], s["v"])
    if call == "spmv":
        return ppg.spmv(s["A"], s["v"])
    if call == "build":
        roots, H = ppg.build_poly(s["A"], c["d"], s["v0"], return_hbar=True)
        return {"hbar": H, "re": roots.complex().real, "im": roots.complex().imag}
    if call == "solve":
        roots = ppg.build_poly(s["A"], c["d"], s["v0"])
        x, _ = ppg.solve(s["A"], s["b"], c["m"], c["tol"], roots=roots)
        return x
    if call == "flex":
        x, _ = ppg.solve_flex(s["A"], s["A32"], s["b"], s["roots"], c["m"], c["tol"])
        return x
    if call == "batch":
        X, _ = ppg.solve_batched(s["As"], s["Bs"], s["v0s"], d=c["d"], m=c["m"], tol=c["tol"])
        return torch.cat([x.reshape(-1) for x in X])
    x = ppg.PPGMRESFunction.apply(s["b"], s["vals"], s["A"], s["roots"], c["m"], c["tol"], None)
    loss = 0.5 * (x - s["target"]).square().sum()
    gb, gv = torch.autograd.grad(loss, (s["b"], s["vals"]))
    return {"x": x, "grad_b": gb, "grad_vals": gv}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------


def _size(case):
    n = math.prod(_shape(case))
    nnz = (6.5 if case["matrix"] == "mesh" else 5 if case["nz"] == 1 else 7) * n
    return n, nnz


def work(case):
    """The matrix and the vectors of the call read and written once; two operations for each entry of the matrix and product.

    Solves are counted at ten outer steps, which no listed or drawn one undercuts by much; more are the method's own."""
    call, d = case["call"], case["d"]
    e = 4 if case["dtype"] == "f32" else 8
    if call == "batch":
        n = sum(s * s for s, _ in _batch_specs(case, 104))
        r = case["nrhs"]
        return {"bytes": n * (5 * 12 + 4 + 16 * r), "flops": n * (10.0 * d + 2.0 * d * d + r * 10 * (10.0 * d + 80))}
    n, nnz = _size(case)
    mat = nnz * (e + 4) + 4 * (n + 1)
    if call == "spmv":
        return {"bytes": mat + 2 * e * n, "flops": 2 * nnz}
    if call in ("p", "phi"):
        return {"bytes": mat + 2 * e * n, "flops": d * (2 * nnz + 2 * n)}
    # Arnoldi's two passes of Gram-Schmidt: 8 n operations for each pair of basis vectors
    build = d * 2 * nnz + 4.0 * n * d * (d + 1)
    steps = 10 * d * (2 * nnz + 2 * n) + 4.0 * n * 10 * 11
    if call == "build":
        return {"bytes": mat + 8 * n, "flops": build}
    if call == "solve":
        return {"bytes": mat + 24 * n, "flops": build + steps}
    if call == "flex":
        return {"bytes": mat + 4 * nnz + 16 * n, "flops": steps}
    return {"bytes": mat + 8 * nnz + 40 * n, "flops": 2 * steps}


# ---------------------------------------------------------------------------
# the same in plain torch, in 64 bits
# ---------------------------------------------------------------------------


def _product(rp, ci, va, transposed=False):
    n = rp.numel() - 1
    row = torch.repeat_interleave(torch.arange(n, device=DEV), (rp[1:] - rp[:-1]).long())
    row, col = (ci.long(), row) if transposed else (row, ci.long())

    def times(x):
        return torch.zeros(n, dtype=x.dtype, device=DEV).index_add_(0, row, va * x[col])
    return times


def _exact_poly(A, theta, v, phi):
    """pi(A) v factor by factor, a conjugate pair in one; p(A) v = sum of the partial products over the roots."""
    prod, p, i = v.clone(), torch.zeros_like(v), 0
    while i < len(theta):
        a, b = theta[i].real, theta[i].imag
        if b == 0:
            p = p + prod / a
            prod = prod - A(prod) / a
            i += 1
        else:
            t = 2 * a * prod - A(prod)
            p = p + t / (a * a + b * b)
            prod = prod - A(t) / (a * a + b * b)
            i += 2
    return v - prod if phi else p


def _solve_const(shape, cells, b):
    """A^-1 b for one 2-D stencil everywhere with no convection in y: sines in y, a tridiagonal solve in x."""
    nx, ny = shape
    k = torch.arange(1, ny + 1, device=DEV, dtype=F64)
    S = torch.sin(math.pi * k[:, None] * k[None, :] / (ny + 1)) * math.sqrt(2 / (ny + 1))
    f = (S @ b.reshape(ny, nx)).T.contiguous()
    c = cells[0] / 2
    lo, up, diag = -1 - c, -1 + c, 4 - 2 * torch.cos(math.pi * k / (ny + 1))
    cp = torch.empty_like(f)
    prev_c = prev_f = torch.zeros((), dtype=F64, device=DEV)
    for i in range(nx):
        den = diag - lo * prev_c
        cp[i] = up / den
        f[i] = (f[i] - lo * prev_f) / den
        prev_c, prev_f = cp[i], f[i]
    for i in range(nx - 2, -1, -1):
        f[i] -= cp[i] * f[i + 1]
    return (S @ f.T).reshape(-1)


def _solve_iter(A, b, rounds=4):
    """A^-1 b by BiCGSTAB and iterative refinement, to the last bits that 64 of them hold; None where it does not converge."""
    x = torch.zeros_like(b)
    for _ in range(rounds):
        r = b - A(x)
        if float(r.norm()) <= 2e-15 * float(b.norm()):
            break
        start, e = float(r.norm()), torch.zeros_like(b)
        hat, rho, alpha, omega = r.clone(), 1.0, 1.0, 1.0
        v = p = torch.zeros_like(b)
        for _ in range(6000):
            rho, old = torch.dot(hat, r), rho
            p = r + (rho / old) * (alpha / omega) * (p - omega * v)
            v = A(p)
            alpha = rho / torch.dot(hat, v)
            t = r - alpha * v
            w = A(t)
            omega = torch.dot(w, t) / torch.dot(w, w)
            e = e + alpha * p + omega * t
            r = t - omega * w
            if float(r.norm()) <= 1e-9 * start:
                break
        x = x + e
    return x if float((b - A(x)).norm()) <= 1e-13 * float(b.norm()) else None


def exact(case, seed):
    call = case["call"]
    if call == "batch":
        out = []
        for i, (side, bh) in enumerate(_batch_specs(case, 104)):
            B = _vector(case["nrhs"] * side * side, 1000 * seed + i, "uniform").reshape(case["nrhs"], -1)
            out += [_solve_const((side, side), (bh, 0.0), row) for row in B]
        return torch.cat(out)
    n = math.prod(_shape(case))
    if call in ("solve", "flex") and case["matrix"] == "const" and case["nz"] == 1:
        return _solve_const(_shape(case), _cells(case, _shape(case), None), _vector(n, seed, "uniform"))
    rp, ci, va = _matrix(case, seed)
    dtype = torch.float32 if case["dtype"] == "f32" else F64
    A = _product(rp, ci, va.to(dtype).to(F64))
    if call in ("p", "phi", "spmv"):
        v = _vector(n, seed, "uniform", dtype).to(F64)
        return A(v) if call == "spmv" else _exact_poly(A, _roots(case, seed), v, call == "phi")
    if call in ("solve", "flex"):
        return _solve_iter(A, _vector(n, seed, "uniform"))
    if call == "adjoint":
        x = _solve_iter(A, _vector(n, seed, "uniform"))
        row = torch.repeat_interleave(torch.arange(n, device=DEV), (rp[1:] - rp[:-1]).long())
        lam = None if x is None else _solve_iter(_product(rp, ci, va, transposed=True), x - _vector(n, seed + 2, "normal"))
        return None if lam is None else {"x": x, "grad_b": lam, "grad_vals": -lam[row] * x[ci.long()]}
    d = case["d"]
    v = _vector(n, seed + 1, "normal")
    V = torch.zeros(d + 1, n, dtype=F64, device=DEV)
    H = torch.zeros(d + 1, d, dtype=F64, device=DEV)
    V[0] = v / v.norm()
    for j in range(d):
        w = A(V[j])
        for _ in range(2):
            h = V[: j + 1] @ w
            w = w - h @ V[: j + 1]
            H[: j + 1, j] += h
        H[j + 1, j] = w.norm()
        V[j + 1] = w / H[j + 1, j]
    return {"hbar": H, "re": None, "im": None}
