"""Workloads of the spaND solver: what a program that uses this package has it do.

A case is one call sequence through the public entry points (Solver, factorize_all / solve_all,
autograd.spand_solve) on a seeded synthetic problem of the shapes the paper evaluates: 2D and 3D
elliptic stencils with constant, log-normal or blockwise 10^U(-3, 3) coefficients, thin extruded
meshes, and k-nearest-neighbour graph Laplacians without coordinates.  The analysis of the pattern is
what a program does once and keeps (prepare); refactorizing with new values and solving is what it
repeats (run).  Solves run to the paper's relative residual, 1e-12, except where the conditioning of
the problem leaves only 1e-11 within reach of FP64 residuals.

Keys of a case:
  call    "factor_solve" (new values, then one right-hand side), "solve" (one right-hand side on a
          kept factorization), "apply" (the preconditioner alone, for a caller's own Krylov loop),
          "grad" (the differentiable solve: forward, and the gradients of a loss in the values and the
          right-hand side), "batch" (k independent problems, factorized and solved together)
  kind    "grid2d", "grid3d", "extruded" (nx, ny[, nz]), "knn" (npts)
  coeff   "const", "lognormal", "blocks" (grids); levels, eps, precision, order: options of Solver
"""
import numpy as np
import torch

from paper_1901_02971_gb300 import Solver, factorize_all, solve_all
from paper_1901_02971_gb300.autograd import spand_solve


# ------------------------------------------------------------------ cases

def _levels(n, dim):
    """Levels giving leaves of about 32 unknowns (2D) or 512 (3D), as the tests and the benchmark have."""
    return max(2, int(round(np.log2(n / (32.0 if dim == 2 else 512.0)))) + 1)


def _grid(name, call, nx, ny, nz, coeff, precision, eps=1e-2, levels=0, order="coloured", tol=1e-12, kind="", count=1):
    dim = 3 if nz > 1 and kind != "extruded" else 2
    case = {"call": call, "kind": kind or ("grid3d" if dim == 3 else "grid2d"), "nx": nx, "ny": ny, "nz": nz,
            "coeff": coeff, "precision": precision, "eps": eps,
            "levels": levels or _levels(nx * ny * (nz if dim == 3 else 1), dim), "order": order, "tol": tol, "count": count}
    return dict(case, name=name) if name else case


def _knn(name, npts, precision="fp32", eps=1e-2):
    case = {"call": "factor_solve", "kind": "knn", "npts": npts, "k": 10, "coeff": "graph", "precision": precision,
            "eps": eps, "levels": max(2, int(round(np.log2(npts / 400.0))) + 1), "order": "coloured", "tol": 1e-11, "count": 1}
    return dict(case, name=name) if name else case


def listed():
    return [
        # a small 2D Poisson problem in the default precision: launch latency (an inner solve of a larger program)
        _grid("lapl2d_64_fp64", "factor_solve", 64, 64, 1, "const", "fp64", levels=8),
        # an odd, small 3D diffusion problem with the options a first-time user leaves alone (FP64, eps 1e-2)
        _grid("diff3d_31x29x27_fp64", "factor_solve", 31, 29, 27, "lognormal", "fp64", levels=8),
        # the benchmark's 64^3 Poisson problem, mixed precision: the ordinary large call
        _grid("lapl3d_64_tf32", "factor_solve", 64, 64, 64, "const", "tf32"),
        # the same size in the plain FP64 form with variable coefficients
        _grid("diff3d_64_fp64", "factor_solve", 64, 64, 64, "lognormal", "fp64"),
        # high-contrast 3D diffusion, the largest: 0.9 M unknowns, FP32 factor
        _grid("contrast3d_96_fp32", "factor_solve", 96, 96, 96, "blocks", "fp32", levels=12, eps=1e-1, tol=1e-11),
        # tighter compression (fewer iterations, larger ranks) on an odd box
        _grid("diff3d_50x43x37_fp32_eps1e-3", "factor_solve", 50, 43, 37, "lognormal", "fp32", eps=1e-3),
        # every interface of a level compressed at once
        _grid("diff3d_48_tf32_simultaneous", "factor_solve", 48, 48, 48, "lognormal", "tf32", order="simultaneous"),
        # an algebraic problem without geometry
        _knn("knn_50k_fp32", 50000),
        # a thin extruded mesh (ice-sheet like), partitioned in the plane
        _grid("extruded_160x144x5_fp32", "factor_solve", 160, 144, 5, "const", "fp32", levels=10, kind="extruded"),
        # time stepping: a new right-hand side on a kept factorization
        _grid("solve_diff3d_64_fp32", "solve", 64, 64, 64, "lognormal", "fp32"),
        # training through the solver: forward, and gradients in the values and the right-hand side
        _grid("grad_diff2d_300x280_fp32", "grad", 300, 280, 1, "lognormal", "fp32", tol=1e-11),
        # a batch of uneven 2D diffusion problems, solved together
        _grid("batch8_diff2d_128to400_fp32", "batch", 128, 400, 1, "lognormal", "fp32", tol=1e-11, count=8, levels=1),
    ]


def draw(rng):
    """Another case of the same ranges: sizes spread over their logarithm, odd ones among them."""
    def size(lo, hi):
        return int(round(lo * (hi / lo) ** rng.random()))

    what = rng.choice(["2d", "2d", "3d", "3d", "3d", "3d", "3d64", "knn", "extruded", "solve", "apply", "grad", "batch", "simultaneous"])
    if what == "knn":
        return _knn("", size(2000, 50000), rng.choice(["fp32", "fp64"]) if rng.random() < 0.3 else "fp32", rng.choice([1e-1, 1e-2]))
    if what == "2d":
        return _grid("", "factor_solve", size(24, 512), size(24, 512), 1, rng.choice(["const", "lognormal"]),
                     rng.choice(["fp64", "fp32", "tf32"]), rng.choice([1e-1, 1e-2, 1e-3]), tol=1e-11)
    if what == "3d":
        p = rng.choice(["fp32", "fp32", "tf32"])
        return _grid("", "factor_solve", size(12, 72), size(12, 72), size(12, 72), rng.choice(["const", "lognormal"]), p,
                     rng.choice([1e-1, 1e-2] if p == "tf32" else [1e-1, 1e-2, 1e-3]))
    if what == "3d64":
        return _grid("", "factor_solve", size(12, 48), size(12, 48), size(12, 48), rng.choice(["const", "lognormal"]), "fp64",
                     rng.choice([1e-1, 1e-2]))
    if what == "extruded":
        return _grid("", "factor_solve", size(32, 192), size(32, 192), rng.randint(3, 8), "const",
                     rng.choice(["fp32", "fp64"]), kind="extruded")
    if what == "solve":
        return _grid("", "solve", size(16, 64), size(16, 64), size(16, 64), "lognormal", rng.choice(["fp32", "fp64"]))
    if what == "apply":
        return _grid("", "apply", size(48, 512), size(48, 512), 1, "lognormal", "fp64")
    if what == "grad":
        return _grid("", "grad", size(48, 400), size(48, 400), 1, "lognormal", rng.choice(["fp32", "fp64"]), tol=1e-11)
    if what == "batch":
        lo = size(32, 128)
        return _grid("", "batch", lo, lo + size(32, 272), 1, "lognormal", "fp32", tol=1e-11, count=rng.randint(2, 8), levels=1)
    return _grid("", "factor_solve", size(16, 56), size(16, 56), size(16, 56), "lognormal", rng.choice(["fp32", "tf32"]),
                 order="simultaneous")


# ------------------------------------------------------------------ problems

def _stencil(shape, cell, scale):
    """CSR (rowptr int64, colind int32, vals float64) of -div(a grad u) on a grid, x fastest: a face carries
    scale[axis] times the harmonic mean of its cells, a Dirichlet face the cell's own value; sorted columns."""
    dim, n = len(shape), int(np.prod(shape))
    ids = np.arange(n, dtype=np.int64).reshape(shape)
    diag, lower, upper = np.zeros(shape), [], []
    for ax in range(dim):  # slowest axis first, so that the entries of a row come out in column order
        s = scale[ax]
        lo, hi = [slice(None)] * dim, [slice(None)] * dim
        lo[ax], hi[ax] = slice(0, -1), slice(1, None)
        lo, hi = tuple(lo), tuple(hi)
        f = s * 2.0 * cell[lo] * cell[hi] / (cell[lo] + cell[hi])
        diag[lo] += f
        diag[hi] += f
        for end in (0, -1):
            at = [slice(None)] * dim
            at[ax] = end
            diag[tuple(at)] += s * cell[tuple(at)]
        step = int(np.prod(shape[ax + 1:]))
        down, up = np.zeros(shape), np.zeros(shape)
        down[hi], up[lo] = -f, -f
        lower.append((-step, down))
        upper.append((step, up))
    parts = lower + [(0, diag)] + upper[::-1]
    v = np.stack([p.reshape(-1) for _, p in parts], 1)
    c = ids.reshape(-1, 1) + np.array([s for s, _ in parts], dtype=np.int64)[None, :]
    keep = v != 0
    rowptr = np.concatenate([[0], np.cumsum(keep.sum(1))]).astype(np.int64)
    return rowptr, c[keep].astype(np.int32), v[keep]


def _cells(shape, coeff, g):
    if coeff == "const":
        return np.ones(shape)
    if coeff == "lognormal":
        return np.exp(g.standard_normal(shape))
    u = g.uniform(-3.0, 3.0, size=[-(-s // 8) for s in shape])  # constant on blocks of 8 cells a side
    for ax in range(len(shape)):
        u = np.repeat(u, 8, ax)
    return 10.0 ** u[tuple(slice(0, s) for s in shape)]


def _smooth_plane(shape, g):
    """A field over six decades varying slowly in the plane: a few random plane waves."""
    y, x = np.meshgrid(np.arange(shape[0]), np.arange(shape[1]), indexing="ij")
    s = sum(a * np.cos(p * x / 20.0 + q * y / 20.0 + t)
            for a, p, q, t in zip(g.random(6), g.standard_normal(6), g.standard_normal(6), g.uniform(0, 6.28, 6)))
    return 10.0 ** (3.0 * (2.0 * (s - s.min()) / (s.max() - s.min()) - 1.0))


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _knn_graph(npts, k, seed):
    """Graph Laplacian + 1e-4 I of the symmetrised k-nearest-neighbour graph of uniform points in the unit
    cube, weights exp(-d^2 / h^2), h the mean distance of the k-th neighbour."""
    pts = torch.from_numpy(np.random.Generator(np.random.PCG64(seed)).random((npts, 3)).astype(np.float32)).to(_device())
    near, dist = [], []
    for i in range(0, npts, 4096):
        q = pts[i:i + 4096]
        d = sum((q[:, a, None] - pts[None, :, a]) ** 2 for a in range(3))
        d[torch.arange(len(q), device=d.device), torch.arange(i, i + len(q), device=d.device)] = float("inf")
        d, j = torch.topk(d, k, dim=1, largest=False)
        near.append(j.cpu().numpy())
        dist.append(d.cpu().numpy().astype(np.float64))
    j, d2 = np.concatenate(near).reshape(-1), np.concatenate(dist)
    h = float(np.mean(np.sqrt(d2[:, -1])))
    i, w = np.repeat(np.arange(npts, dtype=np.int64), k), np.exp(-d2.reshape(-1) / h ** 2)
    key, first = np.unique(np.minimum(i, j) * npts + np.maximum(i, j), return_index=True)
    a, b, w = key // npts, key % npts, w[first]
    deg = np.bincount(a, w, npts) + np.bincount(b, w, npts) + 1e-4
    diag = np.arange(npts, dtype=np.int64)
    key = np.concatenate([a * npts + b, b * npts + a, diag * npts + diag])
    vals = np.concatenate([-w, -w, deg])
    order = np.argsort(key)
    key, vals = key[order], vals[order]
    rowptr = np.concatenate([[0], np.cumsum(np.bincount(key // npts, minlength=npts))]).astype(np.int64)
    return rowptr, (key % npts).astype(np.int32), vals


def _problem(case, seed, shape=None):
    """(rowptr, colind, vals, coords or None) of the case's matrix for this seed."""
    if case["kind"] == "knn":
        return _knn_graph(case["npts"], case["k"], seed) + (None,)
    g = np.random.Generator(np.random.PCG64(seed))
    if case["kind"] == "extruded":  # vertical faces of thin layers are 100 times stronger
        shape = (case["nz"], case["ny"], case["nx"])
        cell, scale = np.broadcast_to(_smooth_plane(shape[1:], g), shape).copy(), (100.0, 1.0, 1.0)
    else:
        shape = shape or ((case["nz"], case["ny"], case["nx"]) if case["kind"] == "grid3d" else (case["ny"], case["nx"]))
        cell, scale = _cells(shape, case["coeff"], g), (1.0,) * len(shape)
    xyz = np.indices(shape).reshape(len(shape), -1)[::-1].T.astype(np.float64)
    return _stencil(shape, cell, scale) + (np.ascontiguousarray(xyz[:, :2] if case["kind"] == "extruded" else xyz),)


def _shapes(case):
    """The grids of a case: one, or those of a batch (uneven squares from nx to ny cells a side)."""
    if case["call"] != "batch":
        return [None]
    k = case["count"]
    return [(n, n) for n in (case["nx"] + (case["ny"] - case["nx"]) * i // max(1, k - 1) for i in range(k))]


def _vector(n, seed, k):
    return torch.from_numpy(np.random.Generator(np.random.PCG64([seed, k])).standard_normal(n))


def prepare(case, seed):
    state = {"call": case["call"], "solvers": [], "vals": [], "b": []}
    for i, shape in enumerate(_shapes(case)):
        rowptr, colind, vals, coords = _problem(case, seed + 1000 * i, shape)
        n = rowptr.size - 1
        levels = case["levels"] if case["call"] != "batch" else _levels(n, 2)
        s = Solver(rowptr, colind, vals, coords, levels=levels, eps=case["eps"], precision=case["precision"], tol=case["tol"],
                   sparsify_order=case["order"])
        state["solvers"].append(s)
        state["vals"].append(torch.from_numpy(vals).cuda())
        state["b"].append(_vector(n, seed, i).cuda())
        if case["call"] == "grad":
            state["y"] = _vector(n, seed, 77).cuda()
        if case["call"] in ("solve", "apply"):
            s.factorize(state["vals"][i])
    return state


def run(state):
    call, s, vals, b = state["call"], state["solvers"][0], state["vals"][0], state["b"][0]
    if call == "factor_solve":
        return s.factorize(vals).solve(b)[0]
    if call == "solve":
        return s.solve(b)[0]
    if call == "apply":
        return s.apply(b)
    if call == "grad":
        vals, b = vals.detach().requires_grad_(), b.detach().requires_grad_()
        x = spand_solve(vals, b, s)
        loss = 0.5 * ((x - state["y"]) ** 2).sum()
        gvals, gb = torch.autograd.grad(loss, (vals, b))
        return {"x": x.detach(), "gvals": gvals, "gb": gb}
    factorize_all(state["solvers"], state["vals"])
    return [x for x, _, _ in solve_all(state["solvers"], state["b"])]


# ------------------------------------------------------------------ 64-bit values and the least work

def _cg(rowptr, colind, vals, b):
    """A^{-1} b in 64 bits: diagonally preconditioned conjugate gradients, restarted on the true residual
    until it no longer falls."""
    dev = _device()
    n = rowptr.size - 1
    A = torch.sparse_csr_tensor(torch.from_numpy(rowptr).to(dev), torch.from_numpy(colind.astype(np.int64)).to(dev),
                                torch.from_numpy(vals).to(dev), size=(n, n))
    rows = np.repeat(np.arange(n), np.diff(rowptr))
    dinv = 1.0 / torch.from_numpy(vals[rows == colind]).to(dev)
    b = b.to(dev)
    x, best, norm = torch.zeros_like(b), float("inf"), float(b.norm())
    for _ in range(6):
        r = b - A @ x
        res = float(r.norm()) / norm
        if res > 0.3 * best or res < 1e-15:
            break
        best, start = res, float(r.norm())
        e, z = torch.zeros_like(b), dinv * r
        p, rz = z.clone(), torch.dot(r, z)
        for it in range(20000):
            q = A @ p
            a = rz / torch.dot(p, q)
            e += a * p
            r -= a * q
            if it % 25 == 0 and float(r.norm()) < 1e-8 * start:
                break
            z = dinv * r
            new = torch.dot(r, z)
            p = z + (new / rz) * p
            rz = new
        x = x + e
    return x


def exact(case, seed):
    if case["call"] == "apply":
        return None  # one application of the preconditioner is no closed expression of A and r
    out = []
    for i, shape in enumerate(_shapes(case)):
        rowptr, colind, vals, _ = _problem(case, seed + 1000 * i, shape)
        n = rowptr.size - 1
        x = _cg(rowptr, colind, vals, _vector(n, seed, i))
        if case["call"] == "grad":
            gb = _cg(rowptr, colind, vals, x.cpu() - _vector(n, seed, 77))
            rows = torch.from_numpy(np.repeat(np.arange(n), np.diff(rowptr))).to(x.device)
            return {"x": x, "gvals": -gb[rows] * x[torch.from_numpy(colind.astype(np.int64)).to(x.device)], "gb": gb}
        out.append(x)
    return out if case["call"] == "batch" else out[0]


def work(case):
    """The matrix, the right-hand side and the solution once; and the elimination of the leaves of the
    dissection alone, s unknowns each of half-bandwidth w with a boundary of a: s w^2 + 2 s w a + s a^2
    (factorizing calls), or the two passes over their factors (calls on a kept factorization)."""
    nbytes = flops = 0.0
    for shape in _shapes(case):
        if case["kind"] == "knn":
            n, d, nnz = case["npts"], 3, case["npts"] * (1.25 * case["k"] + 1)
        else:
            size = shape or [s for s in (case["nx"], case["ny"], case["nz"]) if s > 1]
            n, d = float(np.prod(size)), len(size)
            nnz = n * (2 * d + 1) - 2 * sum(n / s for s in size)
        leaves = 2.0 ** ((case["levels"] if shape is None else _levels(n, 2)) - 1)
        s = n / leaves
        w = s ** ((d - 1.0) / d)
        a = 2 * d * w
        item = 8 if case["precision"] == "fp64" else 4
        factor = leaves * (s * w + s * a)
        nbytes += 16.0 * n
        if case["call"] in ("solve", "apply"):
            nbytes += 2 * factor * item + (12 * nnz if case["call"] == "solve" else 0)
            flops += 4 * factor
        else:
            nbytes += 12.0 * nnz + (16.0 * nnz + 24.0 * n if case["call"] == "grad" else 0)
            flops += leaves * (s * w * w + 2 * s * w * a + s * a * a)
    return {"bytes": nbytes, "flops": flops}
