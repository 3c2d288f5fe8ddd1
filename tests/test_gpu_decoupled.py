"""Systems whose pattern holds stored zeros, so that interfaces have nothing (or
nothing left) to be compressed against: some are cut to rank 0, and those whose
neighbours are all gone are kept whole, wider than their coupling.  x is compared
with a sparse direct solve; with the preconditioner exact up to the factor's
precision, the solve takes a few iterations.  Tolerance: the solve stops at a
relative residual of 1e-12 and the condition numbers here are below 1e3."""
import numpy as np
import pytest
import scipy.sparse.linalg as sla

from oracle import spand_oracle as O
from paper_1901_02971_gb300 import Solver
from paper_1901_02971_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _problem(dim, n, part):
    """The grid Laplacian with stored zeros in place of the couplings of every
    unknown ("all") or of those in the lower half of the first coordinate."""
    p = I.laplacian_2d(n) if dim == 2 else I.laplacian_3d(n)
    rows = np.repeat(np.arange(p.n), np.diff(p.rowptr))
    off = rows != p.colind
    if part == "half":
        low = np.asarray(p.coords)[:, 0] < n // 2
        off &= low[rows] | low[p.colind]
    p.vals = np.where(off, 0.0, p.vals)
    return p


@pytest.mark.parametrize("part", ["all", "half"])
@pytest.mark.parametrize("form", ["coloured", "simultaneous", "InS", "In"])
@pytest.mark.parametrize("precision", ["fp64", "fp32", "tf32"])
@pytest.mark.parametrize("dim,n,levels", [(2, 33, 6), (3, 16, 4), (3, 21, 6)])
def test_decoupled_interfaces(cuda_ok, dim, n, levels, precision, form, part):
    import torch
    p = _problem(dim, n, part)
    b = I.rhs(p.n, 6)
    ref = sla.spsolve(p.to_scipy().tocsc(), b)
    s = Solver.from_problem(p, levels=levels, eps=1e-3, tol=1e-12, precision=precision,
                            **{"variant" if form in ("InS", "In") else "sparsify_order": form})
    try:
        s.factorize()
        x, it, rr = s.solve(torch.from_numpy(b).cuda())
        x = x.cpu().numpy()
    finally:
        s.close()
    assert rr <= 1e-12 and it <= (3 if part == "all" else 20)
    assert np.linalg.norm(x - ref) <= 1e-9 * np.linalg.norm(ref)


@pytest.mark.parametrize("part", ["all", "half"])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("dim,n,levels", [(2, 33, 6), (3, 16, 4)])
def test_decoupled_interfaces_randomized(cuda_ok, dim, n, levels, precision, part):
    """The sketch of a zero coupling is zero; its basis is then the identity's
    columns (none of the rule's thresholds is met, so nothing is dropped), not
    what the device memory held before.  Ranks equal to the oracle's in FP64."""
    import torch
    p = _problem(dim, n, part)
    b = I.rhs(p.n, 6)
    ref = sla.spsolve(p.to_scipy().tocsc(), b)
    s = Solver.from_problem(p, levels=levels, eps=1e-3, tol=1e-12, precision=precision, compression="randomized")
    try:
        for size in (1 << 20, 1 << 24, 1 << 28):  # memory that was used before, and holds NaN
            used = [torch.full((size // 8,), float("nan"), dtype=torch.float64, device="cuda") for _ in range(64 if size < 1 << 28 else 4)]
            del used
        torch.cuda.empty_cache()
        s.factorize(p.vals)
        ranks = [s.ranks(t)[1] for t in range(1, levels + 1)]
        x, it, rr = s.solve(torch.from_numpy(b).cuda())
        x = x.cpu().numpy()
    finally:
        s.close()
    assert rr <= 1e-12 and it <= (3 if part == "all" else 20)
    assert np.linalg.norm(x - ref) <= 1e-9 * np.linalg.norm(ref)
    if precision == "fp64":
        tree = O.analyze(p.n, p.rowptr, p.colind, p.coords, levels)
        F = O.factorize(p.rowptr, p.colind, p.vals, tree, 1e-3, variant="OrthS-rand",
                        sketch=lambda t, c, m, ell: O.sketch_philox(0, t, c, m, ell))
        for t in range(1, levels + 1):
            assert np.array_equal(ranks[t - 1], F.sizes_after[t - 1]), t


@pytest.mark.parametrize("part", ["all", "half"])
def test_tall_interfaces(cuda_ok, part):
    """Interfaces of 578 dofs, beyond the 512 that the basis kernel holds in
    registers, with and without columns to be compressed against."""
    import torch
    p = _problem(3, 34, part)
    s = Solver.from_problem(p, levels=3, eps=1e-3, tol=1e-12, precision="fp32")
    try:
        s.factorize()
        before, after = s.ranks(1)
        tall = np.asarray(before)[np.asarray(s.step(1)["elim"]) == 0].max()
        assert tall > 512
        if part == "all":
            assert np.asarray(after).max() == tall  # kept whole
        x, it, rr = s.solve(torch.from_numpy(I.rhs(p.n, 6)).cuda())
    finally:
        s.close()
    assert rr <= 1e-12 and it <= (3 if part == "all" else 20)
