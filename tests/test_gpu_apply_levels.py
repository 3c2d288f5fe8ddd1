"""The preconditioner apply (spand_apply) on sizes at the edges of its work items.

With eps = 0 nothing is compressed and M M^T = A^{-1}, so z is compared with a
sparse direct solve.  Tolerance, fixed beforehand: the explicit inverse factors
and the products carry rounding errors of a small multiple of cond(A) u
(u = 2^-53 or 2^-24, the factor's unit roundoff); 20 cond(A) u is allowed, with
cond(A) of the grid Laplacian from its known eigenvalues."""
import numpy as np
import pytest
import scipy.sparse.linalg as sla

from paper_1901_02971_gb300 import Solver
from paper_1901_02971_gb300 import inputs as I

pytestmark = pytest.mark.gpu

# (dimension, grid side, levels): a root of 25 unknowns alone; one taller than
# a round of loads; leaves of a few hundred odd-sized rows; leaves beyond 512
# rows; many small clusters that pass through unscaled; a root whose factor is
# large enough for the streaming cut of its items in FP32 (4096 rows) and FP64
CASES = [(2, 5, 1), (2, 31, 1), (3, 9, 2), (3, 12, 2), (2, 33, 6), (3, 17, 6), (3, 16, 1)]


def _cond(dim, n):
    lam = [2 - 2 * np.cos(k * np.pi / (n + 1)) for k in (1, n)]
    return lam[1] / lam[0]  # the dimensions add equally


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("dim,n,levels", CASES)
def test_exact_apply_is_the_inverse(cuda_ok, dim, n, levels, precision):
    import torch
    p = I.laplacian_2d(n) if dim == 2 else I.laplacian_3d(n)
    r = I.rhs(p.n, 3)
    ref = sla.spsolve(p.to_scipy().tocsc(), r)
    s = Solver.from_problem(p, levels=levels, eps=0.0, precision=precision).factorize()
    try:
        z = s.apply(torch.from_numpy(r).cuda()).cpu().numpy()
    finally:
        s.close()
    u = 2.0 ** (-53 if precision == "fp64" else -24)
    err = np.linalg.norm(z - ref) / np.linalg.norm(ref)
    assert err <= 20 * _cond(dim, n) * u, err


@pytest.mark.parametrize("precision", ["fp64", "fp32", "tf32"])
@pytest.mark.parametrize("dim,n,levels,skip", [(2, 33, 6, 5), (3, 13, 5, 2), (3, 17, 4, 3), (2, 65, 4, 0)])
def test_unscaled_steps_and_wide_couplings(cuda_ok, dim, n, levels, skip, precision):
    """skip > 0: the clusters of the first steps pass through the apply unscaled,
    next to scaled ones; couplings of one to several 64-column tiles with ragged
    ends through the elimination's G blocks, the pull and the scaling product.
    TF32 operands of the Schur update carry 2^-11."""
    import torch
    p = I.laplacian_2d(n) if dim == 2 else I.laplacian_3d(n)
    r = I.rhs(p.n, 4)
    ref = sla.spsolve(p.to_scipy().tocsc(), r)
    s = Solver.from_problem(p, levels=levels, eps=0.0, skip=skip, precision=precision).factorize()
    try:
        z = s.apply(torch.from_numpy(r).cuda()).cpu().numpy()
    finally:
        s.close()
    u = 2.0 ** {"fp64": -53, "fp32": -24, "tf32": -11}[precision]
    err = np.linalg.norm(z - ref) / np.linalg.norm(ref)
    assert err <= 20 * _cond(dim, n) * u, err


@pytest.mark.parametrize("precision", ["fp64", "fp32", "tf32"])
@pytest.mark.parametrize("dim,n,levels,skip", [(2, 33, 6, 2), (2, 65, 5, 1), (3, 13, 5, 2), (3, 17, 5, 0), (3, 21, 6, 3)])
def test_unscaled_next_to_scaled_steps(cuda_ok, dim, n, levels, skip, precision):
    """Steps whose clusters pass through unscaled (t <= skip) below scaled ones
    (skip < t < levels), couplings of one to several tiles with ragged ends, on the
    grid Laplacian plus 2 I (condition number at most 5 in 2D, 7 in 3D).  Bound:
    20 cond u for the factors and products; TF32 operands of the Schur update add
    2 * 2^-11 per step, times cond: at most 0.05, so that a missing or misplaced
    contribution shows."""
    import torch
    assert skip + 1 < levels
    p = I.laplacian_2d(n) if dim == 2 else I.laplacian_3d(n)
    rows = np.repeat(np.arange(p.n), np.diff(p.rowptr))
    p.vals = p.vals + np.where(rows == p.colind, 2.0, 0.0)
    r = I.rhs(p.n, 4)
    ref = sla.spsolve(p.to_scipy().tocsc(), r)
    s = Solver.from_problem(p, levels=levels, eps=0.0, skip=skip, precision=precision).factorize()
    try:
        z = s.apply(torch.from_numpy(r).cuda()).cpu().numpy()
    finally:
        s.close()
    cond = 1.0 + 2.0 * dim
    tol = 20 * cond * 2.0 ** (-53 if precision == "fp64" else -24)
    if precision == "tf32":
        tol += 2 * levels * cond * 2.0 ** -11
    assert tol < 0.1
    err = np.linalg.norm(z - ref) / np.linalg.norm(ref)
    assert err <= tol, err
