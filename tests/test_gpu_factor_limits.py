"""The forms that a factorization falls back to: the Schur update per pair of
clusters (no workspace for a separator's couplings as one block), the apply in
several launches, and the factorization that starts again after device memory ran
out.

With eps = 0 nothing is compressed and M M^T = A^{-1}; A is the grid Laplacian
plus 2 I, condition number at most 7.  Tolerances, fixed beforehand: 20 cond u for
the rounding of the factors and products (u = 2^-53, 2^-24); TF32 operands of the
Schur update add 2 * 2^-11 per step, times cond."""
import numpy as np
import pytest
import scipy.sparse.linalg as sla

from paper_1901_02971_gb300 import Solver
from paper_1901_02971_gb300 import _lib as L
from paper_1901_02971_gb300 import inputs as I

pytestmark = pytest.mark.gpu

COND = 7.0


def _shifted(n):
    p = I.laplacian_3d(n)
    rows = np.repeat(np.arange(p.n), np.diff(p.rowptr))
    p.vals = p.vals + np.where(rows == p.colind, 2.0, 0.0)
    return p


def _tol(precision, levels):
    tf32 = 2 * levels * COND * 2.0 ** -11 if precision == "tf32" else 0.0
    return 20 * COND * 2.0 ** (-53 if precision == "fp64" else -24) + tf32


def _err(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("precision", ["fp64", "fp32", "tf32"])
@pytest.mark.parametrize("n,levels", [(9, 2), (13, 3), (17, 5), (21, 6)])
def test_update_without_workspace(cuda_ok, n, levels, precision):
    """No workspace, and one that only the smaller steps fit in."""
    import torch
    p = _shifted(n)
    r = I.rhs(p.n, 4)
    ref = sla.spsolve(p.to_scipy().tocsc(), r)
    tol = _tol(precision, levels)
    assert tol < 0.1
    s = Solver.from_problem(p, levels=levels, eps=0.0, precision=precision)
    try:
        for limit in (-1, 0, 1 << 17):
            L.spand_set_factor_limits(s.h, limit)
            z = s.factorize().apply(torch.from_numpy(r).cuda()).cpu().numpy()
            assert _err(z, ref) <= tol, limit
    finally:
        s.close()


@pytest.mark.parametrize("precision,skip", [("fp64", 0), ("fp32", 0), ("fp32", 2)])
def test_apply_in_several_launches(cuda_ok, precision, skip):
    import torch
    p = I.diffusion_2d(45, 3)
    r = torch.from_numpy(I.rhs(p.n, 5)).cuda()
    s = Solver.from_problem(p, levels=7, eps=1e-2, skip=skip, precision=precision)
    try:
        z_ref = s.factorize().apply(r).cpu().numpy()
        for phases in (1, 2, 7, 96):
            L.spand_set_factor_limits(s.h, -1, phases)
            assert np.array_equal(s.apply(r).cpu().numpy(), z_ref)  # the present factorization's, still
            assert np.array_equal(s.factorize().apply(r).cpu().numpy(), z_ref), phases
            L.spand_set_apply_shape(s.h, 2)
            assert np.array_equal(s.apply(r).cpu().numpy(), z_ref), phases
    finally:
        s.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32", "tf32"])
@pytest.mark.parametrize("step", [1, 3])
def test_out_of_memory_starts_again(cuda_ok, precision, step):
    import torch
    n, levels = 17, 5
    p = _shifted(n)
    r = I.rhs(p.n, 4)
    rd = torch.from_numpy(r).cuda()
    ref = sla.spsolve(p.to_scipy().tocsc(), r)
    full = Solver.from_problem(p, levels=levels, eps=0.0, precision=precision).factorize()
    s = Solver.from_problem(p, levels=levels, eps=0.0, precision=precision)
    try:
        L.spand_set_factor_fault(s.h, step, L.SPAND_ERR_OOM)
        z = s.factorize().apply(rd).cpu().numpy()
        assert _err(z, ref) <= _tol(precision, levels)
        assert s.stats().device_bytes <= full.stats().device_bytes
        assert s.stats().mem_f == full.stats().mem_f
        assert np.array_equal(s.factorize().apply(rd).cpu().numpy(), z)
        assert s.solve(r)[2] <= 1e-10
    finally:
        s.close()
        full.close()
