"""The sparsification QR at the ends of the number range: couplings so weak that
the squared column norms are subnormal (their reciprocal overflows), where the
factorization has to stay finite and the preconditioned solve to converge at
once (the system is diagonal to working precision), and a NaN among the values,
which has to end in an error and not in a finite result."""
import numpy as np
import pytest

from paper_1901_02971_gb300 import Solver, SpandError
from paper_1901_02971_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,levels", [(12, 2), (16, 3), (21, 6)])
@pytest.mark.parametrize("scale", [1e-155, 1e-158, 3e-161])
def test_subnormal_norms(cuda_ok, n, levels, scale):
    import torch
    p = I.laplacian_3d(n)
    rows = np.repeat(np.arange(p.n), np.diff(p.rowptr))
    off = rows != p.colind
    p.vals = np.where(off, p.vals * scale, p.vals)
    s = Solver.from_problem(p, levels=levels, eps=1e-2, precision="fp64").factorize()
    try:
        r = I.rhs(p.n, 5)
        x, it, rr = s.solve(torch.from_numpy(r).cuda())
        x = x.cpu().numpy()
    finally:
        s.close()
    d = p.vals[~off]
    # two roundings of each scaled diagonal and one product each way
    assert np.abs(x * d - r).max() <= 1e-13 * np.abs(r).max()
    assert it <= 2


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_nan_is_an_error(cuda_ok, precision):
    p = I.laplacian_3d(16)
    rows = np.repeat(np.arange(p.n), np.diff(p.rowptr))
    off = np.flatnonzero(rows != p.colind)
    p.vals = p.vals.copy()
    p.vals[off[:: max(1, off.size // 7)]] = np.nan
    with pytest.raises(SpandError):
        s = Solver.from_problem(p, levels=3, eps=1e-2, precision=precision)
        try:
            s.factorize()
        finally:
            s.close()


@pytest.mark.parametrize("order", ["coloured", "simultaneous"])
@pytest.mark.parametrize("n,levels", [(12, 2), (16, 3), (21, 6)])
@pytest.mark.parametrize("scale", [1e-13, 1e-16, 1e-18, 1e-19, 1e-20, 1e-22, 1e-24])
def test_weak_couplings_fp32(cuda_ok, n, levels, scale, order):
    """FP32 factors: squared column norms from 1e-27 down to beyond the subnormals.
    The preconditioner is the inverse to FP32's precision, so the solve takes two
    or three iterations to 1e-12."""
    import torch
    p = I.laplacian_3d(n)
    rows = np.repeat(np.arange(p.n), np.diff(p.rowptr))
    off = rows != p.colind
    p.vals = np.where(off, p.vals * scale, p.vals)
    s = Solver.from_problem(p, levels=levels, eps=1e-2, tol=1e-12, precision="fp32", sparsify_order=order).factorize()
    try:
        r = I.rhs(p.n, 5)
        x, it, rr = s.solve(torch.from_numpy(r).cuda())
        x = x.cpu().numpy()
    finally:
        s.close()
    assert rr <= 1e-12 and it <= 3
    # the residual of the stopping test, and the couplings themselves
    assert np.abs(x * p.vals[~off] - r).max() <= 2e-12 * np.linalg.norm(r)
