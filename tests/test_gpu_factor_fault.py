"""A factorization that fails on the host while its kernels are queued
(spand_set_factor_fault): the call returns the error with nothing left running,
and the handle factorizes again at once, on another stream, to the same bits as a
handle that never failed."""
import numpy as np
import pytest

from paper_1901_02971_gb300 import Solver, SpandError
from paper_1901_02971_gb300 import _lib as L
from paper_1901_02971_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [{"precision": "fp64"}, {"precision": "tf32"}, {"precision": "fp32", "skip": 2},
                                {"precision": "fp32", "sparsify_order": "simultaneous"},
                                {"precision": "fp64", "compression": "randomized"},
                                {"precision": "fp64", "variant": "InS"}], ids=lambda kw: "-".join(map(str, kw.values())))
def test_failure_with_work_queued_then_refactorize(cuda_ok, kw):
    import torch
    p, q = I.diffusion_3d(24, 3, block=4, lo=-0.5, hi=0.5), I.diffusion_3d(24, 4, block=4, lo=-0.5, hi=0.5)
    r = torch.from_numpy(I.rhs(p.n, 5)).cuda()
    ref = Solver.from_problem(p, levels=7, eps=1e-2, **kw).factorize()
    s = Solver.from_problem(q, levels=7, eps=1e-2, **kw)
    vals = torch.from_numpy(p.vals).cuda()
    streams = [torch.cuda.Stream() for _ in range(2)]
    torch.cuda.synchronize()
    try:
        z_ref = ref.apply(r).cpu().numpy()
        for step in (1, 2, 4, 7):
            L.spand_set_factor_fault(s.h, step, L.SPAND_ERR_TIMEOUT)
            with pytest.raises(SpandError) as ei:
                s.factorize(stream=streams[0].cuda_stream)  # q's values
            assert ei.value.code == L.SPAND_ERR_TIMEOUT
            assert streams[0].query()  # nothing left running
            with pytest.raises(SpandError) as ei:
                s.apply(r)
            assert ei.value.code == L.SPAND_ERR_STATE
            s.factorize(vals, stream=streams[1].cuda_stream)
            assert np.array_equal(s.apply(r).cpu().numpy(), z_ref), step
            s.factorize(q.vals)  # q's values again for the next failure
    finally:
        s.close()
        ref.close()


def test_closing_after_a_failure(cuda_ok):
    import torch
    p = I.laplacian_3d(24)
    for step in (1, 3):
        s = Solver.from_problem(p, levels=7, eps=1e-2)
        L.spand_set_factor_fault(s.h, step, L.SPAND_ERR_STATE)
        with pytest.raises(SpandError):
            s.factorize()
        s.close()
    torch.cuda.synchronize()
