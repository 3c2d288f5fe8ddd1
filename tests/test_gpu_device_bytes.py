"""spand_stats.device_bytes against the device memory that a handle takes: its
buffers are a few dozen allocations, each rounded up by the driver to 2 MiB at
most, so the two agree within 64 MiB and 1 % (a few GB are held here)."""
import numpy as np
import pytest

from paper_1901_02971_gb300 import Solver
from paper_1901_02971_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [{"precision": "fp64"}, {"precision": "tf32"}, {"precision": "fp32", "variant": "InS"},
                                {"precision": "fp32", "compression": "randomized"}],
                         ids=lambda kw: "-".join(kw.values()))
def test_device_bytes_is_what_the_handle_holds(cuda_ok, kw):
    import torch
    p = I.laplacian_3d(64)
    b = torch.from_numpy(I.rhs(p.n, 1)).cuda()
    used = []
    for _ in range(2):  # the first handle loads the kernels
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        s = Solver.from_problem(p, levels=10, eps=1e-2, **kw)
        try:
            s.factorize().solve(b, check=False)
            used.append((free - torch.cuda.mem_get_info()[0], s.stats().device_bytes))
        finally:
            s.close()
    taken, told = used[1]
    assert abs(taken - told) <= 0.01 * taken + (64 << 20), used
