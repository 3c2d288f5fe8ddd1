"""The FP64 sparsification QR on interfaces wide enough for clusters of several
CTAs and for every lane grouping of its columns: per-cluster ranks equal to the
FP64 oracle's, and z = M M^T r element by element.  The bound is the element-wise
one of the small cases of the apply parity test (1e-12 of the largest entry) times
ten for the larger blocks (their products are up to eight times longer, their
condition numbers a few times larger)."""
import numpy as np
import pytest

from oracle import spand_oracle as O
from paper_1901_02971_gb300 import Solver
from paper_1901_02971_gb300 import inputs as I

pytestmark = pytest.mark.gpu

# few, wide interfaces (2 to 4 leaves) up to many narrow ones; odd sides
CASES = [(13, 2), (18, 3), (22, 4), (21, 6), (25, 8)]


@pytest.mark.parametrize("n,levels", CASES)
def test_fp64_qr_matches_oracle(cuda_ok, n, levels):
    import torch
    p = I.diffusion_3d(n, 31 + n, block=2, lo=-1.0, hi=1.0)
    tree = O.analyze(p.n, p.rowptr, p.colind, p.coords, levels)
    F = O.factorize(p.rowptr, p.colind, p.vals, tree, 1e-2)
    s = Solver.from_problem(p, levels=levels, eps=1e-2, precision="fp64").factorize()
    try:
        for t in range(1, levels + 1):
            assert np.array_equal(s.ranks(t)[1], F.sizes_after[t - 1]), t
        r = I.rhs(p.n, 5)
        z = s.apply(torch.from_numpy(r).cuda()).cpu().numpy()
    finally:
        s.close()
    z_ref = np.empty(p.n)
    z_ref[tree.perm] = O.apply(F, r[tree.perm])
    err = np.abs(z - z_ref).max() / np.abs(z_ref).max()
    assert err <= 1e-11, err
