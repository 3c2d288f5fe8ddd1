"""A NaN that only the compression of an interface meets: every off-diagonal entry
is a stored zero but those between two clusters that outlive the first step, which
are NaN.  The pivots and the other couplings are sound and every finite column of
the two interfaces' couplings is zero, so a compression that passes NaN columns
over cuts the interfaces to rank 0 and the factorization goes through without
them.  It has to end in an error that names the step and the interface."""
import numpy as np
import pytest

from paper_1901_02971_gb300 import Solver, SpandError
from paper_1901_02971_gb300 import _lib as L
from paper_1901_02971_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _nan_between_survivors(p, levels, sign):
    """Sets the values described above; returns the two clusters."""
    s = Solver.from_problem(p, levels=levels)
    try:
        tree, step = s.tree(), s.step(1)
    finally:
        s.close()
    owner = np.empty(p.n, dtype=np.int64)
    ptr = tree["cluster_ptr"]
    for c in range(len(ptr) - 1):
        owner[tree["perm"][ptr[c]:ptr[c + 1]]] = c
    rows = np.repeat(np.arange(p.n), np.diff(p.rowptr))
    a, b = owner[rows], owner[p.colind]
    alive = np.asarray(step["elim"]) == 0
    between = (a != b) & alive[a] & alive[b]
    e = np.flatnonzero(between)[0]
    pair = {int(a[e]), int(b[e])}
    hit = between & np.isin(a, list(pair)) & np.isin(b, list(pair))
    p.vals = np.where(hit, np.copysign(np.nan, sign), np.where(rows == p.colind, p.vals, 0.0))
    return pair


@pytest.mark.parametrize("form", ["coloured", "simultaneous", "randomized", "InS", "In"])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("dim,n,levels", [(2, 33, 3), (3, 16, 3), (3, 21, 6)])
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_nan_coupling_is_reported(cuda_ok, sign, dim, n, levels, precision, form):
    p = I.laplacian_2d(n) if dim == 2 else I.laplacian_3d(n)
    pair = _nan_between_survivors(p, levels, sign)
    option = {"randomized": "compression", "InS": "variant", "In": "variant"}.get(form, "sparsify_order")
    s = Solver.from_problem(p, levels=levels, eps=1e-2, precision=precision, **{option: form})
    try:
        with pytest.raises(SpandError) as ei:
            s.factorize()
        assert ei.value.code == L.SPAND_ERR_NOT_SPD
        assert "not finite" in str(ei.value)
        st = s.stats()
        assert st.fail_step == 1 and st.fail_cluster in pair
    finally:
        s.close()
