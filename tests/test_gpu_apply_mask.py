"""K and S applied to a user's vectors: entries that are not free are ignored whatever they hold, no copy of the
input stands between the caller and the kernels, and the output may be the input.  The small grids have dense
cells only; the larger one has uncut cells too, and shared factors with tensor-core tiles.

The additions are the same in every form, so the results are compared bit for bit.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1809_00828_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,n", [(1, 5), (2, 3), (2, 14), (3, 3), (4, 2)])
@pytest.mark.parametrize("precision,k", [("fp64", "fp64"), ("mixed", "double_float")])
def test_entries_that_are_not_free_are_ignored(p, n, precision, k):
    from paper_1809_00828_gb300 import fcm
    w = I.workload_porous(5, n, p, 6, 1e-6, 2, 1e-9)
    s = fcm.Solver(w)
    s.set_k_precision(k)
    s.precond_build(precision=precision)
    free = np.zeros(s.n, bool)
    free[O.Problem.from_workload(w).free_lat] = True
    for nr in (1, 3):
        X = np.stack([I.random_vector(40 + c, s.n) for c in range(nr)])
        X[:, ~free] = 0.0
        G = X.copy()
        G[:, ~free] = [np.nan, np.inf, -3.0][nr % 3]
        x, gx = (torch.from_numpy(a.reshape(-1)).cuda() for a in (X, G))
        z = s.apply_S(x)
        assert float(z.abs().max()) > 0 and torch.equal(s.apply_S(gx), z)
        if nr == 1:
            y = s.apply_K(x)
            assert float(y.abs().max()) > 0 and torch.equal(s.apply_K(gx), y)
            h = gx.clone()
            assert torch.equal(s.apply_K(h, out=h), y)
        h = gx.clone()
        assert torch.equal(s.apply_S(h, out=h), z)
    s.close()
