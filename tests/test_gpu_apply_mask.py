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


@pytest.mark.parametrize("p,n", [(2, (7, 5, 6)), (3, (5, 4, 6))])
@pytest.mark.parametrize("blocks", ["vertex", "element"])
@pytest.mark.parametrize("bc", [0, 1])  # one clamped face; three faces with a fixed component each
def test_shared_factors_ignore_entries_that_are_not_free(p, n, blocks, bc):
    """The shared factors' tensor-core product on blocks at fixed faces: NaN in the entries that are not free gives
    the bits that zeros give."""
    from paper_1809_00828_gb300 import fcm
    w = I.Workload("shared", n, p, 1.0, I.uncut(), 1e-9, bc=bc)
    s = fcm.Solver(w)
    s.precond_build(precision="mixed", blocks=blocks, launch="concurrent")
    assert s.info["n_cells_cut"] == 0 and s.info["n_gemm_blocks"] > 0 and s.info["n_blocks_fp32"] > 0
    free = O.Problem.from_workload(w).free_lat
    x = np.zeros(s.n)
    x[free] = I.random_vector(11, len(free))
    z = s.apply_S(torch.from_numpy(x).cuda())
    x[np.setdiff1d(np.arange(s.n), free)] = np.nan
    assert float(z.abs().max()) > 0 and torch.equal(s.apply_S(torch.from_numpy(x).cuda()), z)
    s.close()
