"""K x on both sides of the size rule of the uncut cells: few uncut cells go with the cut cells' dense product,
more of them take the Legendre modal form (32 cells per CTA).  Grids just below and above the rule's line, of
unequal cell sides and counts that are no multiple of 32, in both arithmetics.

Tolerance: the modal form is exact for the uncut integrand, so K x equals the oracle's up to rounding: each of
the three transforms, the weights and the sum of up to 8 cells adds a few ulps of max |K_e| |x_e| (2^-53, or
2^-46 for double-float), far below the 1e-12 of max |y| that the other K tests use.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1809_00828_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# p = 1: dense up to 1,216 uncut cells; p = 2: 608; p = 3: 304; p = 4: always the sum-factorised form
@pytest.mark.parametrize("p,n", [(1, (10, 9, 11)), (1, (12, 13, 11)), (2, (8, 7, 9)), (2, (11, 9, 10)), (3, (6, 7, 5)),
                                 (3, (9, 7, 8)), (4, (3, 4, 2))])
@pytest.mark.parametrize("bc", [0, 1])
def test_k_apply_on_both_sides_of_the_uncut_rule(p, n, bc):
    from paper_1809_00828_gb300 import fcm
    g = I.random_sphere_voids(9, 2, 0.15, 0.25, octree_depth=2)
    w = I.Workload("forms", n, p, 1e-6, g, 1e-8, bc=bc, hi=(1.0, 1.3, 0.8))
    P = O.Problem.from_workload(w)
    K = P.csr()
    s = fcm.Solver(w)
    x = I.random_vector(3, s.n)
    xf = P.from_lattice(x)
    y_ref = K @ xf
    for mode in ("fp64", "double_float"):
        s.set_k_precision(mode)
        xt = torch.from_numpy(x).cuda()
        y = s.apply_K(xt)
        yn = y.cpu().numpy()
        assert np.abs(P.from_lattice(yn) - y_ref).max() < 1e-12 * np.abs(y_ref).max()
        fixed = np.ones(s.n, bool)
        fixed[P.free_lat] = False
        assert not yn[fixed].any()
        z = xt.clone()
        s.apply_K(z, out=z)  # in place
        assert torch.equal(z, y)
    s.close()
