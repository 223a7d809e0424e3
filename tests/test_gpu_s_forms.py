"""S r for one to eight right-hand sides with mixed factors, over the block sizes of both block rules, against
the oracle.  A low threshold (1e3) gives FP32 and double-float factors on one small cube; at p <= 2 they are
stored folded (each symmetric pair of entries once), and every number of right-hand sides is rounded up to an
instantiated number of columns.

Bounds: per DOF as in schwarz_bounds.py, with 2^-20 for the FP32 factors' storage and FP32 product sums.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1809_00828_gb300 import inputs as I
from schwarz_bounds import dof_bound

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,n", [(1, (5, 4, 6)), (2, (3, 4, 3)), (3, (2, 3, 2))])
@pytest.mark.parametrize("blocks", ["vertex", "element"])
def test_mixed_S_for_every_number_of_right_hand_sides(p, n, blocks):
    from paper_1809_00828_gb300 import fcm
    g = I.random_sphere_voids(9, 3, 0.15, 0.3, octree_depth=2)
    w = I.Workload("s_forms", n, p, 1e-6, g, 1e-9, hi=(1.0, 1.2, 0.9))
    P = O.Problem.from_workload(w)
    if blocks == "element":
        P.precond_build(3, 1e-13, 0.9)
    else:
        P.precond_build(0)
    s = fcm.Solver(w)
    s.precond_build(precision="mixed", cond_fp64=1e3, blocks=blocks, eta_bar=0.9)
    assert s.info["n_blocks_fp32"] + s.info["n_factors_ff"] > 0
    R = [I.random_vector(70 + k, s.n) for k in range(8)]
    ref = [P.apply_S(r[P.free_lat]) for r in R]
    bound = [dof_bound(P, r[P.free_lat], u_factor=2.0 ** -20) + 1e-14 * np.abs(z).max() for r, z in zip(R, ref)]
    fixed = np.ones(s.n, bool)
    fixed[P.free_lat] = False
    for nr in range(1, 9):
        # not free: ignored on input, whatever the values
        X = np.stack(R[:nr])
        X[:, fixed] = 3.0
        Z = s.apply_S(torch.from_numpy(X.reshape(-1)).cuda()).cpu().numpy().reshape(nr, -1)
        assert not Z[:, fixed].any()
        for k in range(nr):
            assert np.all(np.abs(Z[k][P.free_lat] - ref[k]) <= bound[k]), (nr, k)
    s.close()


def test_wait_limit_of_the_streamed_factors_and_matrices():
    """fcm_set_wait_limit(0) on a problem whose S and K both wait for bulk copies: timeout, then recovery."""
    from paper_1809_00828_gb300 import fcm
    w = I.workload_porous(5, 8, 2, 6, 1e-8, 3, 1e-9)
    s = fcm.Solver(w)
    s.set_k_precision("double_float")
    s.precond_build(precision="mixed", cond_fp64=10.0)
    assert s.info["n_factors_ff"] > 0 and s.info["n_cells_cut"] > 0
    b = s.rhs()
    u_ref, its_ref, _, _ = s.pcg_solve(b, 1e-9, 2000)
    y_ref = s.apply_K(b)
    s.set_wait_limit(0)
    _, _, _, st = s.pcg_solve(b, 1e-9, 2000, check=False)
    assert st == fcm.FCM_ETIMEOUT
    s.precond_build(precision="mixed", cond_fp64=10.0)  # clears the flag
    s.apply_K(b)
    torch.cuda.synchronize()
    assert s.get_info()["device_error"] == 1
    s.set_wait_limit(-1)
    u, its, _, _ = s.pcg_solve(b, 1e-9, 2000)
    assert its == its_ref and torch.equal(u, u_ref) and torch.equal(s.apply_K(b), y_ref)
    assert s.get_info()["device_error"] == 0
    s.close()


@pytest.mark.parametrize("p,n", [(1, (5, 4, 6)), (2, (3, 4, 3))])
@pytest.mark.parametrize("precision", ["mixed", "mixed_fp64"])
def test_own_blocks_of_several_kinds_in_one_launch(p, n, precision):
    """A small grid's folded FP32 blocks and its double-float or FP64 ones share a launch (then one for the sum)."""
    from paper_1809_00828_gb300 import fcm
    w = I.Workload("s_own", n, p, 1e-6, I.random_sphere_voids(9, 3, 0.15, 0.3, octree_depth=2), 1e-9, hi=(1.0, 1.2, 0.9))
    P = O.Problem.from_workload(w)
    P.precond_build(3, 1e-13, 0.9)
    conds = sorted(P.block(b)[2][0] for b in range(P.nblocks()))
    s = fcm.Solver(w)
    s.precond_build(precision=precision, cond_fp64=conds[len(conds) // 2], blocks="element", eta_bar=0.9)
    kinds = s.info["n_blocks_fp32"], s.info["n_factors"] - s.info["n_blocks_fp32"]
    assert min(kinds) > 0 and s.info["n_gemm_blocks"] == 0 and s.info["s_apply_launches"] == 2
    for nr in (1, 3, 8):
        X = np.stack([I.random_vector(90 + k, s.n) for k in range(nr)])
        Z = s.apply_S(torch.from_numpy(X.reshape(-1)).cuda()).cpu().numpy().reshape(nr, -1)
        for x, z in zip(X, Z):
            ref = P.apply_S(x[P.free_lat])
            bound = dof_bound(P, x[P.free_lat], u_factor=2.0 ** -20) + 1e-14 * np.abs(ref).max()
            assert np.all(np.abs(z[P.free_lat] - ref) <= bound), nr
    s.close()
