"""Bounded waits of the double-float K apply (element matrices copied in bulk, p <= 2) outside the iterations: the true
residual at the end of each solve, and the assembly of the coarse operator by probing K.

A wait limit of 0 makes every K apply give up (the copies land, the kernels return), and a preconditioner without
blocks (pure Jacobi) waits for nothing.  With b = 0 the solves stop before their first iteration, so the only K
apply of the call is the one for the true residual: the call has to say that it failed.
"""
import pytest

from paper_1809_00828_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _solver():
    from paper_1809_00828_gb300 import fcm
    s = fcm.Solver(I.workload_porous(5, 8, 2, 6, 1e-8, 3, 1e-9))
    s.set_k_precision("double_float")
    s.precond_build(blocks="element", eta_bar=0.0)
    assert s.info["n_cells_cut"] > 0 and s.info["n_blocks"] == 0
    return s


@pytest.mark.parametrize("kind", ["pcg", "many", "fpcg"])
def test_a_true_residual_that_timed_out_is_reported(kind):
    from paper_1809_00828_gb300 import fcm
    s = _solver()

    def solve(b):
        if kind == "fpcg":
            return s.fpcg_solve(None, 0.0, b, 1e-6, 50, check=False, coarse_iters=1)
        return s.pcg_solve(b, 1e-6, 50, check=False)

    zero = s.empty(2 if kind == "many" else 1)
    u, its, rel, st = solve(zero)  # builds the coarse operator, with working waits
    assert (its, rel, st) == (0, 0.0, fcm.FCM_OK) and not u.any()
    s.set_wait_limit(0)
    assert solve(zero)[3] == fcm.FCM_ETIMEOUT
    assert s.last_solve()["status"] == fcm.FCM_ETIMEOUT
    s.set_wait_limit(-1)
    assert solve(zero)[3] == fcm.FCM_OK
    assert s.get_info()["device_error"] == 0
    s.close()


def test_a_coarse_operator_from_timed_out_products_is_not_kept():
    from paper_1809_00828_gb300 import fcm
    s = _solver()
    x = torch.from_numpy(I.random_vector(3, 3 * 8 ** 3)).float().cuda()
    s.set_wait_limit(0)
    with pytest.raises(fcm.FcmError) as e:
        s.coarse_apply(x)
    assert e.value.status == fcm.FCM_ETIMEOUT
    s.set_wait_limit(-1)
    y = s.coarse_apply(x)
    fresh = _solver()
    assert torch.equal(y, fresh.coarse_apply(x))
    for q in (s, fresh):
        q.close()
