"""Device memory of S for several right-hand sides: the block products, and not the solver's vectors."""
import pytest

from paper_1809_00828_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_apply_S_many_allocates_no_solver_vectors():
    from paper_1809_00828_gb300 import fcm
    s = fcm.Solver(I.Workload("many", (48, 48, 48), 2, 1.0, I.uncut(), 1e-6))
    s.precond_build(precision="mixed", launch="serial")
    r = torch.randn(8 * s.n, dtype=torch.float64, device="cuda")
    z = torch.empty_like(r)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    s.apply_S(r, out=z)
    torch.cuda.synchronize()
    used = before - torch.cuda.mem_get_info()[0]
    blocks = 8 * s.info["n_blocks"] * (s.info["max_block"] + 16) * 8  # rows of FP64 per block, padded
    assert used < blocks + 64e6 < blocks + 6 * 8 * s.n * 8
    zs = z.clone()
    # a solve of as many right-hand sides brings the vectors, another count and a new build replace the workspace
    u, _, _, st = s.pcg_solve(r[:8 * s.n], 1e-2, 5, check=False)
    assert st in (fcm.FCM_OK, fcm.FCM_ENOTCONV)
    assert torch.equal(s.apply_S(r, out=z), zs)
    s.pcg_solve(r[:2 * s.n], 1e-2, 5, check=False)
    s.precond_build(precision="mixed", launch="serial")
    assert torch.equal(s.apply_S(r, out=z), zs)
    s.close()
