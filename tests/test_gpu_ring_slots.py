"""Ring slots: spare ones only where a launch takes several steps."""
import pytest

torch = pytest.importorskip("torch")
import paper_2404_03399_gb300 as adg  # noqa: E402

pytestmark = pytest.mark.gpu


def test_large_staged_meshes_have_no_spare_slots():
    # 2^20 PEs of one element: fields 50 MB, delays 537 MB, a ring of L - 1 + q = 3 levels of three
    # stages 151 MB (with seven spare ones 503 MB)
    K = 1 << 20
    u0 = torch.ones((K, 2), dtype=torch.float64, device="cuda")
    cfg = adg.Config(pde="advection", K=K, p=1, P=K, a=-1.0, cfl=0.005, mode="at", L=2, q=2)
    adg.Solver(cfg, u0).close()   # the kernels' own memory
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    s = adg.Solver(cfg, u0)
    used = free - torch.cuda.mem_get_info()[0]
    s.step(2)
    s.close()
    assert used < 850e6
