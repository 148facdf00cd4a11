"""Device memory of the gradient: a run that could be recorded whole takes the caller's segments
where the device has no room for the recording."""
import pytest

torch = pytest.importorskip("torch")
import paper_2404_03399_gb300 as adg  # noqa: E402
from oracle import dg  # noqa: E402
from workloads import HALF_PLUS_SIN, random_nodal  # noqa: E402

pytestmark = pytest.mark.gpu
MB = 1 << 20


def _solver(K, P=1):
    cfg = adg.Config(pde="burgers", K=K, p=3, P=P, cfl=0.005, mode="at" if P > 1 else "sync", L=3, q=2, seed=4)
    u0 = torch.tensor(dg.modes_initial(HALF_PLUS_SIN, K, 3), device="cuda")
    return adg.Solver(cfg, u0), u0 + torch.tensor(0.05 * random_nodal(K, 3, 1), device="cuda")


def test_segments_where_the_recording_does_not_fit():
    # fields of 32 MB; nine steps whole are 28 of them and 6 more that any gradient takes, in
    # segments of three 18 of them (28 with the second stream's)
    K, steps = 1 << 20, 9
    s, target = _solver(4096)
    s.grad(target, steps, 3)   # loads the kernels
    s.close()
    s, target = _solver(K)
    ref = s.grad(target, steps, steps)
    s.close()
    s, target = _solver(K)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    fill = torch.empty(torch.cuda.mem_get_info()[0] - 1000 * MB, dtype=torch.uint8, device="cuda")
    try:
        J, grad = s.grad(target, steps, 3)
    finally:
        del fill
        torch.cuda.empty_cache()
    s.close()
    assert J == ref[0] and torch.equal(grad, ref[1])
