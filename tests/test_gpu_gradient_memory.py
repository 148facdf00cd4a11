"""Device memory of the gradient: a run that could be recorded whole takes the caller's segments
where the device has no room for the recording or the caller leaves none, with the same result."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import paper_2404_03399_gb300 as adg  # noqa: E402
from oracle import delays as odelays, dg  # noqa: E402
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


@pytest.mark.parametrize("P", [1, 8])
def test_segments_and_a_whole_recording_agree(P):
    # one recording; segments recomputed on a second stream (7, 40), one after the other (300:
    # two are longer than the delay table's window of 512), and of one step
    s, target = _solver(96, P)
    ref = s.grad(target, 310, 310)
    whole = s.grad(target, 310, 7)
    s.set_grad_memory(0)
    out = [whole] + [s.grad(target, 310, c) for c in (7, 40, 300, 1)]
    s.set_grad_memory(1 << 30)
    out.append(s.grad(target, 310, 7))
    s.close()
    for J, g in out:
        assert J == ref[0] and torch.equal(g, ref[1])


@pytest.mark.parametrize("K,p", [(63300, 1), (70000, 2)])
def test_overlapped_segments_of_16_to_32_warps_an_sm(K, p):
    # blocks are held to an SM's even share, but not those of two streams beside one another
    cfg = adg.Config(pde="burgers", K=K, p=p, P=100, cfl=0.005, mode="at", L=3, q=2, seed=4)
    u0 = torch.tensor(dg.modes_initial(HALF_PLUS_SIN, K, p), device="cuda")
    s = adg.Solver(cfg, u0)
    ref = s.grad(0.9 * u0, 12, 12)
    s.set_grad_memory(0)
    J, g = s.grad(0.9 * u0, 12, 3)
    s.close()
    assert J == ref[0] and torch.equal(g, ref[1])


@pytest.mark.parametrize("K,p,P,mode,q,steps,ckpt", [
    (64, 3, 4, "at", 2, 40, 16), (48, 2, 48, "at", 2, 25, 7), (80, 4, 8, "async", 1, 30, 4), (64, 1, 1, "sync", 0, 20, 4)])
def test_recomputed_gradient_matches_oracle(K, p, P, mode, q, steps, ckpt):
    L = 4 if P > 1 else 1
    cfg = adg.Config(pde="burgers", K=K, p=p, P=P, cfl=0.01, mode=mode, L=L, q=q, seed=9)
    u0 = dg.modes_initial(HALF_PLUS_SIN, K, p)
    g = u0 + 0.05 * random_nodal(K, p, 3)
    s = adg.Solver(cfg, torch.tensor(u0, device="cuda"))
    s.set_grad_memory(0)
    J, grad = s.grad(torch.tensor(g, device="cuda"), steps, ckpt)
    assert np.array_equal(s.state().cpu().numpy(), u0)
    prob = dg.Problem(pde="burgers", K=K, p=p, P=P, dt=s.dt, mode="adg" if P > 1 else "sync",
                      q=q if mode == "at" else 1, delays=odelays.delay_table(9, P, steps, L) if P > 1 else None)
    s.close()
    Jo, go = dg.gradient(prob, u0, g, steps)
    assert abs(J - Jo) <= 1e-12 * abs(Jo)
    assert np.max(np.abs(grad.cpu().numpy() - go)) <= 1e-12 * np.max(np.abs(go))


def test_kept_memory_is_the_callers_choice():
    # nine steps of 32 MB fields: 34 of them kept by default, none after 0, nor by a call under 0
    s, target = _solver(1 << 20)
    ref = s.grad(target, 9, 3)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    s.set_grad_memory(0)
    given = torch.cuda.mem_get_info()[0]
    assert given - free > 800 * MB
    J, grad = s.grad(target, 9, 3)
    torch.cuda.synchronize()
    assert J == ref[0] and torch.equal(grad, ref[1])
    del grad
    torch.cuda.empty_cache()
    assert torch.cuda.mem_get_info()[0] >= given - 64 * MB   # (another result's 32 MB)
    with pytest.raises(adg.AdgError):
        s.set_grad_memory(-1)
    s.close()
