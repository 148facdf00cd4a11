"""The fused Burgers step and its adjoint at mesh sizes where the launch shape changes (one-warp or
four-warp blocks, blocks held to an SM's even share) and inside the ranges between: the whole
field against the CPU oracle, and the gradient of a tiled field against a small mesh's."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import paper_2404_03399_gb300 as adg  # noqa: E402
from oracle import delays as odelays, dg  # noqa: E402
from workloads import random_nodal  # noqa: E402

pytestmark = pytest.mark.gpu
TOL = 1e-12   # the parity bar of the other kernels, relative to the field's maximum


def _edges():
    sm = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 152
    # 26 owned elements a warp: the last mesh below 16 and 32 warps per SM, the first at them,
    # and odd sizes between
    return [26 * 16 * sm - 27, 26 * 16 * sm + 1, 26 * 17 * sm + 13, 26 * 25 * sm - 5,
            26 * (32 * sm - 1), 26 * 32 * sm + 1]


@pytest.mark.parametrize("at", range(6))
@pytest.mark.parametrize("p,rk,nu", [(1, "ssprk3", 0.0), (2, "ssprk3", 0.0), (3, "lsrk3", 0.0), (1, "rk2", 0.1)])
def test_launch_shapes(at, p, rk, nu):
    K = _edges()[at]
    cfg = adg.Config(pde="burgers", K=K, p=p, P=1, mode="sync", rk=rk, seed=4, nu=nu,
                     **({"dt": 2e-3 * (6.28 / K) ** 2} if nu else {"cfl": 0.004}))
    u0 = 0.3 + random_nodal(K, p, 7)
    s = adg.Solver(cfg, torch.tensor(u0, device="cuda"))
    s.step(3)
    got, dt = s.state().cpu().numpy(), s.dt
    s.close()
    prob = dg.Problem(pde="burgers", K=K, p=p, P=1, dt=dt, x0=cfg.x0, x1=cfg.x1, mode="sync", q=1,
                      delays=None, rk=rk, nu=nu)
    ref = dg.run(prob, u0, 3).numpy()
    assert np.max(np.abs(got - ref)) < TOL * np.max(np.abs(ref))


@pytest.mark.parametrize("at", [1, 3])
def test_launch_shapes_with_delays(at):
    K = _edges()[at] // 16 * 16
    cfg = adg.Config(pde="burgers", K=K, p=3, P=K // 16, cfl=0.004, mode="at", L=3, q=2, seed=4)
    u0 = 0.3 + random_nodal(K, 3, 7)
    s = adg.Solver(cfg, torch.tensor(u0, device="cuda"))
    s.step(4)
    got, dt = s.state().cpu().numpy(), s.dt
    s.close()
    prob = dg.Problem(pde="burgers", K=K, p=3, P=cfg.P, dt=dt, x0=cfg.x0, x1=cfg.x1, mode="adg", q=2,
                      delays=odelays.delay_table(cfg.seed, cfg.P, 4, cfg.L))
    ref = dg.run(prob, u0, 4).numpy()
    assert np.max(np.abs(got - ref)) < TOL * np.max(np.abs(ref))


@pytest.mark.parametrize("at", range(6))
def test_gradient_of_a_tiled_field(at):
    # a field of equal tiles: its gradient is the small mesh's, tile by tile
    K0, p = 64, 2
    tiles = _edges()[at] // K0 + at % 2
    u0 = 0.3 + random_nodal(K0, p, 7)
    dt = 0.004 * 6.28 / K0
    grads = []
    for m in (1, tiles):
        cfg = adg.Config(pde="burgers", K=K0 * m, p=p, P=1, dt=dt, mode="sync", x0=0.0, x1=6.28 * m, seed=4)
        u = np.tile(u0, (m, 1))
        s = adg.Solver(cfg, torch.tensor(u, device="cuda"))
        grads.append(s.grad(torch.tensor(np.roll(u, 3, axis=0), device="cuda"), 4, 4)[1].cpu().numpy())
        s.close()
    ref = np.tile(grads[0], (tiles, 1))
    assert np.max(np.abs(grads[1] - ref)) < TOL * np.max(np.abs(ref))
