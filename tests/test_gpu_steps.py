"""Small meshes that take several steps per launch (staged advection, the Euler equations):
sizes around a block's owned elements against the oracle, and every split of a run into calls
(launches of one step up to the largest) bit for bit the same."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import paper_2404_03399_gb300 as adg  # noqa: E402
from oracle import delays as odelays, dg, euler as oeuler  # noqa: E402
from workloads import random_nodal  # noqa: E402

pytestmark = pytest.mark.gpu
TOL = 1e-12   # the parity bar of the staged kernels, relative to the field's maximum


def _run(cfg, u0, calls):
    s = adg.Solver(cfg, torch.tensor(u0, device="cuda"))
    for n in calls:
        s.step(n)
    out, dt = s.state().cpu().numpy(), s.dt
    s.close()
    return out, dt


@pytest.mark.parametrize("a", [1.0, -1.0])
@pytest.mark.parametrize("K,P,p,mode", [(1, 1, 2, "sync"), (7, 7, 1, "at"), (17, 1, 2, "sync"), (18, 6, 2, "at"),
                                        (69, 23, 3, "async"), (200, 50, 4, "at"), (2500, 500, 2, "at")])
def test_advection_steps(K, P, p, mode, a):
    cfg = adg.Config(pde="advection", K=K, p=p, P=P, a=a, cfl=0.004, mode=mode, L=4, q=2, seed=6,
                     variant="staged")
    u0 = random_nodal(K, p, 3)
    got, dt = _run(cfg, u0, [29])
    tbl = odelays.delay_table(cfg.seed, P, 29, 4)
    prob = dg.Problem(pde="advection", K=K, p=p, P=P, a=a, dt=dt, mode="sync" if mode == "sync" else "adg",
                      q=2 if mode == "at" else 1, delays=tbl)
    ref = dg.run(prob, u0, 29).numpy()
    assert np.max(np.abs(got - ref)) < TOL * np.max(np.abs(ref))
    for calls in ([1] * 29, [8, 8, 13], [3, 26]):
        assert np.array_equal(_run(cfg, u0, calls)[0], got)


@pytest.mark.parametrize("K,P,p,rk,limiter", [(5, 1, 1, "rk2", True), (24, 8, 1, "rk2", True), (25, 5, 2, "ssprk3", True),
                                              (33, 3, 4, "rk1", False), (300, 20, 3, "ssprk3", False)])
def test_euler_steps(K, P, p, rk, limiter):
    cfg = adg.Config(pde="euler", K=K, p=p, P=P, x1=0.02, dt=0.002 * 0.02 / K, rk=rk, mode="at" if P > 1 else "sync",
                     L=3, q=2, seed=8, limiter=limiter)
    r = random_nodal(K, p, 5, 0.1), random_nodal(K, p, 6, 0.1), random_nodal(K, p, 7, 0.1)
    u0 = np.stack([1.0 + r[0], 0.3 + r[1], 2.5 + r[2]])
    got, dt = _run(cfg, u0, [23])
    tbl = odelays.delay_table(cfg.seed, P, 23, 3)
    s = oeuler.EulerSolver(oeuler.EulerProblem(K=K, p=p, P=P, dt=dt, rk=rk, mode="adg" if P > 1 else "sync", q=2,
                                               delays=tbl, limiter=limiter), u0)
    for _ in range(23):
        s.step()
    ref = s.u.numpy()
    assert np.max(np.abs(got - ref)) < TOL * np.max(np.abs(ref))
    for calls in ([1] * 23, [2, 3, 18]):
        assert np.array_equal(_run(cfg, u0, calls)[0], got)
