"""The run kernel of the fixed-point composed step (a run of steps in one cooperative launch)
against the step and face kernels (a forced ept takes those), bit for bit, and the oracle: tile
and block edges, faces beside tile boundaries, every degree, three and five stages, differences
past the integer range, any split of a run into calls."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import paper_2404_03399_gb300 as adg  # noqa: E402
from oracle import delays as odelays, dg  # noqa: E402
from workloads import random_nodal  # noqa: E402

pytestmark = pytest.mark.gpu


def _run(cfg, u0, calls):
    s = adg.Solver(cfg, torch.tensor(u0, device="cuda"))
    assert s.variant[0] == "fixed"
    for n in calls:
        s.step(n)
    out, dt = s.state().cpu().numpy(), s.dt
    s.close()
    return out, dt


@pytest.mark.parametrize("rk", ["ssprk3", "lsrk4"])
@pytest.mark.parametrize("K,P,p,mode", [
    (32, 1, 3, "sync"), (33, 3, 2, "at"), (120, 12, 1, "async"), (895, 5, 3, "at"), (897, 1, 4, "sync"),
    (1024, 64, 3, "at"), (1110, 111, 2, "at"), (9728, 76, 3, "at"), (10000, 1000, 4, "async"), (48640, 190, 1, "at"),
    (65536, 256, 3, "at"), (130000, 130, 2, "at")])
def test_runs_equal_the_step_kernels(K, P, p, mode, rk):
    kw = dict(pde="advection", K=K, p=p, P=P, cfl=0.002, mode=mode, L=5, q=min(p + 1, 3), seed=14, rk=rk)
    u0 = random_nodal(K, p, 9)
    got, dt = _run(adg.Config(**kw), u0, [19])
    assert np.array_equal(_run(adg.Config(ept=1, **kw), u0, [19])[0], got)
    assert np.array_equal(_run(adg.Config(**kw), u0, [1, 2, 16])[0], got)
    if K <= 1200:
        sync = mode == "sync"
        prob = dg.Problem(pde="advection", K=K, p=p, P=P, dt=dt, rk=rk, mode="sync" if sync else "adg",
                          q=kw["q"] if mode == "at" else 1, delays=odelays.delay_table(14, P, 19, 5))
        ref = dg.run(prob, u0, 19).numpy()
        assert np.max(np.abs(got - ref)) < 1e-12 * np.max(np.abs(ref))


def test_differences_past_the_integer_range_and_long_runs():
    # rough data, delays up to 7 and AT3 at a Courant number where the PE-face differences pass
    # the integer range (the FP64 correction), over more steps than one launch takes
    kw = dict(pde="advection", K=2048, p=3, P=64, cfl=0.05, mode="at", L=8, q=3, seed=1)
    u0 = random_nodal(2048, 3, 41)
    assert np.array_equal(_run(adg.Config(**kw), u0, [60])[0], _run(adg.Config(ept=1, **kw), u0, [60])[0])
    kw.update(cfl=0.002)
    assert np.array_equal(_run(adg.Config(**kw), u0, [700])[0], _run(adg.Config(ept=1, **kw), u0, [700])[0])
