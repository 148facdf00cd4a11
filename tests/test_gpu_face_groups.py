"""The grouped PE-face kernels of the fixed-point step: face counts around whole warps of the
batched fix-up (eight faces of one degree, padded) in a batch of mixed degrees, bit for bit the
single runs of the step and face kernels, and the oracle; differences left to FP64 among
them."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import paper_2404_03399_gb300 as adg  # noqa: E402
from oracle import delays as odelays, dg  # noqa: E402
from workloads import random_nodal  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cfl", [0.002, 0.03])
def test_batched_faces_equal_single_runs(cfl):
    # cfl 0.03 with delays up to 5: rough data whose differences pass the integer range
    shapes = [(64, 1, 3), (64, 8, 1), (72, 9, 2), (120, 15, 3), (80, 10, 4), (24, 2, 4), (63, 7, 3), (8, 1, 2), (136, 17, 1)]
    cfgs, u0s = [], []
    for i, (K, P, p) in enumerate(shapes):
        cfgs.append(adg.Config(pde="advection", K=K, p=p, P=P, a=0.7 + 0.1 * i, cfl=cfl, mode="at", L=6, q=min(p + 1, 3),
                               seed=50 + i, variant="fixed"))
        u0s.append(random_nodal(K, p, 60 + i))
    b = adg.BatchSolver(cfgs, [torch.tensor(u, device="cuda") for u in u0s])
    b.step(25)
    for i, (cfg, u0) in enumerate(zip(cfgs, u0s)):
        got = b.state(i).cpu().numpy()
        cfg.ept = 1   # the step and face kernels
        s = adg.Solver(cfg, torch.tensor(u0, device="cuda"))
        s.step(25)
        assert np.array_equal(got, s.state().cpu().numpy()), i
        tbl = odelays.delay_table(cfg.seed, cfg.P, 25, cfg.L)
        prob = dg.Problem(pde="advection", K=cfg.K, p=cfg.p, P=cfg.P, a=cfg.a, dt=s.dt, q=cfg.q,
                          mode="adg" if cfg.P > 1 else "sync", delays=tbl)
        s.close()
        ref = dg.run(prob, u0, 25).numpy()
        assert np.max(np.abs(got - ref)) < 1e-12 * np.max(np.abs(ref)), i
    b.close()
