"""Segments of the gradient: checkpoint intervals longer than the delay table's window, runs
recorded whole and runs recomputed give the same gradient bit for bit, call after call (the
working memory is kept between them)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import paper_2404_03399_gb300 as adg  # noqa: E402
from oracle import dg  # noqa: E402
from workloads import HALF_PLUS_SIN, random_nodal  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pde", ["burgers", "advection"])
def test_intervals_beyond_the_delay_window(pde):
    cfg = adg.Config(pde=pde, K=48, p=2, P=6, cfl=0.005, mode="at", L=3, q=2, seed=4)
    u0 = torch.tensor(dg.modes_initial(HALF_PLUS_SIN, 48, 2), device="cuda")
    target = u0 + torch.tensor(0.05 * random_nodal(48, 2, 1), device="cuda")
    s = adg.Solver(cfg, u0)
    out = [s.grad(target, 620, c) for c in (40, 600, 1000, 600)]
    s.close()
    assert np.isfinite(out[0][0])
    for J, g in out[1:]:
        assert J == out[0][0] and torch.equal(g, out[0][1])


def test_whole_and_split_recording_agree():
    # 200 steps recorded whole; the same through the two halves of a longer run's segments
    cfg = adg.Config(pde="burgers", K=200, p=3, P=8, cfl=0.005, mode="at", L=4, q=2, seed=5)
    u0 = torch.tensor(dg.modes_initial(HALF_PLUS_SIN, 200, 3), device="cuda")
    s = adg.Solver(cfg, u0)
    a = s.grad(0.9 * u0, 600, 100)   # past the window: segments of 100, recomputed
    b = s.grad(0.9 * u0, 600, 300)   # segments of 300
    s.close()
    assert a[0] == b[0] and torch.equal(a[1], b[1])
