"""The run kernel's bounded wait: with no polls allowed every block gives up at once, and the calls
say so; a solver made afterwards steps as before."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import paper_2404_03399_gb300 as adg  # noqa: E402
from paper_2404_03399_gb300 import _abi  # noqa: E402
from workloads import random_nodal  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,P,mode", [(9728, 76, "at"), (48640, 1, "sync")])
def test_a_wait_that_runs_out_is_reported(K, P, mode):
    cfg = adg.Config(pde="advection", K=K, p=2, P=P, cfl=0.002, mode=mode, L=5, q=3, seed=1)
    u0 = torch.tensor(random_nodal(K, 2, 5), device="cuda")
    s = adg.Solver(cfg, u0)
    s.step(8)
    ref = s.state()
    s.set_wait_limit(0)
    s.step(8)
    for call in (s.state, lambda: s.step(1), s.integral, s.state):
        with pytest.raises(adg.AdgError) as e:
            call()
        assert e.value.code == _abi.ADG_ETIMEOUT
    s.close()
    s = adg.Solver(cfg, u0)
    with pytest.raises(adg.AdgError):
        s.set_wait_limit(-1)
    s.set_wait_limit(1 << 24)
    s.step(8)
    assert np.array_equal(s.state().cpu().numpy(), ref.cpu().numpy())
    s.close()
