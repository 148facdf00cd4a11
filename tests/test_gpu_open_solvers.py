"""Several solvers open at once: what one needs of a kernel that they share (its limit of shared
memory) leaves the others' launches as they were."""
import ctypes as C

import numpy as np
import pytest

torch = pytest.importorskip("torch")
import paper_2404_03399_gb300 as adg  # noqa: E402
from paper_2404_03399_gb300 import _abi  # noqa: E402
from workloads import random_nodal  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rk", ["ssprk3", "lsrk4"])
@pytest.mark.parametrize("p", [1, 3])
def test_a_run_of_more_faces_steps_after_one_of_fewer_is_made(p, rk):
    # 32 and 2 faces to a tile of some 430 elements, which set its shared memory
    K, u0 = 65536, random_nodal(65536, p, 3)
    kw = dict(pde="advection", K=K, p=p, cfl=0.002, mode="at", L=8, q=min(p + 1, 3), seed=2, rk=rk)
    big = adg.Solver(adg.Config(P=4096, **kw), torch.tensor(u0, device="cuda"))
    small = adg.Solver(adg.Config(P=256, **kw), torch.tensor(u0, device="cuda"))
    for s in (big, small, big):
        s.step(13)
    out = [s.state().cpu().numpy() for s in (big, small)]
    big.close()
    small.close()
    for got, P, n in zip(out, (4096, 256), (26, 13)):
        s = adg.Solver(adg.Config(P=P, ept=1, **kw), torch.tensor(u0, device="cuda"))
        s.step(n)
        ref = s.state().cpu().numpy()
        s.close()
        assert np.array_equal(got, ref)


def test_a_solver_that_does_not_fit_leaves_the_next_one_alone():
    # four fields of 3 x 2^30 x 5 values, 515 GB: refused before u0 is read
    lib, ctx = adg.load(), C.c_void_p()
    u0 = torch.zeros(1, dtype=torch.float64, device="cuda")
    c, keep = adg.Config(pde="euler", K=1 << 30, p=4, dt=1e-9, rk="rk2").to_c()
    assert lib.adg_init(C.byref(c), u0.data_ptr(), None, C.byref(ctx)) == _abi.ADG_ENOMEM
    cfg = adg.Config(pde="advection", K=64, p=2, cfl=0.002)
    s = adg.Solver(cfg, torch.ones((64, 3), dtype=torch.float64, device="cuda"))
    s.step(3)
    assert s.integral() == pytest.approx(cfg.x1 - cfg.x0)
    s.close()
