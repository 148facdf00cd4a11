"""Several solvers open at once: what one needs of a kernel that they share (its limit of shared
memory) leaves the others' launches as they were."""
import ctypes as C
import threading

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


@pytest.mark.parametrize("kind", ["run", "burgers"])
def test_two_streams_and_threads_side_by_side(kind):
    # cooperative runs that fill the chip, and Burgers steps launched as programmatic dependents,
    # each solver stepped by a thread of its own on a stream of its own
    cfgs = [adg.Config(pde="advection", K=65536, p=p, P=256, cfl=0.002, mode="at", L=5, q=2, seed=p) if kind == "run" else
            adg.Config(pde="burgers", K=40000, p=p, P=100, cfl=0.005, mode="at", L=4, q=2, seed=p) for p in (3, 2)]
    u0 = [torch.tensor(0.5 + 0.1 * random_nodal(c.K, c.p, 4), device="cuda") for c in cfgs]

    def steps(s):
        for _ in range(40):
            s.step(17)

    ref = []
    for c, u in zip(cfgs, u0):
        s = adg.Solver(c, u)
        steps(s)
        ref.append(s.state())
        s.close()
    torch.cuda.synchronize()
    solvers = [adg.Solver(c, u, stream=torch.cuda.Stream()) for c, u in zip(cfgs, u0)]
    for s in solvers:
        s.set_wait_limit(1 << 20)
    threads = [threading.Thread(target=steps, args=(s,)) for s in solvers]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for s, r in zip(solvers, ref):
        assert torch.equal(s.state(), r)
        s.close()
