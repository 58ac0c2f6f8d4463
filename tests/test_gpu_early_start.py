"""Steps whose kernels start beside the previous step (one call of many steps)
against one call a step, which never starts early: the whole state bit for
bit, on grids of many waves of CTAs."""
import pytest

import lbm_workloads as W

pytestmark = pytest.mark.gpu

CBC, IN = ("cbc",) * 4, ("inflow", "cbc", "periodic", "periodic")
# the 37-, 17- and 9-velocity bands, with rows and segments that wrap, many
# tiles, an inflow, post-collision sources; and no side at all, per storage
CASES = [
    ("D2Q37", 700, 300, "f64", IN, "eq"), ("D2Q37", 516, 260, "f64", CBC, "neep"),
    ("D2Q17", 600, 400, "f64", CBC, "eq"), ("D2Q17", 200, 20, "f64", ("cbc", "cbc", "periodic", "periodic"), "neep"),
    ("D2Q9", 900, 700, "f64", ("periodic", "periodic", "cbc", "cbc"), "eq"),
    ("D2Q37", 640, 400, "f64", ("periodic",) * 4, "eq"), ("D2Q37", 1025, 700, "f32", ("periodic",) * 4, "eq"),
    ("D2Q37", 900, 801, "f16", ("periodic",) * 4, "eq"), ("D2Q37", 400, 300, "f32", ("inflow", "zg", "periodic", "periodic"), "eq"),
]


@pytest.mark.parametrize("lattice,nx,ny,storage,sides,dirichlet", CASES)
def test_many_steps_in_one_call_equal_one_step_a_call(lattice, nx, ny, storage, sides, dirichlet):
    import paper_2307_16766_gb300 as lbm
    cfg = W.run(lattice, nx, ny, 0.8, storage=storage, sides=sides, schemes=("cbc_relax",) * 4, dirichlet=dirichlet,
                viscous="meso", alpha_T=0.4, inflow=(1.0, 0.03, 0.0, 1.0))
    f = W.smooth_random(nx, ny, seed=9, amp=1e-3, lattice=lattice, u0=(0.03, 0.01))
    a = lbm.Simulation(cfg).init_fields(*f)
    b = lbm.Simulation(cfg).init_fields(*f)
    for n in (60, 1, 59):
        a.step(n)
        for _ in range(n):
            b.step(1)
        assert a.get_state() == b.get_state()
    a.macros()                              # no kernel gave a wait up
    a.close()
    b.close()


@pytest.mark.parametrize("storage,sides", [("f64", CBC), ("f64", ("periodic",) * 4), ("f32", ("periodic",) * 4)])
def test_captured_steps_equal_eager_ones(storage, sides):
    """Four steps captured in a graph (all but the first with early start) and
    replayed."""
    import numpy as np
    import torch
    import paper_2307_16766_gb300 as lbm
    cfg = W.run("D2Q37", 260, 120, 0.8, storage=storage, sides=sides, schemes=("cbc_relax",) * 4, alpha_T=0.4)
    f = W.smooth_random(260, 120, seed=9, amp=1e-3, u0=(0.03, 0.01))
    a = lbm.Simulation(cfg).init_fields(*f).step(4 * 25)
    want = a.macros()
    a.close()
    b = lbm.Simulation(cfg).init_fields(*f)
    torch.cuda.synchronize()
    s, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        lbm.lbm_set_stream(b.handle, s.cuda_stream)
        lbm.lbm_step(b.handle, 4)
    for _ in range(25):
        g.replay()
    torch.cuda.synchronize()
    lbm.lbm_set_stream(b.handle, torch.cuda.current_stream().cuda_stream)
    got = b.macros()
    b.close()
    for x, y in zip(want, got):
        assert np.array_equal(x, y)
