"""FP64 batches with periodic axes: the persistent bulk kernel's work items
alternate between tensor copies and plain stores into one staging buffer."""
import numpy as np
import pytest

import lbm_workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice,sizes", [
    # more work items (128-node row segments) than the 5 CTAs per SM take at once
    ("D2Q37", [(260, 420), (128, 700), (389, 151)]),
    ("D2Q17", [(300, 400), (515, 260)]),
    ("D2Q9", [(385, 640), (64, 900)]),
])
def test_periodic_f64_runs_of_a_batch_are_bit_identical_to_runs_alone(lattice, sizes, tmp_path, monkeypatch):
    import paper_2307_16766_gb300 as lbm
    monkeypatch.setenv("LBM_AUTOTUNE_CACHE", str(tmp_path / "tune.txt"))
    cfgs, fields = [], []
    for k, (nx, ny) in enumerate(sizes):
        # periodic in x and y, and in one axis only (wrapped rows, wrapped segments)
        sides = [("periodic",) * 4, ("zg", "zg", "periodic", "periodic"), ("periodic", "periodic", "zg", "zg")][k % 3]
        cfgs.append(W.run(lattice, nx, ny, 0.6 + 0.1 * k, storage="f64", sides=sides, viscous="off"))
        fields.append(W.smooth_random(nx, ny, seed=20 + k, amp=1e-3, lattice=lattice, u0=(0.03, -0.02)))
    B = lbm.Batch(cfgs)
    for r, f in enumerate(fields):
        B[r].init_fields(*f)
    B.step(100)
    for r, (c, f) in enumerate(zip(cfgs, fields)):
        sim = lbm.Simulation(c).init_fields(*f)
        for _ in range(100):
            sim.step(1)
        for name, x, y in zip(("rho", "ux", "uy", "T"), B[r].macros(), sim.macros()):
            assert np.all(np.isfinite(x)), (r, name)
            assert np.array_equal(x, y), (r, name, np.abs(x - y).max())
        sim.close()
    B.close()
