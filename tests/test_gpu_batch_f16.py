"""FP16 runs of a batch against the same runs alone, bit for bit: the strips'
closed-form non-equilibrium moments in both band kernels."""
import numpy as np
import pytest

import lbm_workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice", ["D2Q9", "D2Q17", "D2Q37"])
@pytest.mark.parametrize("viscous", ["meso", "fd"])
def test_f16_runs_of_a_batch_are_bit_identical_to_runs_alone(lattice, viscous, tmp_path, monkeypatch):
    import paper_2307_16766_gb300 as lbm
    monkeypatch.setenv("LBM_AUTOTUNE_CACHE", str(tmp_path / "tune.txt"))
    cfgs, fields = [], []
    for k, (nx, ny, sides, dirichlet) in enumerate([
            (60, 45, ("cbc",) * 4, "eq"), (131, 40, ("inflow", "cbc", "periodic", "periodic"), "neep"),
            (37, 90, ("periodic", "periodic", "cbc", "cbc"), "reg"), (70, 33, ("periodic",) * 4, "eq")]):
        cfgs.append(W.run(lattice, nx, ny, 0.7 + 0.05 * k, storage="f16", sides=sides, schemes=("cbc_relax",) * 4,
                          viscous=viscous, dirichlet=dirichlet, alpha_T=0.3, beta_P=0.1, inflow=(1.0, 0.03, 0.0, 1.0)))
        fields.append(W.smooth_random(nx, ny, seed=4 + k, amp=1e-3, lattice=lattice, u0=(0.03, 0.01)))
    B = lbm.Batch(cfgs)
    for r, f in enumerate(fields):
        B[r].init_fields(*f)
    B.step(40)
    for r, (c, f) in enumerate(zip(cfgs, fields)):
        sim = lbm.Simulation(c).init_fields(*f).step(40)
        for name, x, y in zip(("rho", "ux", "uy", "T"), B[r].macros(), sim.macros()):
            assert np.all(np.isfinite(x)), (r, name)
            assert np.array_equal(x, y), (r, name, np.abs(x - y).max())
        sim.close()
    B.close()
