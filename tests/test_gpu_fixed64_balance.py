"""Mass, momentum and (thermal lattices) energy over one FP64 step, averaged
over the nodes, against the collision in extended precision (with the same FP64
weights, whose moments are exact to 1e-16 only): what is left is that of the
independent roundings of the stored values and nothing systematic.  A
systematic rest (of a few 1e-17 of the velocity) adds up over the steps of a
stream."""
import numpy as np
import pytest

import lbm_workloads as W
from test_gpu_fixed64 import LD, CLASSES, WEIGHTS, equilibrium, macros, planes, populations

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice,order", [("D2Q9", 2), ("D2Q17", 3), ("D2Q37", 4)])
@pytest.mark.parametrize("tau", [0.55, 0.9])
def test_a_step_leaves_the_mean_of_the_conserved_moments(lattice, order, tau):
    import paper_2307_16766_gb300 as lbm
    nx, ny = 130, 70
    cfg = W.run(lattice, nx, ny, tau, storage="f64", sides=("periodic",) * 4)
    rng = np.random.default_rng(11)
    r = [1e-3 * rng.standard_normal((ny, nx)) for _ in range(4)]
    sim = lbm.Simulation(cfg).init_fields(1 + r[0], 0.083 + r[1], -0.057 + r[2], 1 + r[3] * (order > 2))
    c = planes(lattice).astype(int)
    Q, om, eps = len(c), 1 / LD(tau), LD(2.0) ** -52
    w = np.array([dict(zip(CLASSES[lattice], WEIGHTS[lattice]))[tuple(sorted(map(abs, v), reverse=True))]
                  for v in c.tolist()]).astype(LD)
    old = populations(sim, cfg, Q).astype(LD)
    sim.step(1)
    got = populations(sim, cfg, Q).astype(LD)
    sim.close()
    g = np.array([np.roll(old[i], (c[i, 1], c[i, 0]), (0, 1)) for i in range(Q)])
    cs2 = LD(W.CS2[lattice]) if order > 2 else LD(1) / 3
    ge = equilibrium(macros(g, c, cs2, order > 2), c, w, cs2, order)
    d = (got - g - om * (ge - g)).reshape(Q, -1).mean(1)
    # g' = g + om (g^eq - g): g^eq, the difference and the result are rounded to
    # FP64, each uniformly within half a unit of at most 2^-52 of its value
    # (and so are the sums that the macros come from)
    var = (eps ** 2 / 12 * ((om * ge) ** 2 + (om * (ge - g)) ** 2 + got ** 2)).reshape(Q, -1).mean(1)
    kinds = {"mass": np.ones(Q), "momentum x": c[:, 0], "momentum y": c[:, 1]}
    if order > 2:
        kinds["energy"] = (c * c).sum(1)
    for name, k in kinds.items():
        total = (k[:, None, None] * g).sum(0)
        sigma = np.sqrt(((var * k ** 2).sum() + eps ** 2 / 12 * om ** 2 * (total ** 2).mean()) / (nx * ny))
        assert abs((d * k).sum()) <= 6 * sigma, (name, float((d * k).sum()), float(sigma))
