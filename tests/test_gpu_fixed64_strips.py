"""Non-equilibrium moments (stress, heat flux) of the strip nodes with FP64
storage, summed in block fixed point, against extended precision."""
import numpy as np
import pytest

import lbm_workloads as W
from test_gpu_fixed64 import LD, CLASSES, WEIGHTS, equilibrium, macros, planes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice,order,M", [("D2Q9", 2, 1), ("D2Q17", 3, 3), ("D2Q37", 4, 3)])
@pytest.mark.parametrize("amp,u0", [(1e-3, (0.0, 0.0)), (1e-3, (0.08, 0.03)), (1e-6, (0.05, 0.0))])
def test_strip_moments_have_fp64_rounding(lattice, order, M, amp, u0):
    import paper_2307_16766_gb300 as lbm
    nx, ny, nxp, tau, th = 60, 40, 64, 0.8, order > 2
    cfg = W.run(lattice, nx, ny, tau, storage="f64", sides=("cbc", "cbc", "periodic", "periodic"),
                schemes=("cbc_relax",) * 4, viscous="meso", alpha_T=0.3)
    sim = lbm.Simulation(cfg).init_fields(*W.smooth_random(nx, ny, seed=3, amp=amp, lattice=lattice, u0=u0)).step(10)
    c = planes(lattice).astype(int)
    Q = len(c)
    w = np.array([dict(zip(CLASSES[lattice], WEIGHTS[lattice]))[tuple(sorted(map(abs, v), reverse=True))]
                  for v in c.tolist()]).astype(LD)
    cs2 = LD(W.CS2[lattice]) if th else LD(1) / 3
    old = np.frombuffer(sim.get_state(), np.float64, Q * ny * nxp, 80).reshape(Q, ny, nxp)[:, :, :nx].astype(LD)
    raw = sim.step(1).get_state()
    sim.close()
    # the strips of two sides, depths 0 .. M + 2, both parities: 4 macros, then 5 moments a node
    nslots = 2 * (3 + M) * ny
    N = np.frombuffer(raw, np.float64, 10 * nslots, 80 + 8 * Q * ny * nxp + 64 * nslots).reshape(2, nslots, 5)[1]
    got = N[M * ny:(M + 3) * ny].reshape(3 * ny, 5)             # W side, depths M .. M + 2
    g = np.concatenate([[np.roll(old[i], (c[i, 1], c[i, 0]), (0, 1))[:, 2 * M + d] for i in range(Q)] for d in range(3)], 1)
    s0, ux, uy, t = macros(g[:, None, :], c, cs2, th)
    d = g - equilibrium((s0, ux, uy, t), c, w, cs2, order)[:, 0, :]
    s0, ux, uy, t = s0[0], ux[0], uy[0], t[0]
    cx, cy, c2, fac = c[:, :1], c[:, 1:], (c * c).sum(1)[:, None], 1 - LD(0.5) / LD(tau)
    h = d * ((cx - ux) ** 2 + (cy - uy) ** 2) / 2 * th
    want = np.array([-fac * (cx * cx * d).sum(0), -fac * (cx * cy * d).sum(0), -fac * (cy * cy * d).sum(0),
                     fac * (h * (cx - ux)).sum(0), fac * (h * (cy - uy)).sum(0)]).T
    # operands are within half of 2^-58 of the node's largest, independently;
    # then each sum and each term of the closed form is rounded a few times
    e, rho, u2, gmax = LD(2.0) ** -53, 1 + s0, ux * ux + uy * uy, np.abs(g).max()
    q = [(c2 - 4 * cs2) * c[:, k:k + 1] for k in (0, 1)]
    se = (c2 * g).sum(0)
    stress = [cx * cx - cy * cy * th, cx * cy, cy * cy - cx * cx * th]
    size = [np.abs((k * g).sum(0)) + rho * u2 + (not th) * cs2 * np.abs(s0) for k in stress]
    heat = [np.abs((k * g).sum(0)) + rho * np.sqrt(u2) * (u2 + 4 * cs2 * np.abs(t) + 2 * (np.abs(se) + 2 * cs2 * np.abs(s0)))
            + np.sqrt(u2) * (size[0] + size[1]) for k in q]
    for j, (k, terms) in enumerate(zip(stress + q, size + heat)):
        rms = np.sqrt(((got[:, j] - want[:, j]) ** 2).mean())
        tol = e / 32 * gmax * np.sqrt((k.astype(LD) ** 2).sum() / 12) + 4 * e * np.sqrt((terms ** 2).mean())
        assert rms <= tol, (j, float(rms / e / gmax), float(tol / e / gmax))
