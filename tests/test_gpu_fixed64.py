"""FP64 bulk update and macroscopic fields, formed in block fixed point
(fix64.cuh), against extended-precision sums of the stored populations."""
import numpy as np
import pytest

import lbm_workloads as W
from test_gpu_macros import CLASSES, WEIGHTS, planes

pytestmark = pytest.mark.gpu
LD = np.longdouble


def populations(sim, cfg, Q):
    nx, ny = cfg["nx"], cfg["ny"]
    nxp = (nx + 63) // 64 * 64
    return np.frombuffer(sim.get_state(), np.float64, Q * ny * nxp, 80).reshape(Q, ny, nxp)[:, :, :nx]


def macros(g, c, cs2, thermal):
    cx, cy = c[:, 0, None, None], c[:, 1, None, None]
    s0, sx, sy, se = g.sum(0), (g * cx).sum(0), (g * cy).sum(0), (g * (cx * cx + cy * cy)).sum(0)
    rho = 1 + s0
    ux, uy = sx / rho, sy / rho
    t = (se - 2 * cs2 * s0 - rho * (ux * ux + uy * uy)) / (2 * cs2 * rho) if thermal else 0 * s0
    return s0, ux, uy, t


def equilibrium(m, c, w, cs2, order):
    """The Hermite expansion (Eqs. feq-3, feq-4) minus w rho0."""
    s0, ux, uy, t = m
    out = []
    for (cx, cy), wi in zip(c, w):
        p, q, u2 = (cx * ux + cy * uy) / cs2, (cx * cx + cy * cy) / cs2, (ux * ux + uy * uy) / cs2
        h = p + (p * p - u2 + t * (q - 2)) / 2 if order > 2 else p + (p * p - u2) / 2
        if order >= 3:
            h = h + p * (p * p - 3 * u2 + 3 * t * (q - 4)) / 6
        if order >= 4:
            h = h + (p ** 4 - 6 * p * p * u2 + 3 * u2 * u2 + 6 * t * (p * p * (q - 6) + u2 * (4 - q))
                     + 3 * t * t * (q * q - 8 * q + 8)) / 24
        out.append(wi * (s0 + (1 + s0) * h))
    return np.array(out)


@pytest.mark.parametrize("lattice,order", [("D2Q9", 2), ("D2Q17", 3), ("D2Q37", 4)])
@pytest.mark.parametrize("nx,ny", [(7, 7), (129, 9), (260, 17)])
@pytest.mark.parametrize("amp", [0.0, 1e-290, 1e-30, 1e-3, 0.1])
def test_fp64_step_and_fields(lattice, order, nx, ny, amp):
    import paper_2307_16766_gb300 as lbm
    sides = ("periodic",) * 4
    cfg = W.run(lattice, nx, ny, 0.8, storage="f64", sides=sides)
    rng = np.random.default_rng(3)
    r = [amp * rng.standard_normal((ny, nx)) / 4 for _ in range(4)]
    sim = lbm.Simulation(cfg).init_fields(1 + r[0], r[1], r[2], 1 + r[3] * (order > 2))
    c = planes(lattice).astype(int)
    Q = len(c)
    w = np.array([dict(zip(CLASSES[lattice], WEIGHTS[lattice]))[tuple(sorted(map(abs, v), reverse=True))]
                  for v in c.tolist()]).astype(LD)
    cs2 = LD(W.CS2[lattice])
    old = populations(sim, cfg, Q)
    sim.step(1)
    got = populations(sim, cfg, Q)
    fields = sim.macros()
    sim.close()
    g = np.array([np.roll(old[i], (c[i, 1], c[i, 0]), (0, 1)) for i in range(Q)]).astype(LD)
    m = macros(g, c, cs2, order > 2)
    want = g + (equilibrium(m, c, w, cs2, order) - g) / LD(0.8)
    # sums truncated at 2^-54 of twice the largest population: at most
    # 216 2^-53 gmax in sum g |c|^2, hence 300 2^-53 gmax in theta, which
    # enters g^eq / w with a factor up to 11 (|c|^2 / (2 c_s^2)), and less
    # from the momentum; FP64 roundings of the stored values on top
    gmax, eps = np.abs(g).max(), LD(2.0) ** -53
    for i in range(Q):
        tol = eps * (4 * np.abs(want[i]).max() + 8192 * w[i] * gmax) + LD(2.0) ** -1060
        assert np.abs(got[i] - want[i]).max() <= tol, (i, np.abs(got[i] - want[i]).max(), tol)
    f = macros(got.astype(LD), c, cs2, order > 2)
    tol = 1024 * eps * np.abs(got).max() + LD(2.0) ** -1060
    for a, b in ((fields[0], 1 + f[0]), (fields[1], f[1]), (fields[2], f[2]), (fields[3], 1 + f[3])):
        assert np.abs(a - b).max() <= tol + (2 * eps if np.abs(b).max() > 0.5 else 0)
