"""Macroscopic fields of FP32 and FP16 populations against FP64 sums of the
stored values (Eq. macro), read back with lbm_get_state."""
import math

import numpy as np
import pytest

import lbm_workloads as W

pytestmark = pytest.mark.gpu

# velocity classes (|c_x|, |c_y|) with c_x >= c_y, in the order of the weights
CLASSES = {"D2Q9": [(0, 0), (1, 0), (1, 1)], "D2Q17": [(0, 0), (1, 0), (1, 1), (2, 2), (3, 0)],
           "D2Q37": [(0, 0), (1, 0), (1, 1), (2, 0), (2, 1), (2, 2), (3, 0), (3, 1)]}


def planes(lattice):
    """Velocities in storage order: groups c_y = 0, 1, -1, ...; inside a group
    c_x = 0, then opposite values, the sign of c_y first."""
    out = []
    for cy in (0, 1, -1, 2, -2, 3, -3):
        for a in range(4):
            if tuple(sorted((a, abs(cy)), reverse=True)) in CLASSES[lattice]:
                s = -1 if cy < 0 else 1
                out += [(0, cy)] if a == 0 else [(s * a, cy), (-s * a, cy)]
    return np.array(out, dtype=np.float64)


def fp64_macros(sim, cfg, w):
    c = planes(cfg["lattice"])
    nx, ny, Q = cfg["nx"], cfg["ny"], len(c)
    nxp = (nx + 63) // 64 * 64
    dt = {"f32": np.float32, "f16": np.float16}[cfg["storage"]]
    raw = sim.get_state()
    head = 80                                   # magic, 5 ints (padded), steps, 3 sizes, u_ref
    g = np.frombuffer(raw, dt, Q * ny * nxp, head).astype(np.float64).reshape(Q, ny, nxp)[:, :, :nx]
    if cfg["storage"] == "f16":
        g = g * np.array([w[tuple(sorted(map(abs, v), reverse=True))] for v in c.astype(int).tolist()])[:, None, None]
    cs2, cx, cy = W.CS2[cfg["lattice"]], c[:, 0, None, None], c[:, 1, None, None]
    Ux, Uy = (float(np.float32(v)) for v in cfg["u_ref"])
    s0, sx, sy, se = g.sum(0), (g * cx).sum(0), (g * cy).sum(0), (g * (cx * cx + cy * cy)).sum(0)
    rho = 1.0 + s0
    vx, vy = (sx - s0 * Ux) / rho, (sy - s0 * Uy) / rho
    t = (se - 2 * cs2 * s0 - s0 * (Ux * Ux + Uy * Uy) - rho * (2 * (Ux * vx + Uy * vy) + vx * vx + vy * vy)) / (2 * cs2 * rho)
    scale = np.abs(g * (1.0 + cx * cx + cy * cy)).sum(0).max() + abs(Ux) + abs(Uy)
    return (rho, vx + Ux, vy + Uy, 1.0 + t * (cfg["lattice"] != "D2Q9")), scale


WEIGHTS = {"D2Q9": [4 / 9, 1 / 9, 1 / 36],
           "D2Q17": [0.4020051469091126259416644, 0.1161548664977815438740355, 0.0330063536229869139497538,
                     0.0000790786021659181312371, 0.0002584145497874675595575],
           "D2Q37": [0.23315066913235250229, 0.10730609154221900241, 0.05766785988879488203, 0.014208216158450750265,
                     0.0053530490005137752327, 0.0010119375926735754754, 0.00024530102775771734547,
                     0.0002834142529941982174]}


@pytest.mark.parametrize("lattice", ["D2Q9", "D2Q17", "D2Q37"])
@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("nx,ny,u", [(3, 3, 0.0), (129, 5, 0.0), (257, 33, 0.05)])
def test_macros_equal_the_fp64_sums(lattice, storage, nx, ny, u):
    import paper_2307_16766_gb300 as lbm
    cfg = W.run(lattice, nx, ny, 0.8, storage=storage, u_ref=(u, -0.5 * u))
    fields = W.smooth_random(nx, ny, 5, amp=2e-2, lattice=lattice, u0=(0.05, 0.02))
    sim = lbm.Simulation(cfg).init_fields(*fields).step(3)
    got = sim.macros()
    want, scale = fp64_macros(sim, cfg, dict(zip(CLASSES[lattice], WEIGHTS[lattice])))
    # float-float sums: ~40 accumulations of relative error 2^-47 each, then
    # a handful of products and one reciprocal; 1 / (2 c_s^2) < 1.6
    tol = 64 * 2.0 ** -47 * 2 * scale + 4e-16
    for a, b in zip(got, want):
        assert np.abs(a - b).max() <= tol, (np.abs(a - b).max(), tol)
    sim.close()


@pytest.mark.parametrize("storage", ["f32", "f16"])
def test_macros_of_values_beyond_the_float_products(storage):
    """Finite populations whose float products would overflow still give the
    FP64 result, and non-finite ones are reported."""
    import paper_2307_16766_gb300 as lbm
    big = 1e25 if storage == "f32" else 1e4
    cfg = W.run("D2Q9", 40, 8, 0.8, storage=storage)
    rho, ux, uy, T = W.uniform(40, 8, rho=1.0 + big)
    sim = lbm.Simulation(cfg).init_fields(rho, ux, uy, T)
    got = sim.macros()
    assert np.allclose(got[0], 1.0 + big, rtol=1e-3) and np.abs(got[1]).max() < 1e-3
    sim.init_fields(np.full_like(rho, math.inf), ux, uy, T)
    with pytest.raises(lbm.LbmError):
        sim.macros()
    sim.close()
