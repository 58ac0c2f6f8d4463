"""Macroscopic fields of arbitrary FP32 and FP16 populations (Eq. macro) to
FP64 rounding, against extended-precision sums of the stored values."""
import numpy as np
import pytest

import lbm_workloads as W
from test_gpu_macros import CLASSES, WEIGHTS, planes

pytestmark = pytest.mark.gpu
LD = np.longdouble


@pytest.mark.parametrize("lattice", ["D2Q9", "D2Q17", "D2Q37"])
@pytest.mark.parametrize("spread", [0, 6])              # magnitudes of one node over 2^spread either way
@pytest.mark.parametrize("storage,u,scale", [
    ("f32", 0.0, 0), ("f32", 0.05, 0), ("f16", 0.0, 0), ("f16", 0.05, 0),
    ("f32", 0.0, -66), ("f32", 0.0, -140)])             # far below the usual range, into the denormals
def test_fields_have_fp64_rounding(lattice, storage, spread, u, scale):
    import paper_2307_16766_gb300 as lbm
    nx, ny = 131, 9
    cfg = W.run(lattice, nx, ny, 0.8, storage=storage, u_ref=(u, -0.5 * u))
    c = planes(lattice).astype(int)
    Q, nxp, dt = len(c), (nx + 63) // 64 * 64, {"f32": np.float32, "f16": np.float16}[storage]
    w = np.array([dict(zip(CLASSES[lattice], WEIGHTS[lattice]))[tuple(sorted(map(abs, v), reverse=True))]
                  for v in c.tolist()]).astype(LD)[:, None, None]
    sim = lbm.Simulation(cfg).init_fields(*W.uniform(nx, ny))
    raw = bytearray(sim.get_state())
    rng = np.random.default_rng(Q + spread)
    # nodes of their own scale (density up to 1.1), populations held as g or g / w
    h = 0.1 * rng.standard_normal((Q, ny, nxp)) * 2.0 ** rng.uniform(-spread, 0, (Q, ny, nxp))
    h = h * 2.0 ** rng.uniform(scale - 10, scale, (1, ny, nxp)) * (1.0 if storage == "f16" else w.astype(float))
    raw[80:80 + h.size * np.dtype(dt).itemsize] = h.astype(dt).tobytes()
    sim.set_state(bytes(raw))
    got = sim.macros()
    sim.close()
    g = h.astype(dt).astype(LD)[:, :, :nx] * (w if storage == "f16" else 1)
    cx, cy, cs2 = c[:, 0, None, None], c[:, 1, None, None], LD(W.CS2[lattice])
    Ux, Uy = (LD(np.float32(v)) for v in cfg["u_ref"])
    s0, sx, sy, se = g.sum(0), (g * cx).sum(0), (g * cy).sum(0), (g * (cx * cx + cy * cy)).sum(0)
    rho = 1 + s0
    vx, vy = (sx - s0 * Ux) / rho, (sy - s0 * Uy) / rho
    k = s0 * (Ux * Ux + Uy * Uy) + rho * (2 * (Ux * vx + Uy * vy) + vx * vx + vy * vy)
    t = (se - 2 * cs2 * s0 - k) / (2 * cs2 * rho) * (lattice != "D2Q9")
    # each sum is rounded once (operands at 2^-57 of the node's largest, the
    # weights of g / w at 2^-65 and 2^-54), then a handful of FP64 operations,
    # each 2^-53 of a term; |c| <= 3
    e = LD(2.0) ** -53
    big = np.abs(g / (w if storage == "f16" else 1)).max(0) * (1 if storage == "f16" else Q)
    term = np.abs(s0) + np.abs(sx) + np.abs(sy) + (np.abs(Ux) + np.abs(Uy)) * (1 + np.abs(s0))
    tol = [2 * e * (1 + np.abs(s0)) + e * big] + [8 * e * (term + big)] * 2 + \
        [e + 8 * e * (big + np.abs(se) + 2 * cs2 * np.abs(s0) + term ** 2) / (2 * cs2)]
    for n, a, b, x in zip(("rho", "ux", "uy", "T"), got, (rho, vx + Ux, vy + Uy, 1 + t), tol):
        assert (np.abs(a - b) <= x).all(), (n, float((np.abs(a - b) / x).max()))
