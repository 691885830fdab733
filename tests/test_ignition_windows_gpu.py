"""Growing ignition windows and drip torches at given times, in both forms of the
kernel (every segment at every node; segments bounded over tiles) and both
precisions: psi and the ignition times against a per-node, per-segment
evaluation in 64 bits, rounded once.  The step that follows the ignition in
fire_step is 1e-9 s long: it moves psi by less than 1e-9 times 30 m/s."""
import numpy as np
import pytest

from gpu_helpers import state_np
from paper_1102_1343_gb300 import synth

pytestmark = pytest.mark.gpu


def ignited(w, t, psi, tign, real):
    y, x = np.indices(psi.shape)
    x, y = (x + 0.5) * w.dx, (y + 0.5) * w.dy
    psi, tign = psi.copy(), tign.copy()
    close = np.abs(psi) < 1e-6  # rims: rounding decides
    for g in w.ignitions:
        R = g["speed"] * (t - g["t_start"])
        bx, by, tt = g["bx"], g["by"], t
        if "vx" in g:
            if not g["t_start"] <= t <= g["t_end"] + g["radius"] / g["speed"]:
                continue
            tt = min(t, g["t_end"])
            bx, by = g["ax"] + g["vx"] * (tt - g["t_start"]), g["ay"] + g["vy"] * (tt - g["t_start"])
            R = min(R, g["radius"])
        elif not g["t_start"] <= t <= g["t_start"] + g["radius"] / g["speed"]:
            continue
        dx, dy = bx - g["ax"], by - g["ay"]
        l2 = dx * dx + dy * dy
        u = np.clip(((x - g["ax"]) * dx + (y - g["ay"]) * dy) / l2, 0, 1) if l2 > 0 else np.zeros_like(x)
        d = np.hypot(x - g["ax"] - u * dx, y - g["ay"] - u * dy)
        new = (psi > 0) & (d - R <= 0) & np.isinf(tign)
        ta = g["t_start"] + u * (tt - g["t_start"]) + d / g["speed"] if "vx" in g else g["t_start"] + d / g["speed"]
        tign[new] = np.minimum(ta, t)[new] if "vx" in g else ta[new]
        close |= np.abs(d - R) < 1e-6
        psi = np.minimum(psi, (d - R).astype(real))
    return psi, tign, close


# nodes and segments on both sides of the line between the two forms, ragged tiles
@pytest.mark.parametrize("mesh,lines,torches", [
    ((7, 3, 9), 3, 2), ((13, 9, 5), 60, 10), ((33, 17, 7), 90, 10), ((25, 12, 10), 63, 1), ((26, 12, 10), 63, 1),
    ((40, 25, 10), 3, 4), ((40, 25, 10), 4, 4), ((41, 40, 7), 120, 10)])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_growing_windows(mesh, lines, torches, prec):
    from paper_1102_1343_gb300 import build
    build.build()
    import paper_1102_1343_gb300 as pkg
    nxa, nya, sr = mesh
    rng = np.random.default_rng(nxa + lines)
    w = synth.random_landscape(nxa, nya, sr=sr, dx_atm=6.0 * sr, seed=4, ignition="none", steps=1)
    Lx, Ly = w.nx * w.dx, w.ny * w.dy
    at = lambda: (rng.uniform(0, Lx), rng.uniform(0, Ly))
    w.ignitions = [synth.line_ignition(*at(), *at(), radius=9.0, t_start=0.02 * k, speed=1.5) for k in range(lines - 1)]
    w.ignitions += [synth.point_ignition(*at(), radius=30.0, t_start=0.1, speed=4.0)]
    w.ignitions += [synth.drip_torch(*at(), rng.uniform(-3, 3), 1.0, 0.2 * k, 4.0, 5.0, 2.0) for k in range(torches)]
    real = np.float64 if prec == "fp64" else np.float32
    m = pkg.FireModel.from_workload(w, precision=prec)
    y, x = np.indices((w.ny, w.nx))
    psi0 = (25 + 30 * np.sin(x * 0.18) * np.cos(y * 0.15)).astype(real)
    t0 = np.where(psi0 <= 0, -5.0, np.inf)
    u, v = m.wind(w.u, w.v)
    T = m.torch.as_tensor
    for t in (0.3, 2.6, 5.5):
        m.set_state(T(psi0).cuda(), T(t0).cuda(), T(np.ones_like(psi0)).cuda(), t)
        m.step(u, v, 1e-9)
        psi, tign, _, _ = state_np(m)
        ref, tref, close = ignited(w, t, psi0, t0, real)
        assert (ref != psi0).any() and (tref != t0).any()
        assert np.abs(psi - ref).max() <= 3e-8 + 2 * np.finfo(real).eps * np.abs(ref).max()
        ok = ~close
        assert np.array_equal(np.isfinite(tign)[ok], np.isfinite(tref)[ok])
        f = ok & np.isfinite(tref)
        assert np.abs(tign[f] - tref[f]).max() <= 1e-12 * max(Lx, Ly)
    m.close()
