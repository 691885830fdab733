"""Edges of the element-wise kernels: ignition tiles (64 x 16 nodes) at every
remainder, with segments that cover, border on or miss a tile and more of them
than one launch takes; heat insertion over layer counts around a thread's
four, with columns without a fire beside burning ones; the heat adjoint's ghost
gather on meshes whose outer rings overlap and with fire at every edge."""
import dataclasses

import numpy as np
import pytest

import oracle
from gpu_helpers import compare_fp64, state_np
from paper_1102_1343_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    from paper_1102_1343_gb300 import build
    build.build()
    import paper_1102_1343_gb300 as p
    p.load_library()
    return p


@pytest.mark.parametrize("mesh", [(2, 2, 1), (7, 3, 9), (13, 9, 5), (16, 4, 4), (33, 17, 7)])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_ignition_tiles(pkg, mesh, prec):
    """The state after fire_init with 150 instantaneous points and lines, and
    after steps inside 90 growing windows and torches, against the oracle: the
    level set to 1e-12 (FP32: one rounding of the distances), the same nodes
    ignited and their times to 1e-12."""
    nxa, nya, sr = mesh
    rng = np.random.default_rng(nxa * 10 + sr)
    dx = 6.0
    nx, ny = nxa * sr, nya * sr
    Lx, Ly = nx * dx, ny * dx
    at = lambda: (rng.uniform(0, Lx), rng.uniform(0, Ly))
    now = [synth.point_ignition(*at(), radius=rng.uniform(1, 15)) for _ in range(75)]
    now += [synth.line_ignition(*at(), *at(), radius=rng.uniform(0.1, 4), t_start=-float(k)) for k in range(75)]
    grow = [synth.line_ignition(*at(), *at(), radius=6.0, t_start=0.1 * k, speed=1.5) for k in range(80)]
    grow += [synth.drip_torch(*at(), rng.uniform(-3, 3), 1.0, 0.2 * k, 8.0, 5.0, 2.0) for k in range(10)]
    w = synth.random_landscape(nxa, nya, sr=sr, dx_atm=dx * sr, seed=4, ignition="none", steps=20, dt=0.25)
    for ign, steps in ((now, 0), (grow, 20)):
        w = dataclasses.replace(w, ignitions=ign)
        m = pkg.FireModel.from_workload(w, precision=prec)
        orc = oracle.OracleFire.from_workload(w)
        u, v = m.wind(w.u, w.v)
        for _ in range(steps):
            m.step(u, v, w.dt)
            orc.step(w.u, w.v, w.dt)
        psi, tign, frac, _ = state_np(m)
        if prec == "fp64":
            ok, e = compare_fp64((psi, tign, frac, 0.0), orc, tol=1e-12 if steps == 0 else 1e-10)
            assert ok, e
        elif steps == 0:
            # psi: the distance rounded once; a node lies within rounding of the rim or agrees
            assert np.abs(psi - orc.psi).max() <= 6e-8 * np.abs(orc.psi).max()
            assert np.array_equal(np.isfinite(tign), np.isfinite(orc.tign))
            f = np.isfinite(tign)
            assert np.abs(tign[f] - orc.tign[f]).max(initial=0) <= 1e-12 * 80
        m.close()


@pytest.mark.parametrize("nz", [1, 3, 4, 5, 20])
@pytest.mark.parametrize("ncols", [1, 127, 300])
def test_heat_insertion_layers(pkg, nz, ncols):
    import torch
    rng = np.random.default_rng(nz * 1000 + ncols)
    zw, _, _, _ = synth.atmos_columns(rng, (ncols,), nz=nz, top=400.0)
    rho, mu = synth.air_columns(rng, (ncols,), zw)
    hs = np.where(rng.uniform(size=ncols) < 0.3, rng.uniform(1e3, 1e5, ncols), 0.0)
    hl = np.where(rng.uniform(size=ncols) < 0.3, rng.uniform(1e3, 1e5, ncols), 0.0)
    rth0, rqv0 = rng.standard_normal((2, nz, ncols))
    bad = ncols // 2
    rho[0, bad] = np.nan  # reported as before, also where nothing burns
    hs[bad] = 0.0
    d = lambda a: torch.as_tensor(np.ascontiguousarray(a)).cuda()
    rth, rqv = d(rth0), d(rqv0)
    pkg.fire_heat_insertion(d(hs), d(hl), d(zw), d(rho), d(mu), 50.0, rth, rqv)
    S = (np.exp(-zw[:-1] / 50.0) - np.exp(-zw[1:] / 50.0)) / (zw[1:] - zw[:-1])
    for got, f, base, c in ((rth, hs, rth0, 1004.0), (rqv, hl, rqv0, 2.5e6)):
        add = mu * f / (c * rho) * S
        got = got.cpu().numpy()
        assert np.isnan(got[0, bad]) and np.isnan(got).sum() == 1
        fin = np.isfinite(got)
        assert np.abs(got - (base + add))[fin].max(initial=0) <= 1e-13 * (np.abs(base) + np.abs(add))[fin].max(initial=0)
        assert np.array_equal(got[:, f == 0][fin[:, f == 0]], base[:, f == 0][fin[:, f == 0]])


@pytest.mark.parametrize("mesh", [(2, 2, 1), (3, 2, 1), (2, 3, 2), (3, 4, 1), (6, 5, 3)])
def test_heat_adjoint_ghost_rings(pkg, mesh):
    """Meshes of 2 to 18 nodes a side, burning at every edge: FP64 gradients of
    the heat misfit against the oracle's reference adjoint."""
    nxa, nya, sr = mesh
    w = synth.random_landscape(nxa, nya, sr=sr, dx_atm=10.0 * sr, seed=17, ignition="none", steps=6, dt=0.25)
    rng = np.random.default_rng(3)
    w = dataclasses.replace(w, mult=np.full((w.ny, w.nx), 2.0),
                            ignitions=[synth.point_ignition(x * w.nx * 10.0, y * w.ny * 10.0, radius=6.0)
                                       for x, y in ((0.02, 0.1), (0.95, 0.9), (0.9, 0.05))])
    qobs = rng.uniform(0.0, 1e5, (nya, nxa))
    Jr, *ref = oracle.OracleFire.from_workload(w).adjoint_heat(w.u, w.v, w.dt, w.steps, qobs)
    m = pkg.FireModel.from_workload(w, precision="fp64")
    u, v = m.wind(w.u, w.v)
    J, *g = m.adjoint_heat(u, v, w.dt, w.steps, qobs, ckpt_every=2)
    assert abs(J - Jr) <= 1e-10 * abs(Jr)
    for a, b in zip(g, ref):
        a = a.cpu().numpy()
        assert np.linalg.norm((a - b).ravel()) <= 1e-8 * max(np.linalg.norm(b.ravel()), 1e-300)
    m.close()
