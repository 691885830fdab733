"""Where the FP64 kernels decide branches on the bits of a number: a spread rate
whose sum is negative is S0, a wind that is not a number counts as none, and a
node whose psi is not a number (of either sign) gets no ignition time and burns
no fuel around it."""
import dataclasses

import numpy as np
import pytest

import oracle
from paper_1102_1343_gb300 import synth

pytestmark = pytest.mark.gpu

KERNELS = ["TILE1", "TILE", "MARCH", "WARP"]


@pytest.fixture(scope="module")
def pkg():
    from paper_1102_1343_gb300 import build
    build.build()
    import paper_1102_1343_gb300 as p
    p.load_library()
    return p


def landscape(nxa=8, nya=7, **kw):
    w = synth.random_landscape(nxa, nya, sr=10, dx_atm=60.0, seed=9, ignition="center", steps=6, dt=0.5)
    return dataclasses.replace(w, **kw)


def model(pkg, w, prec, kernel):
    m = pkg.FireModel.from_workload(w, precision=prec)
    shape = {"TILE1": (pkg.FIRE_KERNEL_TILE, 1, 1), "TILE": (pkg.FIRE_KERNEL_TILE, 4, 3) if prec == "fp64" else (pkg.FIRE_KERNEL_TILE, w.nxa, w.nya),
             "MARCH": (pkg.FIRE_KERNEL_MARCH, w.nxa, 2), "WARP": (pkg.FIRE_KERNEL_WARP, 6, 2)}[kernel]
    pkg.fire_set_kernel(m.ctx, *shape)
    return m


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("kernel", KERNELS)
def test_negative_sum_gives_S0(pkg, kernel, prec):
    w = landscape(classes=[dict(synth.nominal_class(), cmbcnst=-18.6e6)], fuel=np.zeros((70, 80), np.uint8))
    m = model(pkg, w, prec, kernel)
    u, v = m.wind(w.u, w.v)
    before = m.state()[0]
    m.run(4, u, v, w.dt)
    assert m.torch.equal(before, m.state()[0])  # S0 is 0
    m.close()


def test_negative_sum_in_the_adjoint(pkg):
    """Stripes of a class that does not spread (its sum is negative) beside
    burning ones: gradients against the oracle's reference adjoint."""
    good = synth.nominal_class(fgi=0.5)
    y, x = np.indices((70, 80))
    w = landscape(classes=[good, dict(good, cmbcnst=-18.6e6)], fuel=((x // 4) % 3 == 2).astype(np.uint8))
    w = dataclasses.replace(w, ignitions=[synth.point_ignition(240.0, 210.0, radius=20.0)], mult=np.full((70, 80), 10.0))
    tobs = np.where((x - 40) ** 2 + (y - 35) ** 2 < 100, 2.0, np.nan)
    Jr, *ref = oracle.OracleFire.from_workload(w).adjoint(w.u, w.v, w.dt, w.steps, tobs)
    m = pkg.FireModel.from_workload(w, precision="fp64")
    u, v = m.wind(w.u, w.v)
    J, *g = m.adjoint(u, v, w.dt, w.steps, tobs, ckpt_every=2)
    assert np.abs(ref[0]).max() > 0 and abs(J - Jr) <= 1e-10 * Jr
    for a, b in zip(g, ref):
        a = a.cpu().numpy()
        assert np.linalg.norm(a - b) <= 1e-8 * np.linalg.norm(b)
    m.close()


@pytest.mark.parametrize("kernel", KERNELS)
def test_wind_that_is_not_a_number_counts_as_none(pkg, kernel):
    w = landscape()
    psi = []
    for wind in (np.nan, -np.nan, 0.0):
        m = model(pkg, w, "fp64", kernel)
        u, v = m.wind(np.full_like(w.u, wind), np.full_like(w.v, wind))
        m.step(u, v, w.dt)
        psi.append(m.state()[0].cpu().numpy())
        assert m.status() == (pkg.FIRE_OK if wind == 0.0 else pkg.FIRE_ERR_NONFINITE)
        m.close()
    assert np.array_equal(psi[0], psi[2]) and np.array_equal(psi[1], psi[2])


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("kernel", KERNELS)
def test_psi_that_is_not_a_number(pkg, kernel, sign, prec):
    w = landscape(ignitions=[])
    m = model(pkg, w, prec, kernel)
    torch = m.torch
    psi, tign, frac, _ = m.state()
    psi.fill_(50.0)
    bad = torch.copysign(torch.tensor(float("nan"), dtype=m.dtype), torch.tensor(sign, dtype=m.dtype))
    for y, x in ((30, 40), (0, 0), (69, 79), (35, 0), (20, 59), (20, 60)):
        psi[y, x] = bad
    m.set_state(psi, tign, frac, 0.0)
    u, v = m.wind(w.u, w.v)
    m.step(u, v, w.dt)
    psi, tign, frac, _ = m.state()
    assert torch.isinf(tign).all()
    assert (frac[torch.isfinite(psi)] == 1).all()
    assert m.status() == pkg.FIRE_ERR_NONFINITE
    m.close()
