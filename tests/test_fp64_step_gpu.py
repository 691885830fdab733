"""The FP64 right-hand side (its own square roots, reciprocals and power) and
the tile kernel's two forms (wind from tables of the tile, wind per node for
tiles too large for them) against the oracle, norm-wise 1e-10: unequal node
distances, winds of zero and far outside the fast range of the power, a
chaparral class; refinement 1, a single atmospheric row, tiles cut by the
mesh.  In FP32 both forms of the tile kernel give the same bits."""
import dataclasses

import numpy as np
import pytest

import oracle
from gpu_helpers import compare_fp64, state_np
from paper_1102_1343_gb300 import synth

pytestmark = pytest.mark.gpu

# atmospheric cells x, y, refinement x, y, a tile too large for the tables
MESHES = [(41, 45, 1, 1, (41, 41)), (1, 5, 10, 10, (1, 5)), (9, 1, 7, 5, (9, 1)),
          (6, 7, 10, 6, (6, 7)), (3, 2, 23, 31, (3, 2))]


def workload(mesh, wind):
    nxa, nya, srx, sry, _ = mesh
    dx, dy = 6.0, 8.5
    nx, ny = nxa * srx, nya * sry
    rng = np.random.default_rng(7 * nx + ny)
    w = synth.random_landscape(nxa, nya, sr=1, seed=3, ignition="none", steps=12)
    zx, zy = synth.hills_gradient(rng, nx, ny, dx, dy)
    fires = [synth.point_ignition(0.5 * nx * dx, 0.5 * ny * dy, radius=0.3 * min(nx * dx, ny * dy)),
             synth.point_ignition(0.9 * nx * dx, 0.1 * ny * dy, radius=12.0)]
    return dataclasses.replace(w, srx=srx, sry=sry, dx_atm=dx * srx, dy_atm=dy * sry, dt=0.25,
                               fuel=synth.voronoi_fuel(rng, nx, ny, dx, n_sites=20), dzdx=zx, dzdy=zy,
                               u=w.u * wind, v=w.v * wind, ignitions=fires)


def run(w, prec, var, kx, ky):
    import torch

    import paper_1102_1343_gb300 as pkg
    m = pkg.FireModel.from_workload(w, precision=prec)
    pkg.fire_set_kernel(m.ctx, var, kx, ky)
    u, v = m.wind(w.u, w.v)
    for _ in range(w.steps):
        hs, hl = m.step(u, v, w.dt)
    torch.cuda.synchronize()
    out = state_np(m) + (hs.cpu().numpy(), hl.cpu().numpy())
    m.close()
    return out


@pytest.mark.parametrize("mesh", MESHES)
@pytest.mark.parametrize("wind", [1.0, 0.0, 1e-30])
def test_fp64_step_against_oracle(mesh, wind):
    from paper_1102_1343_gb300 import build
    build.build()
    import paper_1102_1343_gb300 as pkg
    nxa, nya, srx, sry, big = mesh
    w = workload(mesh, wind)
    orc = oracle.OracleFire.from_workload(w)
    for _ in range(w.steps):
        orc.step(w.u, w.v, w.dt)
    kx = 60 // srx
    kx -= (kx * srx) % 2
    shapes = [(pkg.FIRE_KERNEL_TILE, 1, 1), (pkg.FIRE_KERNEL_TILE,) + big]
    if kx:
        shapes += [(pkg.FIRE_KERNEL_MARCH, kx, 2), (pkg.FIRE_KERNEL_WARP, kx, 2)]
    for var, kx, ky in shapes:
        ok, e = compare_fp64(run(w, "fp64", var, kx, ky)[:4], orc)
        assert ok, (var, kx, ky, e)
    a, b = (run(w, "fp32", pkg.FIRE_KERNEL_TILE, *k) for k in ((1, 1), big))
    for x, y in zip(a[:3] + a[4:], b[:3] + b[4:]):
        assert np.array_equal(x, y)
