"""The warp kernel (a CTA of four warps marching down a strip, a row per warp
and stage) against the four-column warp kernel, which computes every node with
the same operations in another order of rows and lanes: the same bits for psi,
t_i, F and both heat grids, at the strip heights where its stages run in, run
out and end bands (one band, several bands per iteration, bands of more rows
than any other test, strips cut into several CTAs, the launch's own height),
on even and odd widths, inside the mesh and along every edge of it."""
import dataclasses

import numpy as np
import pytest

from gpu_helpers import node_moisture, state_np
from paper_1102_1343_gb300 import synth

pytestmark = pytest.mark.gpu

# atmospheric cells x, y, refinement x, y
MESHES = [(23, 1, 10, 10), (13, 40, 10, 10), (47, 9, 5, 7), (14, 3, 12, 40), (5, 2, 20, 130),
          (121, 37, 2, 1), (33, 33, 4, 3), (19, 27, 9, 5)]


@pytest.mark.parametrize("mesh", MESHES)
@pytest.mark.parametrize("extra", ["plain", "mult", "moisture"])
def test_row_strips_equal_four_column_strips(mesh, extra):
    import torch

    from paper_1102_1343_gb300 import build
    build.build()
    import paper_1102_1343_gb300 as pkg
    nxa, nya, srx, sry = mesh
    dx = 6.0
    nx, ny = nxa * srx, nya * sry
    rng = np.random.default_rng(nx * 1000 + ny)
    w = synth.random_landscape(nxa, nya, sr=1, seed=12, ignition="none", steps=25)
    zx, zy = synth.hills_gradient(rng, nx, ny, dx, dx)
    fires = [synth.point_ignition(x * nx * dx, y * ny * dx, radius=r) for x, y, r in
             ((0.5, 0.5, 30.0), (0.04, 0.9, 20.0), (0.97, 0.08, 25.0), (0.7, 0.97, 15.0))]
    w = dataclasses.replace(w, srx=srx, sry=sry, dx_atm=dx * srx, dy_atm=dx * sry, dt=0.25,
                            fuel=synth.voronoi_fuel(rng, nx, ny, dx, n_sites=60), dzdx=zx, dzdy=zy,
                            ignitions=fires)
    if extra != "plain":
        w.mult = rng.uniform(0.7, 1.3, (ny, nx))
    if extra == "moisture":
        w = node_moisture(w)
    kx = 60 // srx
    kx -= (kx * srx) % 2
    runs = []
    for var, k, ky in ((pkg.FIRE_KERNEL_WARP4, max(1, 120 // srx - (120 // srx * srx) % 2), min(nya, max(1, 60 // sry))),
                       (pkg.FIRE_KERNEL_WARP, kx, 1), (pkg.FIRE_KERNEL_WARP, kx, min(nya, 512 // sry)),
                       (pkg.FIRE_KERNEL_WARP_DENSE, kx, min(nya, 3))):
        m = pkg.FireModel.from_workload(w, precision="fp32")
        pkg.fire_set_kernel(m.ctx, var, k, ky)
        u, v = m.wind(w.u, w.v)
        for _ in range(w.steps):
            hs, hl = m.step(u, v, w.dt)
        torch.cuda.synchronize()
        runs.append(state_np(m)[:3] + (hs.cpu().numpy(), hl.cpu().numpy()))
        m.close()
    assert np.isfinite(runs[0][1]).sum() > 20 and np.abs(runs[0][3]).max() > 0
    for other in runs[1:]:
        for a, b in zip(runs[0], other):
            assert np.array_equal(a, b)


def test_launch_rows_change_no_bit():
    """fire_init's default strips run with the launch's own rows per CTA: the
    same bits as the same strips set explicitly."""
    import torch

    from paper_1102_1343_gb300 import build
    build.build()
    import paper_1102_1343_gb300 as pkg
    w = synth.random_landscape(150, 61, seed=9, ignition="points", n_points=4, edge_margin=800.0,
                               ignition_radius=90.0, steps=30)
    runs = []
    for explicit in (False, True):
        m = pkg.FireModel.from_workload(w, precision="fp32")
        var, kx, ky = pkg.fire_get_kernel(m.ctx)
        assert var in (pkg.FIRE_KERNEL_WARP, pkg.FIRE_KERNEL_WARP_DENSE)
        if explicit:
            pkg.fire_set_kernel(m.ctx, var, kx, ky)
        u, v = m.wind(w.u, w.v)
        hs, hl = m.run(w.steps, u, v, w.dt)
        torch.cuda.synchronize()
        runs.append(state_np(m)[:3] + (hs.cpu().numpy(), hl.cpu().numpy()))
        m.close()
    for a, b in zip(*runs):
        assert np.array_equal(a, b)
