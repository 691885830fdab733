"""Meshes with more rows of strips than one grid dimension holds (65535): the
default launch and tall strips set explicitly step them, to the same bits as
kernels whose grids stay below it."""
import numpy as np
import pytest

from gpu_helpers import state_np
from paper_1102_1343_gb300 import synth

pytestmark = pytest.mark.gpu

NY = 2_200_000


@pytest.mark.parametrize("prec,kernel", [("fp32", None), ("fp64", None), ("fp32", "WARP"), ("fp64", "WARP")])
def test_more_than_65535_rows_of_strips(prec, kernel):
    import torch

    from paper_1102_1343_gb300 import build
    build.build()
    import paper_1102_1343_gb300 as pkg
    z = np.zeros((NY, 2))
    fires = [synth.point_ignition(6.0, 6.0 * y, radius=30.0) for y in (3, 1_048_576, 1_835_000, NY - 40)]
    u, v = synth.constant_wind(2, NY, 1.0, 4.0)
    runs = []
    for ref in (False, True):
        m = pkg.FireModel(2, NY, 1, 6.0, [synth.nominal_class()], z.astype(np.uint8), z, z, fires, precision=prec)
        if ref:
            pkg.fire_set_kernel(m.ctx, *((pkg.FIRE_KERNEL_WARP4, 2, 500) if prec == "fp32" else (pkg.FIRE_KERNEL_MARCH, 2, 60)))
        elif kernel:
            pkg.fire_set_kernel(m.ctx, pkg.FIRE_KERNEL_WARP, 2, 4)
        ud, vd = m.wind(u, v)
        hs, hl = m.run(5, ud, vd, 0.25)
        torch.cuda.synchronize()
        assert m.status() == pkg.FIRE_ERR_BOUNDARY  # (every node of two columns is a boundary node)
        runs.append(state_np(m)[:3] + (hs.cpu().numpy(), hl.cpu().numpy()))
        m.close()
    t = runs[0][1]
    for y in (3, 1_048_576, 1_835_000, NY - 40):
        assert np.isfinite(t[y]).all()
    for a, b in zip(*runs):
        assert np.array_equal(a, b)
