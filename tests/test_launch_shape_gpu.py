"""fire_init's default shape is launched in another form where that is faster
(FP64 marching strips as warp strips, one-cell tiles merged): the same bits as
the reported shape set explicitly, on square and oblong meshes, odd widths,
refinements whose strips leave lanes over, and with per-node moisture."""
import numpy as np
import pytest

from gpu_helpers import node_moisture, state_np
from paper_1102_1343_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,nxa,nya,sr", [
    ("fp64", 70, 51, 10), ("fp64", 51, 101, 7), ("fp64", 61, 90, 9), ("fp64", 44, 52, 16),
    ("fp64", 10, 10, 10), ("fp64", 21, 17, 10), ("fp32", 37, 29, 10), ("fp32", 21, 33, 11),
    ("fp64", 31, 7, 3), ("fp32", 60, 41, 1)])
@pytest.mark.parametrize("moisture", [False, True])
def test_launch_shape_changes_no_bit(prec, nxa, nya, sr, moisture):
    import torch

    from paper_1102_1343_gb300 import build
    build.build()
    import paper_1102_1343_gb300 as pkg
    w = synth.random_landscape(nxa, nya, sr=sr, dx_atm=6.0 * sr, seed=nxa + nya, ignition="none", steps=9, dt=0.25)
    w.ignitions = [synth.point_ignition(x * nxa * sr * 6.0, y * nya * sr * 6.0, radius=20.0)
                   for x, y in ((0.5, 0.5), (0.05, 0.9), (0.96, 0.1))]
    if moisture:
        w = node_moisture(w)
    runs = []
    for explicit in (False, True):
        m = pkg.FireModel.from_workload(w, precision=prec)
        if explicit:
            pkg.fire_set_kernel(m.ctx, *pkg.fire_get_kernel(m.ctx))
        u, v = m.wind(w.u, w.v)
        hs, hl = m.run(w.steps, u, v, w.dt)
        torch.cuda.synchronize()
        runs.append(state_np(m)[:3] + (hs.cpu().numpy(), hl.cpu().numpy()))
        m.close()
    assert np.isfinite(runs[0][1]).any()
    for a, b in zip(*runs):
        assert np.array_equal(a, b)
