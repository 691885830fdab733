"""A launch that the device refuses is reported by the call that made it, and by
that call alone: the next call on the context, or on another, runs."""
import numpy as np
import pytest

from paper_1102_1343_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call", ["step", "run"])
def test_the_call_after_a_refused_launch_runs(call):
    from paper_1102_1343_gb300 import build
    build.build()
    import paper_1102_1343_gb300 as pkg
    ny = 70_000
    z = np.zeros((ny, 2))
    m = pkg.FireModel(2, ny, 1, 6.0, [synth.nominal_class()], z.astype(np.uint8), z, z, precision="fp64")
    u, v = m.wind(*synth.constant_wind(2, ny, 1.0, 4.0))
    pkg.fire_set_kernel(m.ctx, pkg.FIRE_KERNEL_TILE, 1, 1)  # 70000 rows of tiles: more than a grid takes
    with pytest.raises(pkg.FireError, match="CUDA"):
        m.step(u, v, 0.25) if call == "step" else m.run(4, u, v, 0.25)
    pkg.fire_set_kernel(m.ctx, pkg.FIRE_KERNEL_TILE, 1, 4)
    m.run(4, u, v, 0.25)
    m.close()
    w = synth.plain_circle(3, 3)
    m = pkg.FireModel.from_workload(w, precision="fp64")
    m.step(*m.wind(w.u, w.v), w.dt)
    assert m.status() == pkg.FIRE_OK
    m.close()
