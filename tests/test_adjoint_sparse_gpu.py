"""The reverse steps leave out the parts of the mesh where the adjoint is
exactly 0: gradients against the oracle's on meshes larger than a fire's reach,
with fires inside, on an edge and in a corner, widths that are and are not
multiples of the 32 nodes of a segment or a tile, and observations of one fire
only.  The bounds are those of the whole-mesh comparisons: 1e-8 in FP64, 2e-3
(the rounding of the forward states) in FP32; where the oracle's gradient of a
node is exactly 0 far from any fire, so is the GPU's."""
import numpy as np
import pytest

import oracle
from paper_1102_1343_gb300 import synth
from test_adjoint_gpu import gpu_adjoint, observations, pkg, rel  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nxa,nya,sr", [(23, 11, 7), (16, 9, 10), (33, 6, 5), (4, 40, 5)])
@pytest.mark.parametrize("where", [((0.5, 0.5), (0.02, 0.97)), ((0.98, 0.4),)])
@pytest.mark.parametrize("ckpt", [1, 5])
def test_sparse_adjoint_matches_oracle(pkg, nxa, nya, sr, where, ckpt):  # noqa: F811
    nsteps = 14
    w = synth.random_landscape(nxa, nya, sr=sr, dx_atm=2.0 * sr, seed=nxa, ignition="none", steps=nsteps, dt=0.25)
    Lx, Ly = nxa * sr * 2.0, nya * sr * 2.0
    w.ignitions = [synth.point_ignition(x * Lx, y * Ly, radius=7.0) for x, y in where]
    rng = np.random.default_rng(nya)
    w.mult = 3.0 * (1.0 + 0.05 * rng.standard_normal((w.ny, w.nx)))
    tobs = observations(w, nsteps)
    if len(where) > 1:  # the second fire is not observed
        tobs[:, : w.nx // 5] = np.nan
    ref = oracle.OracleFire.from_workload(w)
    Jr, *gr = ref.adjoint(w.u, w.v, w.dt, nsteps, tobs)
    assert Jr > 0 and np.abs(gr[0]).max() > 0
    far = np.ones((w.ny, w.nx), bool)  # nodes out of reach of every crossing
    ys, xs = np.nonzero(np.isfinite(ref.tign) & np.isfinite(tobs))
    far[max(0, ys.min() - 4 * nsteps):ys.max() + 4 * nsteps + 1, max(0, xs.min() - 4 * nsteps):xs.max() + 4 * nsteps + 1] = False
    for prec, tol in (("fp64", 1e-8), ("fp32", 2e-3)):
        (J, *g), _ = gpu_adjoint(pkg, w, prec, nsteps, tobs, ckpt=ckpt)
        assert abs(J - Jr) <= (1e-10 if prec == "fp64" else tol) * Jr
        for a, b in zip(g, gr):
            assert rel(a, b) <= tol
        assert not np.asarray(g[0]).reshape(w.ny, w.nx)[far].any()
