"""Ensembles of several sizes alive at once: the shared-memory limit of a member
kernel belongs to the function, so an ensemble created or reshaped later (fewer
classes, shorter strips, an odd mesh width) leaves the earlier ones able to
launch, to capture a new step count and to be created again."""
import numpy as np
import pytest

from paper_1102_1343_gb300 import synth
from test_ensemble_gpu import make_ensemble, member_state, pkg  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("sr", [10, 34])  # 34: marching strips in FP32 too
def test_limit_of_a_shared_kernel_is_never_lowered(pkg, prec, sr):  # noqa: F811
    big = [synth.random_landscape(12, 9, sr=sr, seed=51, ignition="center"),
           synth.random_landscape(8, 8, sr=sr, seed=53, ignition="center")]
    small = [synth.plain_circle(3, 4, sr=5, steps=1), synth.plain_circle(4, 3, sr=5, steps=1)]
    if prec == "fp32" and sr > 30:
        small = [synth.plain_circle(3, 4, sr=35, steps=1)]

    def step(ens, winds, n):
        pkg.fire_ensemble_step(ens, n, 0.25, [u for u, _ in winds], [v for _, v in winds])
        assert pkg.fire_ensemble_status(ens, len(winds))[0] == pkg.FIRE_OK

    first, wf = make_ensemble(pkg, big, prec)
    step(first, wf, 4)
    other, wo = make_ensemble(pkg, small, prec)
    pkg.fire_ensemble_set_kernel(other, 40, 20)
    step(other, wo, 4)
    step(first, wf, 5)
    before = [member_state(pkg, first, k, w, prec) for k, w in enumerate(big)]
    pkg.fire_ensemble_destroy(first)
    first, wf = make_ensemble(pkg, big, prec)
    step(first, wf, 9)
    for k, w in enumerate(big):
        for a, b in zip(before[k], member_state(pkg, first, k, w, prec)):
            assert np.array_equal(a, b)
    pkg.fire_ensemble_destroy(first)
    pkg.fire_ensemble_destroy(other)
