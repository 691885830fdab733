"""fire_get_launch tells the kernel and shape that a context's launches take:
fire_init's default in the form that stands for it, a shape set explicitly as it
stands, the same before and after the adaptive choice changes its name."""
import ctypes as C

import pytest

from paper_1102_1343_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    from paper_1102_1343_gb300 import build
    build.build()
    import paper_1102_1343_gb300 as p
    p.load_library()
    return p


def model(pkg, nxa, nya, sr, prec, radius=10.0, steps=1):
    w = synth.random_landscape(nxa, nya, sr=sr, dx_atm=6.0 * sr, seed=3, ignition="center", ignition_radius=radius, steps=steps)
    if radius != 10.0:
        w.ignitions = [synth.point_ignition(w.nx * w.dx / 2, w.ny * w.dy / 2, radius=radius)]
    return w, pkg.FireModel.from_workload(w, precision=prec)


def test_forms_of_the_default(pkg):
    T, M, W = pkg.FIRE_KERNEL_TILE, pkg.FIRE_KERNEL_MARCH, pkg.FIRE_KERNEL_WARP
    for nxa, nya, sr, prec, kind, launched in ((51, 51, 10, "fp64", M, W), (200, 150, 10, "fp32", W, W),
                                               (40, 30, 10, "fp32", T, T), (20, 20, 40, "fp64", M, M)):
        _, m = model(pkg, nxa, nya, sr, prec)
        shape, launch = pkg.fire_get_kernel(m.ctx), pkg.fire_get_launch(m.ctx)
        assert shape[0] == kind and launch[0] == launched
        if (kind, launched) == (T, T):
            assert shape == (T, 1, 1) and launch[1] * launch[2] > 1
        m.close()
    for var, k, want in ((W, (6, 40), (W, 6, 16)), (pkg.FIRE_KERNEL_WARP_DENSE, (6, 3), (W, 6, 3)), (T, (2, 3), (T, 2, 3)),
                         (pkg.FIRE_KERNEL_WARP4, (12, 40), (pkg.FIRE_KERNEL_WARP4, 12, 40))):
        _, m = model(pkg, 51, 51, 10, "fp32")
        pkg.fire_set_kernel(m.ctx, var, *k)
        assert pkg.fire_get_kernel(m.ctx) == (var, *k) and pkg.fire_get_launch(m.ctx) == want
        m.close()
    i = C.c_int()
    assert pkg.load_library().fire_get_launch(None, C.byref(i), C.byref(i), C.byref(i)) == pkg.FIRE_ERR_ARG


@pytest.mark.parametrize("nxa,nya,sr", [(200, 200, 10), (300, 140, 7), (560, 560, 10)])
def test_adaptive_choice_keeps_the_launches(pkg, nxa, nya, sr):
    """Sparse, then burning, then sparse again, and the choice turned on anew: the
    name changes, the launches of a default context do not (on 560 x 560 cells
    the default rows and the launch's are the same)."""
    w, m = model(pkg, nxa, nya, sr, "fp32")
    torch = m.torch
    shape, launch = pkg.fire_get_kernel(m.ctx), pkg.fire_get_launch(m.ctx)
    assert shape[0] == pkg.FIRE_KERNEL_WARP
    u, v = m.wind(w.u, w.v)
    psi, tign, frac, t = m.state()
    for burnt in (True, False, True):
        p = torch.where(torch.arange(m.ny, device="cuda")[:, None] < m.ny // 3, -psi.abs(), psi.abs()) if burnt else psi
        m.set_state(p, torch.where(p <= 0, -9.0, torch.inf).double(), frac, t)
        m.step(u, v, 0.25)
        torch.cuda.synchronize()
        m.step(u, v, 0.25)  # the count has landed
        name = pkg.fire_get_kernel(m.ctx)[0]
        assert name == (pkg.FIRE_KERNEL_WARP_DENSE if burnt else pkg.FIRE_KERNEL_WARP)
        assert pkg.fire_get_launch(m.ctx) == launch
    pkg.fire_set_adaptive(m.ctx, True)
    assert pkg.fire_get_kernel(m.ctx)[0] == pkg.FIRE_KERNEL_WARP and pkg.fire_get_launch(m.ctx) == launch
    m.close()


@pytest.mark.parametrize("n,prec", [(10, "fp64"), (51, "fp64"), (40, "fp32")])
def test_autotune_leaves_no_context_slower(pkg, n, prec):
    """The form that stands for the default is among the candidates: after
    fire_autotune 200 steps take at most 1.3 times as long as before."""
    import torch
    w, m = model(pkg, n, n, 10, prec)
    u, v = m.wind(w.u, w.v)
    e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]

    def ms():
        best = 1e9
        for _ in range(4):
            e[0].record()
            m.run(200, u, v, 0.01)
            e[1].record()
            torch.cuda.synchronize()
            best = min(best, e[0].elapsed_time(e[1]))
        return best

    before = ms()
    assert m.autotune(u, v, 0.01) == pkg.fire_get_kernel(m.ctx)
    assert ms() <= 1.3 * before
    m.close()
