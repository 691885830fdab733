"""The FP64 root, reciprocals, quotient and power of fp64_math.cuh against
values of extended precision, in units of u = 2^-53 relative, over every entry
of the power's tables and the ends of the ranges the functions state.

Bounds.  rsqrt64, sqrt64: the last rounding (1 u), the rounding of x y (half of
it enters, 0.5 u) and what the series leaves out (2^-7 u), so 1.6 u.  rcp64 and
the quotient: the last rounding and a residual below 2^-6 u, so 1.1 u.  The
power: y = b log2 x is rounded once (|y| u, times ln 2), the table, its product
and the last sum 3 u more.  Outside its fast range it is exp2(b log2 x) of the
CUDA functions: three roundings of y (each to 1.5 u) and 3 u.  And the adjoint's quotient by a capped wind component
below the normal range."""
import ctypes as C
import dataclasses
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

U = 2.0 ** -53
RSQRT, SQRT, RCP, DIV, POW = range(5)


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    from paper_1102_1343_gb300 import build
    so = str(tmp_path_factory.mktemp("probe") / "fp64_probe.so")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "fp64_probe.cu")
    flags = [f for f in build.NVCC_FLAGS if f not in ("-Xptxas", "-v")]
    subprocess.run([build.nvcc()] + build.ARCH + flags + ["-I", build.CSRC, "-shared", "-o", so, src, "-cudart", "static"], check=True)
    lib = C.CDLL(so)

    def run(op, a, b=None):
        a = np.ascontiguousarray(a, np.float64)
        b = np.ascontiguousarray(np.ones_like(a) if b is None else b, np.float64)
        o = np.empty_like(a)
        p = lambda x: x.ctypes.data_as(C.POINTER(C.c_double))
        assert lib.probe(op, a.size, p(a), p(b), p(o)) == 0
        return o

    return run


def normals(rng, lo, hi, n=40000):
    """Numbers in [2^lo, 2^hi): random and the ends of the binades."""
    e = rng.integers(lo, hi, n)
    m = 1 + rng.integers(0, 2 ** 52, n) * 2.0 ** -52
    e[:4], m[:4] = (lo, hi - 1, lo, hi - 1), (1.0, 2 - 2 ** -52, 1 + 2 ** -52, 1.0)
    return np.ldexp(m, e)


def error(got, want):
    assert np.isfinite(got).all()
    return float(np.abs((got.astype(np.longdouble) - want) / want).max() / U)


def test_roots(probe):
    x = normals(np.random.default_rng(1), -1021, 1024)
    root = np.sqrt(x.astype(np.longdouble))
    assert error(probe(RSQRT, x), 1 / root) <= 1.6
    assert error(probe(SQRT, x), root) <= 1.6
    s = np.array([0.0, -0.0, 5e-324, 1e-310, 2.2250738585072014e-308, np.inf, np.nan, -1.0])
    assert np.array_equal(probe(SQRT, s), np.sqrt(s, where=s >= 0, out=np.full_like(s, np.nan)), equal_nan=True)


def test_reciprocal_and_quotient(probe):
    rng = np.random.default_rng(2)
    x = normals(rng, -1021, 1022)
    assert error(probe(RCP, x), 1 / x.astype(np.longdouble)) <= 1.1
    a, b = normals(rng, -400, 400), normals(rng, -500, 500)
    assert error(probe(DIV, a, b), a.astype(np.longdouble) / b) <= 1.1
    # divisors without a normal reciprocal: the ordinary quotient
    b = np.array([5e-324, 1e-310, 2.2250738585072014e-308, 2.0 ** 1022, 1.7e308, np.inf, 0.0])
    for a in (0.0, 1e-309, 0.75, 3.0):
        with np.errstate(all="ignore"):
            assert np.array_equal(probe(DIV, np.full_like(b, a), b), a / b, equal_nan=True)


def test_power(probe):
    edges = 1 + np.arange(128) / 128.0
    m = np.concatenate([edges, np.nextafter(edges[1:], 0), [2 - 2 ** -52], edges + 1 / 256.0,
                        1 + np.random.default_rng(3).uniform(0, 1, 200)])
    for e in (-64, -63, -43, -1, 0, 1, 4, 63):
        for b in (0.03, 0.9, 1.0, 1.5, 2.2, 13.9):
            x = np.ldexp(m, e)
            y = np.float64(b).astype(np.longdouble) * np.log2(x.astype(np.longdouble))
            got = probe(POW, x, np.full_like(x, b))
            err = np.abs(got.astype(np.longdouble) / np.exp2(y) - 1) / U
            assert (err <= 0.7 * np.abs(y) + 3).all(), (e, b, float(err.max()))
    # beyond the fast range, and 0
    x = np.array([1e-300, 1e-200, 1e-30, 1e25, 1e100, 2.2250738585072014e-308, 1e-310, 5e-324])
    for b in (0.03, 0.9, 1.0):
        y = np.float64(b).astype(np.longdouble) * np.log2(x.astype(np.longdouble))
        want = np.exp2(y)
        got = probe(POW, x, np.full_like(x, b)).astype(np.longdouble)
        assert (np.abs(got - want) <= want * U * (3.2 * np.abs(y) + 3) + 5e-324).all(), b
    assert (probe(POW, np.zeros(3), np.array([0.5, 1.0, 2.0])) == 0).all()


def test_wind_below_the_normal_range():
    """Capped wind components between 0 and the smallest normal number: the
    gradients are the oracle's (the quotient by such a component)."""
    import oracle
    import paper_1102_1343_gb300 as pkg
    from paper_1102_1343_gb300 import build, synth
    build.build()
    w = synth.random_landscape(8, 7, sr=10, dx_atm=60.0, seed=9, ignition="center", steps=6, dt=0.5)
    w = dataclasses.replace(w, classes=[synth.nominal_class(fgi=0.5)], fuel=np.zeros((70, 80), np.uint8))
    w = dataclasses.replace(w, ignitions=[synth.point_ignition(240.0, 210.0, radius=20.0)], mult=np.full((70, 80), 40.0),
                            u=w.u * 1e-310, v=w.v * 1e-310)
    y, x = np.indices((70, 80))
    tobs = np.where((x - 40) ** 2 + (y - 35) ** 2 < 400, 2.0, np.nan)
    Jr, *ref = oracle.OracleFire.from_workload(w).adjoint(w.u, w.v, w.dt, w.steps, tobs)
    m = pkg.FireModel.from_workload(w, precision="fp64")
    u, v = m.wind(w.u, w.v)
    J, *g = m.adjoint(u, v, w.dt, w.steps, tobs, ckpt_every=2)
    assert np.abs(ref[0]).max() > 0 and abs(J - Jr) <= 1e-10 * Jr
    for a, b in zip(g[:2], ref[:2]):
        a = a.cpu().numpy()
        assert np.isfinite(a).all() and np.linalg.norm(a - b) <= 1e-8 * np.linalg.norm(b)
    for a in g[2:]:
        assert np.isfinite(a.cpu().numpy()).all()
    m.close()
