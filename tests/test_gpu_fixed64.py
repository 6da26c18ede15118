"""FP64 grids: the fixed-point form of the update.  Every schedule gives the
same bits (the form a cell takes depends on its stencil alone); cells outside
the form's range (small, large, infinite, NaN) take the FP64 operations; and
against extended precision a step is no less exact than those."""
import numpy as np
import pytest

import oracle
import paper_2105_09671_gb300 as ac
from paper_2105_09671_gb300 import workloads as wl

from gpu_util import gpu_run, schedules

pytestmark = pytest.mark.gpu

# marching kernels from 512^2 cells on: strips of 124 (2D) and 60 (3D) columns, bands of 2 rows
SHAPES = [(1, 1), (3, 5), (9, 123), (33, 125), (130, 249), (1, 1, 1), (2, 3, 5), (5, 9, 59), (9, 13, 61), (4, 4, 121), (600, 700),
          (65, 64, 66)]


def _step_long(phi, h, eps, dt):
    """One step in extended precision (x87 or quad, whichever the host has)."""
    L = np.longdouble
    p = phi.astype(L)
    alpha, beta = L(dt / (eps * eps)), L(dt / (h * h))
    s = np.zeros_like(p)
    for ax in range(p.ndim):
        n = p.shape[ax]
        lo = np.take(p, np.maximum(np.arange(n) - 1, 0), axis=ax)
        hi = np.take(p, np.minimum(np.arange(n) + 1, n - 1), axis=ax)
        s = s + (lo + hi)
    return p + alpha * (p - p * p * p) + beta * (s - 2 * p.ndim * p)


@pytest.mark.parametrize("shape", [(1, 1), (3, 5), (29, 31), (64, 64), (97, 200), (515, 517), (700, 900)])
@pytest.mark.parametrize("amp", [1.0, 0.1, 3.0])
def test_default_equals_one_step_a_launch_bitwise(shape, amp):
    # the register-tile kernel (several steps a launch; tiles with a value out
    # of range mix both forms) and, from 512^2 cells on, the marching kernel
    h = 1.0 / max(shape)
    eps, dt = 2.5 * h, (0.1 if amp < 2 else 0.02) * h * h
    phi0 = amp * wl.random_field(shape, seed=sum(shape))
    for n in (1, 2, 7, 16, 50):
        a = gpu_run(phi0, h, eps, dt, n, "f64")
        b = gpu_run(phi0, h, eps, dt, n, "f64", ac.AC_VARIANT_STREAM, 1, 0)
        assert np.array_equal(a, b), f"{shape} amplitude {amp} n={n}"


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("amp", [1.0, 0.05, 1e-3, 3.0])
def test_schedules_give_the_same_bits(shape, amp):
    h = 1.0 / max(shape)
    eps, dt = 2.5 * h, 0.1 * h * h
    if amp > 1:
        dt *= 0.2
    phi0 = amp * wl.random_field(shape, seed=sum(shape))
    out = {}
    for v, k, tile in schedules(len(shape), "f64"):
        out[(v, k, tile)] = gpu_run(phi0, h, eps, dt, 3, "f64", v, k, tile)
    ref = out[(ac.AC_VARIANT_DIRECT, 1, 0)]
    for key, o in out.items():
        assert np.array_equal(o, ref), f"{shape} amplitude {amp} schedule {key}"
    o = oracle.step(phi0, h, eps, dt, 3)
    assert np.max(np.abs(ref - o)) <= 1e-14 * max(1.0, np.max(np.abs(o)))


def test_special_values_propagate_as_in_fp64():
    shape = (40, 260)
    h = 1.0 / 260
    phi0 = np.tile(np.linspace(-1.0, 1.0, 260), (40, 1))
    phi0[5, 7] = np.nan
    phi0[20, 130] = np.inf
    phi0[30, 200] = -np.inf
    phi0[35, 60:64] = [1.25, -1.25, 1e300, -1e300]
    phi0[10, 100] = 5e-324
    phi0[10, 101] = -0.0
    with np.errstate(all="ignore"):
        ref = oracle.step(phi0, h, 2.5 * h, 0.1 * h * h, 1)
    sim = ac.Simulation(shape, h, 2.5 * h, 0.1 * h * h, dtype="f64")
    try:
        sim.load(phi0)
        sim.step(1)
        out = sim.to_numpy()
    finally:
        sim.close()
    assert np.array_equal(np.isnan(out), np.isnan(ref))
    assert np.array_equal(np.isinf(out), np.isinf(ref))
    f = np.isfinite(ref)
    assert np.allclose(out[f], ref[f], rtol=1e-14, atol=1e-16)


@pytest.mark.parametrize("shape", [(200, 300), (20, 40, 70)])
@pytest.mark.parametrize("amp,smooth", [(1.0, 0), (0.1, 0), (0.02, 0), (1.0, 1)])
def test_a_step_is_no_less_exact_than_fp64_operations(shape, amp, smooth):
    # the FP64 form's error, by the same operations in NumPy (products rounded
    # where the GPU fuses them adds at most a third): rms over 6e4 cells
    h = 1.0 / max(shape)
    eps, dt = 2.5 * h, 0.1 * h * h
    phi0 = (wl.smooth_field(shape, seed=3, amp=0.98) if smooth else amp * wl.random_field(shape, seed=5))
    exact = _step_long(phi0, h, eps, dt)
    out = gpu_run(phi0, h, eps, dt, 1, "f64", ac.AC_VARIANT_DIRECT, 1)
    alpha, beta = dt / (eps * eps), dt / (h * h)
    p = phi0
    s = 0.0
    for ax in range(p.ndim):
        n = p.shape[ax]
        s = s + (np.take(p, np.maximum(np.arange(n) - 1, 0), axis=ax) +
                 np.take(p, np.minimum(np.arange(n) + 1, n - 1), axis=ax))
    native = (p + beta * (s - 2 * p.ndim * p)) + alpha * (p - p * p * p)
    rms = lambda a: float(np.sqrt(np.mean(((a - exact).astype(np.float64)) ** 2)))
    assert rms(out) <= rms(native), f"{rms(out):.3e} against {rms(native):.3e}"


@pytest.mark.parametrize("shape", [(200, 197, 203), (3001, 3100), (7, 1030, 130), (2, 600, 1300)])
def test_marches_of_several_rounds_give_the_same_bits(shape):
    # items of a warp each, in several rounds of the resident CTAs (the first
    # two) and in one; the last item is shorter than the others
    h = 1.0 / max(shape)
    a = oracle.init_random(shape, seed=11)
    got = []
    for variant in (ac.AC_VARIANT_DIRECT, ac.AC_VARIANT_STREAM):
        sim = ac.Simulation(shape, h, 2.5 * h, 0.1 * h * h, dtype="f64")
        try:
            sim.load(a)
            sim.set_schedule(variant, 1)
            sim.step(3)
            got.append(sim.to_numpy())
        finally:
            sim.close()
    assert np.array_equal(*got)
