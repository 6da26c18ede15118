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

# marching kernels from 1 M cells on (3D 0.7 M): strips of 124 (2D) and 60 (3D) columns, bands of 2 rows
SHAPES = [(1, 1), (3, 5), (9, 123), (33, 125), (130, 249), (1, 1, 1), (2, 3, 5), (5, 9, 59), (9, 13, 61), (4, 4, 121), (600, 700),
          (65, 64, 66), (1003, 1001), (99, 101, 103)]


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


@pytest.mark.parametrize("shape", [(1, 1), (3, 5), (29, 31), (64, 64), (97, 200), (515, 517), (700, 900),
                                   (1003, 1009)])
@pytest.mark.parametrize("amp", [1.0, 0.1, 3.0])
def test_default_equals_one_step_a_launch_bitwise(shape, amp):
    # the register-tile kernel up to 50000 cells (several steps a launch; tiles
    # with a value out of range mix both forms), one thread a cell and, from 1 M
    # cells on, the marching kernel
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


# fields whose small cells have large neighbours: fronts that cross zero close
# to cell centres, planar and slightly tilted, and rough noise
def _crossing_field(shape, seed):
    rng = np.random.default_rng(seed)
    x = np.arange(shape[-1], dtype=np.float64)
    rows = int(np.prod(shape[:-1]))
    off = 10.0 ** rng.uniform(-9, -0.3, rows) * rng.choice([-1.0, 1.0], rows)
    if seed % 2 == 0:
        off = off[0] + 1e-4 * np.sin(np.arange(rows) * 0.1)
    mid = shape[-1] // 2
    return np.tanh((x[None, :] - mid + off[:, None]) / 3.0).reshape(shape)


def _axis_neighbours(p):
    out = []
    for ax in reversed(range(p.ndim)):  # x, y, z
        n = p.shape[ax]
        out.append(np.take(p, np.maximum(np.arange(n) - 1, 0), axis=ax))
        out.append(np.take(p, np.minimum(np.arange(n) + 1, n - 1), axis=ax))
    return out


@pytest.mark.parametrize("shape", [(24, 40), (5, 6, 40)])
@pytest.mark.parametrize("kind", [0, 1, "rough"])
@pytest.mark.parametrize("heat", [False, True])
def test_cells_of_every_size_are_no_less_exact_than_fp64_operations(shape, kind, heat):
    # against exact rationals, cells binned by their result's size relative to
    # the stencil's largest value; the baseline is ac_update with its fused
    # operations, each rounded once
    from fractions import Fraction as Q
    h = 1.0 / 64
    eps, dt = np.inf if heat else 2.5 * h, 0.1 * h * h
    phi0 = 0.1 * wl.random_field(shape, seed=4) if kind == "rough" else _crossing_field(shape, kind)
    phi0 = (300.0 if heat else 1.0) * phi0
    out = gpu_run(phi0, h, eps, dt, 1, "f64", ac.AC_VARIANT_DIRECT, 1).reshape(-1)
    alpha, beta = dt / (eps * eps), dt / (h * h)
    nb = [a.reshape(-1) for a in _axis_neighbours(phi0)]
    p = phi0.reshape(-1)
    m2d = -2 * phi0.ndim
    bins = {}
    for i in range(p.size):
        v = [float(a[i]) for a in nb]
        c = float(p[i])
        exact = Q(c) + Q(beta) * (sum(map(Q, v)) + m2d * Q(c)) + Q(alpha) * (Q(c) - Q(c) ** 3)
        ns = (v[0] + v[1]) + (v[2] + v[3])
        if phi0.ndim == 3:
            ns += v[4] + v[5]
        lap = float(Q(m2d) * Q(c) + Q(ns))
        re = float(Q(-c * c) * Q(c) + Q(c))
        fused = float(Q(alpha) * Q(re) + Q(float(Q(beta) * Q(lap) + Q(c))))
        top = max(abs(c), max(map(abs, v)))
        b = min(14, int(-np.log2(abs(float(exact)) / top))) if exact else 14
        e = bins.setdefault(b // 2, [0, 0.0, 0.0])
        e[0] += 1
        e[1] += float(Q(float(out[i])) - exact) ** 2
        e[2] += float(Q(fused) - exact) ** 2
    assert len(bins) > 1
    for b, (n, mine, base) in sorted(bins.items()):
        if n >= 20:
            assert mine <= base, f"2^-{2 * b}: {np.sqrt(mine / n):.3e} against {np.sqrt(base / n):.3e} ({n} cells)"


@pytest.mark.parametrize("shape", [(24, 40), (130, 249), (515, 517), (1003, 1001), (5, 6, 40), (65, 64, 66), (99, 101, 103)])
@pytest.mark.parametrize("kind", [0, 1, "rough", "large"])
def test_negated_fields_step_to_the_negated_result(shape, kind):
    h = 1.0 / 64
    eps, dt = 2.5 * h, 0.1 * h * h
    if kind in (0, 1):
        phi0 = _crossing_field(shape, kind)
    else:
        phi0 = (3.0 if kind == "large" else 0.1) * wl.random_field(shape, seed=4)
        dt *= 0.2 if kind == "large" else 1.0
    phi0.reshape(-1)[7:9] = [0.0, -0.0]
    for v, k in ((None, None), (ac.AC_VARIANT_DIRECT, 1), (ac.AC_VARIANT_STREAM, 2)):
        a = gpu_run(phi0, h, eps, dt, 6, "f64", v, k) if v is not None else gpu_run(phi0, h, eps, dt, 6, "f64")
        b = gpu_run(-phi0, h, eps, dt, 6, "f64", v, k) if v is not None else gpu_run(-phi0, h, eps, dt, 6, "f64")
        assert np.array_equal(a, -b), f"{shape} {kind} schedule {v} {k}"


@pytest.mark.parametrize("shape", [(40, 64), (300, 310), (1003, 1001), (9, 13, 61), (64, 65, 66), (99, 101, 103)])
def test_temperatures_of_any_size_give_the_same_bits_on_every_kernel(shape):
    # the heat equation: no bound on the field; from 2^340 = 2.2e102 on the FP64
    # operations
    h = 1.0 / 64
    phi0 = wl.random_field(shape, seed=4) * np.linspace(1.0, 400.0, shape[-1])
    spikes = phi0.copy()
    spikes.reshape(-1)[11:14] = [1e101, 3e102, -5e102]
    for f in (phi0, spikes):
        outs = [gpu_run(f, h, np.inf, 0.1 * h * h, 3, "f64", *s)
                for s in ((), (ac.AC_VARIANT_DIRECT, 1), (ac.AC_VARIANT_STREAM, 1), (ac.AC_VARIANT_STREAM, 2))]
        assert np.isfinite(outs[0]).all()
        for o in outs[1:]:
            assert np.array_equal(outs[0], o)
        if f is phi0:
            ref = oracle.step(f, h, np.inf, 0.1 * h * h, 3)
            assert np.max(np.abs(outs[0] - ref)) <= 1e-14 * 400


@pytest.mark.parametrize("shape", [(40, 64), (200, 210), (1003, 1001), (9, 13, 61), (99, 101, 103)])
@pytest.mark.parametrize("eps", [np.inf, 2.5 / 64])
def test_fields_at_rest_stay_so_beside_others(shape, eps):
    # zeros of either sign, a square of other values among them and subnormal ones
    # in its neighbourhood; the same bits on every kernel
    h = 1.0 / 64
    phi0 = np.zeros(shape)
    phi0[..., ::3] = -0.0
    mid = tuple(slice(n // 3, n // 3 + max(1, n // 8)) for n in shape)
    phi0[mid] = 0.9 * wl.random_field(phi0[mid].shape, seed=4)
    phi0.reshape(-1)[3:6] = [5e-324, -3e-310, 1e-300]
    outs = [gpu_run(phi0, h, eps, 0.1 * h * h, 4, "f64", *s)
            for s in ((), (ac.AC_VARIANT_DIRECT, 1), (ac.AC_VARIANT_STREAM, 1), (ac.AC_VARIANT_STREAM, 2))]
    for o in outs[1:]:
        assert np.array_equal(outs[0], o)
    ref = oracle.step(phi0, h, eps, 0.1 * h * h, 4)
    assert np.max(np.abs(outs[0] - ref)) <= 1e-14
    assert np.array_equal(outs[0] == 0.0, ref == 0.0)


@pytest.mark.parametrize("shape,n", [((16, 16), 2000), ((40, 64), 600), ((520, 510), 100), ((4, 6, 64), 600)])
def test_a_field_odd_about_its_middle_stays_so(shape, n):
    h = 1.0 / 64
    x = np.arange(shape[-1]) - (shape[-1] - 1) / 2
    phi0 = np.broadcast_to(np.tanh(x / 3.0), shape).copy()
    phi0 += np.broadcast_to(1e-3 * np.sin(x), shape)
    phi0 = 0.5 * (phi0 - phi0[..., ::-1])
    assert np.array_equal(phi0, -phi0[..., ::-1])
    out = gpu_run(phi0, h, 2.5 * h, 0.1 * h * h, n, "f64")
    assert np.array_equal(out, -out[..., ::-1])
