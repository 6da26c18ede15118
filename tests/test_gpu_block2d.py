"""The kernels that stand in for the default schedule (2D register tiles, small
3D grids) against the streaming kernel at the schedule they stand for: the
same bits, for every variant that the rules can pick (on 152 SMs), with ragged
tiles, grids smaller than a tile (the halo reflected several times), and step
counts that split unevenly over the launches."""
import numpy as np
import pytest

import oracle
import paper_2105_09671_gb300 as ac
from paper_2105_09671_gb300 import workloads as wl

from gpu_util import assert_parity, oracle_run

pytestmark = pytest.mark.gpu

# (16 and more steps: 4 rows a lane up to 513 x 509, 8 at 1023 x 1030, 7 for FP32
# from 2049 x 2100 on and FP16 storage at 1500 x 1500, 9 beyond; 4100 x 4200: passes of
# six steps; wide grids of few rows and large ones with few steps: streamed)
SHAPES = [(1, 1), (1, 37), (29, 1), (3, 5), (17, 130), (200, 400), (513, 509), (1023, 1030), (1500, 1500),
          (2049, 2100), (4100, 4200), (1, 200000), (3, 140000), (12, 130000)]


@pytest.mark.parametrize("dtype", ["f32", "f16s"])
@pytest.mark.parametrize("shape", SHAPES)
def test_default_equals_the_streaming_schedule_bitwise(shape, dtype):
    h = 1.0 / max(shape)
    eps, dt = 2.5 * h, 0.1 * h * h
    phi0 = wl.random_field(shape, seed=sum(shape))
    nx = shape[-1]
    a = ac.Simulation(shape, h, eps, dt, dtype=dtype, pitch_x=-(-nx // 8) * 8 + 8)
    b = ac.Simulation(shape, h, eps, dt, dtype=dtype)
    try:
        v, k = b.schedule()
        b.set_schedule(v, k)  # forced: the streaming kernel, rounding at the same pass ends
        for n in (1, 2, 3, 16, 17, 33, 100):
            a.padded.fill_(float("nan"))
            a._ws.fill_(float("nan"))
            a.load(phi0)
            b.load(phi0)
            a.step(n)
            b.step(n)
            out = a.to_numpy()
            assert np.array_equal(out, b.to_numpy()), f"{shape} {dtype} n={n}"
        assert bool(a.padded[:, :, nx:].isnan().all()), "padding written"
        if np.prod(shape) < 1 << 19:
            assert_parity(out.astype(np.float64), oracle_run(phi0, h, eps, dt, 100, dtype), dtype)
    finally:
        a.close()
        b.close()


@pytest.mark.parametrize("shape", [(1, 1, 1), (2, 3, 5), (7, 1, 64), (33, 35, 31), (40, 60, 70), (81, 90, 101),
                                   (1, 300, 301), (3, 200, 301), (5, 280, 283), (6, 300, 301)])
def test_small_3d_default_equals_the_streaming_schedule_bitwise(shape):
    # one step to a launch, in each of its plane counts a thread; odd step
    # counts start with a pass of two
    h = 1.0 / max(shape)
    eps, dt = 2.5 * h, 0.1 * h * h
    phi0 = wl.random_field(shape, seed=sum(shape))
    nx = shape[-1]
    a = ac.Simulation(shape, h, eps, dt, dtype="f32", pitch_x=-(-nx // 4) * 4 + 4)
    b = ac.Simulation(shape, h, eps, dt, dtype="f32")
    try:
        b.set_schedule(*b.schedule())
        for n in (1, 2, 3, 8, 17):
            a.padded.fill_(float("nan"))
            a._ws.fill_(float("nan"))
            a.load(phi0)
            b.load(phi0)
            a.step(n)
            b.step(n)
            out = a.to_numpy()
            assert np.array_equal(out, b.to_numpy()), f"{shape} n={n}"
        assert bool(a.padded[:, :, nx:].isnan().all()), "padding written"
        assert_parity(out.astype(np.float64), oracle_run(phi0, h, eps, dt, 17, "f32"), "f32")
    finally:
        a.close()
        b.close()


def test_forcing_a_schedule_recaptures_the_graph():
    import torch
    shape = (96, 200)
    h = 1.0 / 200
    phi0 = wl.smooth_field(shape, seed=2)
    sim = ac.Simulation(shape, h, 2.5 * h, 0.1 * h * h, dtype="f32", stream=torch.cuda.Stream())
    try:
        sim.load(phi0)
        sim.set_graph(True)
        v, k = sim.schedule()
        sim.step(24)
        n0 = sim.launch_count()
        sim.step(24)
        default = sim.launch_count() - n0
        sim.set_schedule(v, k)
        n0 = sim.launch_count()
        sim.step(24)
        assert sim.launch_count() - n0 == 24 // k > default
        out = sim.to_numpy().astype(np.float64)
    finally:
        sim.close()
    assert_parity(out, oracle_run(phi0, h, 2.5 * h, 0.1 * h * h, 72, "f32"), "f32")
