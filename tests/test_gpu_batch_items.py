"""Batches whose work items are of the fewest rows (8), of a middle height and
of the most (256; FP64 64), with a last chunk of one row, against the
single-grid stepper, bit for bit."""
import numpy as np
import pytest

import oracle
import paper_2105_09671_gb300 as ac

pytestmark = pytest.mark.gpu


# (513, 500) is 5 strips: 2 grids take 8 rows (FP32: 1.25 items to each of 2432
# resident warps), 60 grids 52, 300 grids 256 (even these leave 4500 items); FP16
# storage, 3 strips, 80 grids 64 rows.  Depths 4 and 3 round the rows up to 4 and 0
# modulo 6.
@pytest.mark.parametrize("dtype,k,copies", [("f32", 4, 2), ("f32", 4, 60), ("f32", 4, 300), ("f32", 2, 60),
                                            ("f16s", 3, 300), ("f16s", 4, 80), ("f16s", 3, 80), ("f64", 1, 60),
                                            ("f64", 3, 2)])
def test_item_heights_equal_single_grid_stepper(dtype, k, copies):
    shapes = [(513, 500), (9, 130), (257, 33)]
    inits = [oracle.init_random(s, seed=7 + i) for i, s in enumerate(shapes)]
    which = [0] * copies + [1, 2]
    specs = [(shapes[w], 1 / 513, 4 / 513, 0.1 / 513**2) for w in which]
    n = 2 * k + 1
    b = ac.Batch(specs, dtype=dtype)
    try:
        b.set_schedule(k)
        for i, w in enumerate(which):
            b.load(i, inits[w])
        b.step([n] * len(which))
        assert b.status() == ac.AC_OK
        got = {i: b.to_numpy(i) for i in (0, copies // 2, copies - 1, copies, copies + 1)}
    finally:
        b.close()
    for i, g in got.items():
        sim = ac.Simulation(*specs[i], dtype=dtype)
        try:
            sim.load(inits[which[i]])
            sim.set_schedule(ac.AC_VARIANT_STREAM, k)
            sim.step(n)
            assert np.array_equal(g, sim.to_numpy()), f"instance {i}"
        finally:
            sim.close()
