"""Raster read-back: every step's spikes in ascending order, whole or cut at
the caller's capacity, at network sizes around the words and ranges of the
device sort (bits of 32 neurons; a block's shared memory holds 1.75 M)."""
import ctypes

import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu

FORCE_Q16 = 300 * 65536


@pytest.fixture(scope="module")
def eng():
    import paper_1310_8478_gb300 as e
    e.build_engine()
    return e


@pytest.mark.parametrize("columns,npc", [(1, 2), (1, 31), (1, 33), (3, 341), (2, 1250), (17, 1000), (1400, 1250), (1401, 1250)])
def test_steps_are_sorted_and_cut_at_the_capacity(eng, columns, npc):
    cfg = workloads.custom(grid_x=columns, grid_y=1, neurons_per_col=npc, exc_per_col=max(1, npc * 4 // 5), fanout=1,
                           pct_ring=(100, 0, 0, 0), seed=columns + npc, thal_per_col_per_ms=0, max_delay_ms=5)
    n = columns * npc
    rng = np.random.default_rng(npc)
    # step 0: every neuron; step 2: one; step 3: none; step 4: a random tenth
    some = np.sort(rng.choice(n, max(1, n // 10), replace=False))
    at = {0: np.arange(n), 2: np.array([n - 1]), 4: some}
    t = np.concatenate([np.full(len(g), k) for k, g in at.items()])
    g = np.concatenate(list(at.values()))
    with eng.Network(cfg, raster_capacity=4 * n + 64) as net:
        net.set_stimulus(t, g, np.full(len(g), FORCE_Q16))
        net.run(5)
        rt, rg = net.raster()
        assert net.counters()["spikes"] == len(rt)
        assert np.all(np.diff(rt) >= 0)
        for k in range(5):
            step = rg[rt == k]
            assert np.all(np.diff(step) > 0)
            assert set(at.get(k, [])) <= set(step.tolist())
        assert np.array_equal(rg[rt == 0], np.arange(n))
        # a second read, and one cut inside step 0 and inside step 4
        again = net.raster()
        assert np.array_equal(again[0], rt) and np.array_equal(again[1], rg)
        for cap in {max(1, n // 2), len(rt) - 1}:
            buf = np.full(cap + 1, -7, eng.snn.SPIKE_DTYPE)
            got = ctypes.c_size_t()
            rc = net._lib.snn_read_raster(net.h, 0, 5, buf.ctypes.data_as(ctypes.c_void_p), cap, ctypes.byref(got))
            assert rc == eng.snn.ETRUNC and got.value == len(rt)
            assert np.array_equal(buf["t"][:cap], rt[:cap]) and np.array_equal(buf["gid"][:cap], rg[:cap])
            assert buf["gid"][cap] == -7
