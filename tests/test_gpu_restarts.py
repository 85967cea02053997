"""Restarts and long lives of a net: what a grid that gave up, a clock far from
0, a refused allocation or a read-back on a full device leave behind.  Device
state that no call can make is written into the net's own blocks, which the
allocator hook knows."""
import numpy as np
import pytest

import workloads
from device_blocks import Blocks, WIN_BAR, up, window_block
from test_gpu_parity import assert_same_run

pytestmark = pytest.mark.gpu

@pytest.fixture(scope="module")
def eng():
    import paper_1310_8478_gb300 as e
    e.build_engine()
    return e


def _cfg(gx, gy, npc, m, **kw):
    kw.setdefault("exc_per_col", npc * 4 // 5)
    return workloads.custom(grid_x=gx, grid_y=gy, neurons_per_col=npc, fanout=m,
                            pct_ring=(40, 30, 20, 10) if gx * gy > 1 else (100, 0, 0, 0), **kw)


@pytest.mark.parametrize("restart", ["reset", "load"])
def test_a_restart_clears_both_inputs_of_a_resident_grid(eng, orc, restart):
    import torch
    cfg = _cfg(3, 2, 130, 60, seed=91, thal_per_col_per_ms=2, deriv_period_ms=70)
    o = orc.Oracle(cfg)
    o.run(90)
    with Blocks() as b, eng.Network(cfg, raster_capacity=1 << 20) as n:
        N = n.n_neurons
        n.run(30)
        state = n.save_state()
        n.run(20)
        words = b.words(window_block(b, N))
        words[len(words) - up(4 * N) // 4:] = 15 * 65536
        torch.cuda.synchronize()
        if restart == "reset":
            n.reset()
            n.run(90)
            assert_same_run(o, n)
        else:
            n.load_state(state)
            n.run(60)
            s, x = o.synapses(), n.neurons()
            w, sd = n.weights()
            assert np.array_equal(w, s["w"]) and np.array_equal(sd, s["sd"])
            assert np.array_equal(x["v"].view(np.int32), o.neurons()["v"].view(np.int32))
            assert n.counters()["spikes"] == o.counters()["spikes"]


def test_a_grid_barrier_that_runs_out_is_an_error_until_a_restart(eng, orc):
    """Arrivals that start a million short: every block gives up at its first
    barrier."""
    import torch
    cfg = _cfg(4, 3, 130, 60, seed=92, thal_per_col_per_ms=2, deriv_period_ms=70)
    o = orc.Oracle(cfg)
    o.run(90)
    with Blocks() as b, eng.Network(cfg, raster_capacity=1 << 20) as n:
        n.run(30)
        state = n.save_state()
        for restart in ("reset", "load"):
            b.words(window_block(b, n.n_neurons))[WIN_BAR] = -1000000
            torch.cuda.synchronize()
            for _ in range(2):
                with pytest.raises(eng.snn.SnnError) as e:
                    n.run(50)
                assert e.value.code == eng.snn.ETIMEOUT
            if restart == "reset":
                n.reset()
                n.run(90)
                assert_same_run(o, n)
            else:
                n.load_state(state)
                n.run(60)
                w, sd = n.weights()
                assert np.array_equal(w, o.synapses()["w"]) and np.array_equal(sd, o.synapses()["sd"])
                assert n.counters()["spikes"] == o.counters()["spikes"] and n.counters()["error"] == 0


def test_a_drive_whose_events_per_window_pass_32_bits(eng):
    """50 steps of 85 899 346 events are 4 more than 2^32: too many to be drawn
    ahead by a resident grid; one call against short ones."""
    cfg = _cfg(1, 1, 300, 20, seed=93, thal_per_col_per_ms=85899346, thal_amp_q16=2, wmax_q16=65536, w_exc0_q16=65536)
    with eng.Network(cfg, raster_capacity=1 << 16) as a, eng.Network(cfg, raster_capacity=1 << 16) as b:
        a.run(50)
        for _ in range(25):
            b.run(2)
        for x, y in zip(a.raster() + a.weights(), b.raster() + b.weights()):
            assert np.array_equal(x, y)
        assert a.counters() == b.counters() and a.counters()["spikes"] > 10


def test_a_drive_switched_off_does_not_hide_its_events(eng):
    """A net with target lists and more drive events per step than every block
    should look at takes no grid, whether the drive is on or off."""
    cfg = _cfg(1, 1, 300, 1, seed=94, thal_per_col_per_ms=5000, thal_amp_q16=100)
    ex = dict(row_off=np.arange(301), tgt=np.arange(300)[::-1].copy(), delay=np.ones(300, np.int64), w=np.ones(300, np.int64))
    with Blocks() as b, eng.Network(cfg, raster_capacity=1 << 16, explicit=ex) as n:
        asked = len(b.asked)
        n.set_thalamic(False)
        n.set_launch(neuron_block=128)
        n.set_thalamic(True)
        assert len(b.asked) == asked
        n.run(20)


# ---------------------------------------------------------------------------
# a clock beyond 2^30: the distance to the time stamp of a neuron that never
# fired, -2^30, is then beyond an int
# ---------------------------------------------------------------------------
NEVER = -(1 << 30)


def _later(eng, cfg, state, n_stored, ahead):
    """The checkpoint with its clock, and every spike's time, moved ahead."""
    import ctypes
    N, D = cfg["grid_x"] * cfg["grid_y"] * cfg["neurons_per_col"], cfg["max_delay_ms"]
    b = bytearray(state)
    head = 32 + ctypes.sizeof(eng.snn.SnnConfig)
    assert len(b) == head + N * 24 + D * N * 4 + D * 8 + n_stored * 8 + 184
    np.frombuffer(b, np.int32, 2, 24)[:] += ahead              # t, raster_t0
    hl = np.frombuffer(b, np.int32, 2 * N, head + 12 * N)[1::2]
    last = np.frombuffer(b, np.int32, N, head + 20 * N)
    assert np.count_nonzero(last == NEVER) > 2 and np.count_nonzero(last != NEVER) > 2
    for x in (hl, last):
        x[x != NEVER] += ahead
    return bytes(b)


LATE = {  # launch shape, net, its calls from the checkpoint on
    "resident": ({}, _cfg(3, 2, 110, 40, seed=95, deriv_period_ms=60, thal_per_col_per_ms=0), [50, 47]),
    "single_steps": ({}, _cfg(2, 2, 110, 40, seed=95, deriv_period_ms=60, thal_per_col_per_ms=0), [1] * 70),
    "explicit": ({}, _cfg(2, 1, 150, 1, seed=96, deriv_period_ms=60, thal_per_col_per_ms=0), [50, 3, 30]),
    # windows of the step kernels, whose dense steps leave their STDP to them
    "windows": ({}, _cfg(8, 8, 1000, 200, seed=97, deriv_period_ms=60, thal_per_col_per_ms=0), [90]),
}
for _mode, _shape in (("sparse", dict(dense_permille=1001)), ("staged", dict(dense_permille=1001, staged_permille=1)),
                      ("dense", dict(dense_permille=1)), ("ring", dict(dense_permille=1001, ring_permille=0xffffffff))):
    LATE[_mode] = (_shape, LATE["single_steps"][1], [70])


@pytest.mark.parametrize("name", sorted(LATE))
def test_a_clock_beyond_two_to_the_thirty_changes_nothing(eng, name):
    shape, cfg, calls = LATE[name]
    ahead = ((1 << 30) // 960 + 1) * 960                        # whole rings, periods and windows' slots
    N, T = cfg["grid_x"] * cfg["grid_y"] * cfg["neurons_per_col"], 40 + sum(calls)
    rng = np.random.default_rng(5)
    ex = None
    if name == "explicit":
        off = np.arange(N + 1) * 30
        exc = np.repeat(np.arange(N) % 150 < 120, 30)
        ex = dict(row_off=off, tgt=rng.integers(0, N, off[-1]), delay=np.where(exc, rng.integers(1, 21, off[-1]), 1),
                  w=np.where(exc, 6 * 65536, -5 * 65536))
    # every step some of the first half fire; later, in every sixth step, nearly half of them at once
    few = 4 * max(1, N // 400)
    t = np.repeat(np.arange(T), few)
    g = rng.integers(0, N // 2, len(t))
    many = np.arange(60, T, 6)
    t, g = np.concatenate([t, np.repeat(many, N // 2)]), np.concatenate([g, np.tile(np.arange(N // 2), len(many))])
    order = np.argsort(t, kind="stable")
    t, g, q = t[order], g[order], np.full(len(t), 300 * 65536)
    with eng.Network(cfg, raster_capacity=1 << 22, explicit=ex) as a, \
            eng.Network(cfg, raster_capacity=1 << 22, explicit=ex) as b:
        for n in (a, b):
            n.set_launch(**shape)
        a.set_stimulus(t[t < 40], g[t < 40], q[t < 40])
        a.run(40)
        stored = N * ((cfg["fanout"] + 7) // 8 * 8) if ex is None else len(ex["tgt"])
        b.load_state(_later(eng, cfg, a.save_state(), stored, ahead))
        a.set_stimulus(t, g, q)
        b.set_stimulus(t[t >= 40] + ahead, g[t >= 40], q[t >= 40])
        for steps in calls:
            a.run(steps)
            b.run(steps)
        assert b.t == a.t + ahead
        for x, y in zip(a.weights() + tuple(a.neurons().values()), b.weights() + tuple(b.neurons().values())):
            assert np.array_equal(x, y)
        ta, ga = a.raster(40, T)
        tb, gb = b.raster(40 + ahead, T + ahead)
        assert np.array_equal(ta + ahead, tb) and np.array_equal(ga, gb) and len(ta) > 20
        ca, cb = a.counters(), b.counters()
        assert all(ca[k] == cb[k] for k in ("spikes", "e_all", "e_exc", "l_exc")) and cb["error"] == 0
        if name in ("windows", "dense"):
            assert a.profile()["dense_steps"] == b.profile()["dense_steps"] > 3


@pytest.mark.parametrize("batch", [False, True], ids=["alone", "batch"])
def test_a_refused_stimulus_leaves_no_graph_with_the_old_one(eng, batch):
    """The events of an earlier call are gone once a larger upload was refused,
    also from the captured steps."""
    cfg = _cfg(1, 1, 200, 30, seed=98, thal_per_col_per_ms=1)
    t = np.repeat(np.arange(200), 3)
    g, q = np.arange(len(t)) % 200, np.full(len(t), 40 * 65536)
    more = np.repeat(np.arange(200), 50)
    with Blocks() as b, eng.Network(cfg, raster_capacity=1 << 18) as n, eng.Network(cfg, raster_capacity=1 << 18) as ref:
        runs = []
        for x in (n, ref):
            x.set_launch(dense_permille=1001, graph_steps=10)
            runs.append(eng.Batch([x], graph_steps=10) if batch else x)
            x.set_stimulus(t, g, q)
            runs[-1].run(60)
        b.refuse = lambda size: True
        with pytest.raises(eng.snn.SnnError) as e:
            n.set_stimulus(more, np.arange(len(more)) % 200, np.full(len(more), 40 * 65536))
        assert e.value.code == eng.snn.ENOMEM
        b.refuse = lambda size: False
        ref.set_stimulus([], [], [])
        for r in runs:
            r.run(60)
        for x, y in zip(n.raster() + n.weights(), ref.raster() + ref.weights()):
            assert np.array_equal(x, y)
        if batch:
            for r in runs:
                r.close()


@pytest.mark.parametrize("pinch", ["large_blocks", "until_windows_go"])
def test_a_read_back_keeps_or_returns_the_windows_arrays(eng, pinch):
    """Where the large scratch of a read-back is not to be had, small chunks are
    tried before the arrays of the plasticity windows make room; where those do,
    they are taken again after the read."""
    cfg = _cfg(2, 2, 1000, 100, seed=99, deriv_period_ms=60)
    with Blocks() as b, eng.Network(cfg, raster_capacity=0) as n, eng.Network(cfg, raster_capacity=0) as ref:
        n.run(70)
        ref.run(70)
        w, sd = ref.weights()
        ref.close()
        win = window_block(b, n.n_neurons)
        largest = 1024 * 100 * 4
        b.refuse = (lambda size: size > largest) if pinch == "large_blocks" else (lambda size: win in b.live)
        held = n.synapses(0, 4000, fields=("w", "sd"))
        assert np.array_equal(held["w"], w) and np.array_equal(held["sd"], sd)
        window_block(b, n.n_neurons)
        assert (win in b.live) == (pinch == "large_blocks")
        b.refuse = lambda size: False
        n.run(70)
        assert n.counters()["spikes"] > 100
