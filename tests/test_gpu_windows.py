"""Plasticity windows and resident grids against the oracle, where they can go
wrong: columns that are no multiple of 32 neurons, slices, the shortest and
longest delays, calls that end inside, at and behind a window or a period,
external events, activity that stops a resident grid, FP64, and step kernels
that start a window's deferral in its middle.  Everything is bit-exact."""
import numpy as np
import pytest

import workloads
from test_gpu_parity import assert_same_run, gpu_net

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eng():
    import paper_1310_8478_gb300 as e
    e.build_engine()
    return e


def _cfg(gx, gy, npc, m, mix=(40, 30, 20, 10), **kw):
    kw.setdefault("exc_per_col", max(1, npc * 4 // 5))
    return workloads.custom(grid_x=gx, grid_y=gy, neurons_per_col=npc, fanout=m,
                            pct_ring=mix if gx * gy > 1 else (100, 0, 0, 0), **kw)


CASES = {
    # calls of every remainder of a window, across two periods of 70 ms
    "ragged_columns": (_cfg(3, 2, 333, 61, seed=61, deriv_period_ms=70), [4, 50, 3, 51, 1, 49, 101, 5]),
    "one_column_odd": (_cfg(1, 1, 77, 40, seed=62, thal_per_col_per_ms=3, deriv_period_ms=60), [50, 7, 64, 99]),
    # three neurons per column, a single excitatory one
    "tiny_columns": (_cfg(5, 4, 3, 9, seed=63, exc_per_col=1, thal_per_col_per_ms=1), [60, 120]),
    "longest_delay": (_cfg(2, 2, 100, 33, seed=64, max_delay_ms=31, thal_per_col_per_ms=2), [55, 130]),
    "shortest_delay": (_cfg(2, 3, 65, 24, seed=65, max_delay_ms=1, w_exc0_q16=7 * 65536, thal_per_col_per_ms=2), [120]),
    # thousands of drive events per column and window are not drawn ahead
    "strong_drive": (_cfg(2, 1, 200, 20, seed=66, thal_per_col_per_ms=40, thal_amp_q16=4 * 65536), [53, 60]),
    # runs away: the resident grid stops, the step kernels go on and defer
    "runaway": (_cfg(2, 2, 400, 400, seed=67, w_exc0_q16=8 * 65536, thal_per_col_per_ms=2, deriv_period_ms=90), [40, 120, 70]),
    # columns whose trains leave room for fewer warps' tables
    "wide_columns": (_cfg(2, 1, 1801, 30, seed=74, thal_per_col_per_ms=9, deriv_period_ms=50), [60, 49]),
    # other STDP tables, the depression too wide for 15 bits
    "wide_depression": (_cfg(2, 2, 100, 50, seed=68, a_minus_mv=1.0, tau_plus_ms=12.0, thal_per_col_per_ms=2), [75, 75]),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_calls_of_any_length_equal_the_oracle(eng, orc, name):
    cfg, calls = CASES[name]
    o = orc.Oracle(cfg)
    with gpu_net(eng, cfg) as n:
        for steps in calls:
            o.run(steps)
            n.run(steps)
            assert_same_run(o, n)
        assert n.counters()["spikes"] > 10          # something happened


def test_fp64_and_events_inside_windows(eng, orc):
    cfg = _cfg(2, 2, 90, 45, seed=69)
    rng = np.random.default_rng(3)
    t, g = rng.integers(0, 130, 300), rng.integers(0, 360, 300)
    t.sort()
    q = np.full(300, 25 * 65536)
    o = orc.Oracle(cfg)
    o.set_stimulus(t, g, q)
    o.run(140)
    with gpu_net(eng, cfg) as n:
        n.set_stimulus(t, g, q)
        n.run(140)
        assert_same_run(o, n)
    cfg["flags"] = eng.snn.FP64
    o = orc.Oracle(cfg, flags=4)
    o.run(140)
    with gpu_net(eng, cfg) as n:
        n.run(140)
        ot, og = o.raster()
        gt, gg = n.raster()
        assert np.array_equal(gt, ot) and np.array_equal(gg, og)
        s, x = o.neurons(), n.neurons_f64()
        assert np.array_equal(x["v"], s["vd"]) and np.array_equal(x["u"], s["ud"])
        w, sd = n.weights()
        assert np.array_equal(w, o.synapses()["w"]) and np.array_equal(sd, o.synapses()["sd"])


def test_resident_and_step_kernels_share_a_net(eng, orc):
    """Windows of one call and single steps of the next, checkpoints between
    them, and the spike lists that a later launch shape delivers from."""
    cfg = _cfg(3, 3, 120, 60, seed=70, thal_per_col_per_ms=2, deriv_period_ms=110)
    o = orc.Oracle(cfg)
    o.run(300)
    with gpu_net(eng, cfg) as n, gpu_net(eng, cfg) as other:
        n.run(64)
        for _ in range(20):
            n.step()
        n.run(50)
        other.load_state(n.save_state())
        for net in (n, other):
            if net is other:
                net.set_launch(dense_permille=1001, ring_permille=0xffffffff)
            net.run(26)
            net.set_launch(dense_permille=1001, ring_permille=0xffffffff)
            net.run(40)
            net.set_launch(dense_permille=250)
            net.run(100)
            s = o.synapses()
            w, sd = net.weights()
            assert np.array_equal(w, s["w"]) and np.array_equal(sd, s["sd"])
            assert net.counters()["spikes"] == o.counters()["spikes"]
            x = net.neurons()
            assert np.array_equal(x["v"].view(np.int32), o.neurons()["v"].view(np.int32))
        assert_same_run(o, n)


@pytest.mark.parametrize("npc,m", [(1000, 300), (1250, 1125)])
def test_step_kernels_defer_inside_a_window(eng, npc, m):
    """A net too large for a resident grid: the windows of long calls against
    single steps (which never defer), whose own results the parity tests hold
    against the oracle on small nets."""
    cfg = _cfg(20, 20, npc, m, seed=71, mix=(76, 12, 8, 4) if m == 300 else (40, 30, 20, 10), deriv_period_ms=60)
    T = 150 if m == 300 else 75
    with eng.Network(cfg, raster_capacity=0) as a, eng.Network(cfg, raster_capacity=0) as b:
        a.run(T)
        for _ in range(T // 3):
            b.run(3)
        ca, cb = a.counters(), b.counters()
        assert ca == cb and ca["spikes"] > 400 * npc // 2
        for first in (0, 7 * npc, 399 * npc):
            x, y = a.synapses(first, npc, fields=("w", "sd")), b.synapses(first, npc, fields=("w", "sd"))
            assert np.array_equal(x["w"], y["w"]) and np.array_equal(x["sd"], y["sd"])
            assert np.count_nonzero(x["sd"]) > npc
        x, y = a.neurons(), b.neurons()
        assert np.array_equal(x["v"].view(np.int32), y["v"].view(np.int32))


@pytest.mark.parametrize("before", ["few_steps", "single_steps", "a_period", "a_checkpoint"])
def test_reset_restores_whatever_moved(eng, before):
    cfg = _cfg(3, 2, 130, 70, seed=72, thal_per_col_per_ms=2, deriv_period_ms=60)
    with eng.Network(cfg, raster_capacity=1 << 18) as fresh, eng.Network(cfg, raster_capacity=1 << 18) as n:
        if before == "few_steps":
            n.run(40)
        elif before == "single_steps":
            for _ in range(40):
                n.step()
        elif before == "a_period":
            n.run(61)
        else:
            other = eng.Network(cfg, raster_capacity=1 << 18)
            other.run(100)
            n.load_state(other.save_state())
            other.close()
            n.reset()
            n.run(5)
        n.reset()
        for steps in (0, 75):
            if steps:
                n.run(steps)
                fresh.run(steps)
            for a, b in zip(n.weights() + n.raster(), fresh.weights() + fresh.raster()):
                assert np.array_equal(a, b)
            assert n.counters() == fresh.counters()


@pytest.mark.parametrize("lists", [False, True], ids=["generated", "explicit"])
def test_closed_loop_of_single_steps_equals_the_oracle(eng, orc, lists):
    """One call per millisecond with that step's host events: quiet steps,
    whose successor has nothing to potentiate, between single spikes; events of
    changing number; a period's end on the way."""
    cfg = _cfg(2, 1, 60, 30, seed=73, thal_per_col_per_ms=0, deriv_period_ms=50)
    rng = np.random.default_rng(9)
    explicit = None
    if lists:
        rows = rng.integers(20, 40, 120)
        off = np.concatenate([[0], np.cumsum(rows)])
        exc = np.repeat(np.arange(120) % 60 < 48, rows)
        explicit = dict(row_off=off, tgt=rng.integers(0, 120, off[-1]),
                        delay=np.where(exc, rng.integers(1, 21, off[-1]), 1),
                        w=np.where(exc, 7 * 65536, -5 * 65536))
    T = 130
    counts = rng.integers(0, 6, T)
    t = np.repeat(np.arange(T), counts)
    g = rng.integers(0, 120, len(t))
    q = rng.integers(10, 60, len(t)) * 65536
    o = orc.Oracle(cfg, explicit=explicit)
    o.set_stimulus(t, g, q)
    o.run(T)
    ev = np.zeros(len(t), eng.snn.STIM_DTYPE)
    ev["t"], ev["gid"], ev["q16"] = t, g, q
    with gpu_net(eng, cfg, explicit=explicit) as n:
        total, quiet = 0, 0
        for k in range(T):
            got = n.run_host_counts(1, ev[t == k])
            total += got
            quiet += got == 0
        assert_same_run(o, n)
        assert total == o.counters()["spikes"] and quiet > 10 and total > 10


def _explicit(rng, cfg, rows_lo, rows_hi, w_exc):
    """Random rows of both kinds with individual delays and weights; some rows
    empty, some targets repeated or the source itself."""
    n, npc = cfg["grid_x"] * cfg["grid_y"] * cfg["neurons_per_col"], cfg["neurons_per_col"]
    rows = rng.integers(rows_lo, rows_hi, n)
    rows[rng.random(n) < 0.1] = 0
    off = np.concatenate([[0], np.cumsum(rows)])
    src = np.repeat(np.arange(n), rows)
    exc = src % npc < cfg["exc_per_col"]
    tgt = rng.integers(0, n, off[-1])
    tgt[rng.integers(0, off[-1], min(200, off[-1] // 50))] = 0     # (a Q16 input holds some 500 at wmax)
    tgt = np.where(rng.random(off[-1]) < 0.02, src, tgt)
    D = cfg["max_delay_ms"]
    return dict(row_off=off, tgt=tgt, delay=np.where(exc, rng.integers(1, D + 1, off[-1]), rng.integers(1, 4, off[-1])),
                w=np.where(exc, (w_exc * 65536 * (0.5 + rng.random(off[-1]))).astype(np.int64), -rng.integers(2, 6, off[-1]) * 65536))


LISTS = {
    # one block: no grid barrier; two, the second with a single neuron
    "one_block": (_cfg(1, 1, 31, 0, seed=81, thal_per_col_per_ms=1, deriv_period_ms=70), (5, 25), 8, [4, 50, 51, 3, 90]),
    "two_blocks": (_cfg(1, 1, 33, 0, seed=82, thal_per_col_per_ms=1, deriv_period_ms=60), (5, 25), 8, [64, 99]),
    # columns of odd size, slices across columns, the longest delay
    "ragged": (_cfg(3, 2, 111, 0, seed=83, thal_per_col_per_ms=1, deriv_period_ms=70, max_delay_ms=31), (10, 50), 6, [53, 120]),
    # runs away: trains with many spikes, drive events that are not drawn ahead
    "runaway": (_cfg(5, 4, 800, 0, seed=84, thal_per_col_per_ms=30, deriv_period_ms=40), (30, 70), 9, [30, 45]),
    # forced spikes in every neuron: more pending rows than a block lists at once
    "all_fire": (_cfg(2, 1, 45000, 0, seed=86, max_delay_ms=31), (2, 8), 3, [60]),
}


@pytest.mark.parametrize("fp64", [False, True], ids=["fp32", "fp64"])
@pytest.mark.parametrize("name", sorted(LISTS))
def test_resident_grids_of_target_lists_equal_the_oracle(eng, orc, name, fp64):
    cfg, rows, w_exc, calls = LISTS[name]
    cfg = dict(cfg, fanout=1)
    rng = np.random.default_rng(cfg["seed"])
    ex = _explicit(rng, cfg, *rows, w_exc)
    N, T = len(ex["row_off"]) - 1, sum(calls)
    t, g, q = np.sort(rng.integers(0, T, 200)), rng.integers(0, N, 200), np.full(200, 30 * 65536)
    if name == "all_fire":
        t, g, q = np.repeat(np.arange(4, 44, 4), N), np.tile(np.arange(N), 10), np.full(10 * N, 250 * 65536)
    if fp64:
        cfg["flags"] = eng.snn.FP64
    o = orc.Oracle(cfg, explicit=ex, **(dict(flags=4) if fp64 else {}))
    o.set_stimulus(t, g, q)
    with gpu_net(eng, cfg, explicit=ex) as n:
        n.set_stimulus(t, g, q)
        for k, steps in enumerate(calls):
            o.run(steps)
            n.run(steps)
            if k == 0:
                n.step()
                o.run(1)
        for a, b in zip(n.raster(), o.raster()):
            assert np.array_equal(a, b)
        s, x = o.synapses(), n.neurons_f64() if fp64 else n.neurons()
        w, sd = n.weights()
        assert np.array_equal(w, s["w"]) and np.array_equal(sd, s["sd"]) and np.count_nonzero(sd) > 10
        v = "vd" if fp64 else "v"
        assert np.array_equal(o.neurons()[v], x["v"])
        for key in ("spikes", "e_all", "e_exc", "l_exc"):
            assert n.counters()[key] == o.counters()[key], key
        assert n.counters()["spikes"] > 100


def test_resident_grid_of_a_big_column_equals_the_oracle(eng, orc):
    """Columns above 4096 neurons are generated with target lists."""
    cfg = _cfg(2, 1, 4200, 24, seed=85, thal_per_col_per_ms=20, thal_amp_q16=30 * 65536, deriv_period_ms=50, w_exc0_q16=8 * 65536)
    o = orc.Oracle(cfg)
    with gpu_net(eng, cfg) as n:
        for steps in (70, 33):
            o.run(steps)
            n.run(steps)
            assert_same_run(o, n)
        assert n.counters()["spikes"] > 100


@pytest.mark.parametrize("stdp", [True, False], ids=["stdp", "static"])
@pytest.mark.parametrize("npc,m,D", [(75, 300, 20), (130, 401, 31), (64, 13, 1), (33, 160, 16), (101, 60, 2)])
def test_ordered_delivery_chunk_by_chunk_equals_the_oracle(eng, orc, npc, m, D, stdp):
    """Event-driven steps of the step kernels: buckets of a few synapses to a
    whole row, at any alignment, on a torus whose rings lead back."""
    cfg = _cfg(2, 3, npc, m, seed=90, max_delay_ms=D, thal_per_col_per_ms=2, w_exc0_q16=4 * 65536, deriv_period_ms=60)
    if not stdp:
        cfg["flags"] = eng.snn.STDP_OFF
    o = orc.Oracle(cfg, **({} if stdp else dict(flags=1)))
    o.run(130)
    with gpu_net(eng, cfg) as n:
        n.set_launch(dense_permille=1001)
        n.run(130)
        assert_same_run(o, n)
        assert n.counters()["spikes"] > 100
