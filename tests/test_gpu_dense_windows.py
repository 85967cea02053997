"""Dense steps that leave their STDP to a window's pass, in the launch of the
dense pass (nets of 8 to 64 M plastic synapses), in one of their own (larger
ones) and in those of a batch, against calls of at most three steps, which
never leave any: bit-exact, across the ends of periods."""
import numpy as np
import pytest

import workloads
from device_blocks import Blocks, WIN_BYTES, up, window_block

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eng():
    import paper_1310_8478_gb300 as e
    e.build_engine()
    return e


def _cfg(side, period, m=1125, seed=71, **kw):
    return workloads.custom(grid_x=side, grid_y=side, fanout=m, pct_ring=(40, 30, 20, 10) if side > 1 else (100, 0, 0, 0),
                            seed=seed, deriv_period_ms=period, **kw)


def _busiest_train(blocks, n):
    """Most spikes of a neuron in the last window whose STDP went to its pass:
    a resident grid stops at the second dense step, so that a train of many is
    one of dense steps that deferred."""
    N = n.n_neurons
    at = (WIN_BYTES + up(8 * N)) // 4
    words = blocks.words(window_block(blocks, N))[at:at + 2 * N].cpu().numpy().view(np.uint64)
    return int(max(bin(int(w) & ((1 << 56) - 1)).count("1") for w in words[::7]))


def _same(x, y):
    for k in ("t", "spikes", "e_all", "e_exc", "l_exc", "error"):
        assert x.counters()[k] == y.counters()[k], k
    npc, N = x.cfg["neurons_per_col"], x.n_neurons
    for first in {0, N // 2 // npc * npc, N - npc}:
        a, b = x.synapses(first, npc, fields=("w", "sd")), y.synapses(first, npc, fields=("w", "sd"))
        assert np.array_equal(a["w"], b["w"]) and np.array_equal(a["sd"], b["sd"])
        assert np.count_nonzero(a["sd"]) > npc
    for k, v in x.neurons().items():
        assert np.array_equal(v.view(np.int32), y.neurons()[k].view(np.int32))
    for a, b in zip(x.raster(), y.raster()):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("merged", [True, False], ids=["one_launch", "two_launches"])
@pytest.mark.parametrize("side", [3, 5, 7])
def test_deferred_dense_steps_of_a_mid_size_net(eng, side, merged):
    """10, 28 and 55 M plastic synapses; the delivery and the dense pass in one
    launch, or in two of other block sizes."""
    cfg, calls = _cfg(side, 90), [47, 60, 40]
    cap = side * side * 1250 * sum(calls)
    with Blocks() as b, eng.Network(cfg, raster_capacity=cap) as n:
        if not merged:
            n.set_launch(dense_block=256)
        for steps in calls:
            n.run(steps)
        assert _busiest_train(b, n) > 20
        assert n.profile()["dense_steps"] > 40
        with eng.Network(cfg, raster_capacity=cap) as ref:
            for _ in range(sum(calls) // 3):
                ref.run(3)
            assert ref.profile()["dense_steps"] > 40
            _same(n, ref)


def test_windows_of_a_batch(eng):
    """Nets below and above 64 M plastic synapses with periods of 120 and 130 ms,
    and two without windows; calls that end in single steps."""
    cfgs = [_cfg(5, 120, seed=72), _cfg(8, 130, seed=73), _cfg(1, 60, m=100, seed=74), _cfg(2, 90, m=400, seed=75)]
    calls = [60, 57, 33, 30]
    with Blocks() as b:
        nets = [eng.Network(c, raster_capacity=1 << 25) for c in cfgs]
        batch = eng.Batch(nets, graph_steps=10)
        for k, steps in enumerate(calls):
            batch.run(steps)
            for n in nets[:2] if k == 1 else []:       # the window of steps 60 to 109
                assert _busiest_train(b, n) > 20
                assert n.profile()["dense_steps"] > 40
        batch.close()
        for c, n in zip(cfgs, nets):
            with eng.Network(c, raster_capacity=1 << 25) as ref:
                for _ in range(sum(calls) // 3):
                    ref.run(3)
                _same(n, ref)
            n.close()
