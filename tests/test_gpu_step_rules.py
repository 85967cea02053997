"""Which form a call's steps take, and what the choice costs: the rules that
pick among resident grids, plasticity windows, captured graphs and single steps
change no result, so they are held by what they leave on the device and by the
time of one form against another, with a margin well below the ratio that a
wrong choice gives."""
import time

import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eng():
    import paper_1310_8478_gb300 as e
    e.build_engine()
    return e


def test_the_neuron_update_is_one_wave_at_any_block_size(eng):
    """ms of the update of 5.1 M neurons, small blocks against the default
    (blocks that hold the spike lists of 32 warps each take 1.5 times as long at
    128 threads and 2.4 times at 32; blocks of their own size 1.0 and 1.1)."""
    with eng.Network(workloads.workload("grid64_m16"), raster_capacity=0) as n:
        n.run(20)
        ms = {}
        for _ in range(3):
            for block in (256, 128, 32):
                n.set_launch(neuron_block=block)
                n.step()
                n.set_profile(True)
                n.run(10)
                ms[block] = min(ms.get(block, 1e9), n.profile()["neuron"][1])
                n.set_profile(False)
        assert max(ms[128], ms[32]) < 1.3 * ms[256], ms
