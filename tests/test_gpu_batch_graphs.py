"""GPU checks of the batch's captured launches: long calls replay a few steps'
graph and give the single contexts' bits, and keep no memory by their length."""

import numpy as np
import pytest

from inputs import workloads as W

from helpers import BatchRun, GpuContext

pytestmark = pytest.mark.gpu


def _boxes():
    return [W.box((2, 2, 2), N, (0.0, 0.0, 0.0), (2000.0, 2000.0, 2000.0), (True, True, False), seed=N) for N in (3, 4, 5, 6)]


@pytest.mark.parametrize("steps", [[1], [7], [8], [9], [16], [23], [3, 8, 2, 17, 1]])
def test_any_number_of_steps_gives_the_single_contexts_bits(cuda_device, steps):
    wls = _boxes()
    with BatchRun(wls) as b:
        for n in steps:
            b.step(n)
        got = b.states()
    for wl, q in zip(wls, got):
        with GpuContext(wl, precision=1) as g:
            g.step(sum(steps))
            assert np.array_equal(g.state(), q)


def _resident():
    with open("/proc/self/statm") as f:
        return int(f.read().split()[1]) * 4096


def test_long_calls_keep_no_memory_by_their_length(cuda_device):
    """24,000 kernel nodes, a thousand steps of four orders, hold at least the
    launch's arguments each, some 300 bytes, and with the graph's own records
    several times that: 7 MB at the least for every step count.  Graphs of a
    few steps hold less than a megabyte in all."""
    import torch
    with BatchRun(_boxes()) as b:
        for n in (16, 17, 18, 19, 20, 21, 22, 23):
            b.step(n)
        torch.cuda.synchronize()
        before = _resident()
        for n in (1000, 1001, 1002, 1003):
            b.step(n)
        assert _resident() - before <= 8 * 2 ** 20
