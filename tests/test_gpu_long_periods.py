"""Sampling periods of any length (GPU, through the C ABI): preparing the step
graphs takes the same time for every period, and a long one samples when it is due."""
import time

import numpy as np
import pytest

from workloads import case

from gpu_helpers import require_cuda

pytestmark = pytest.mark.gpu

SMALL = case("channel_64x32x32").with_(nx=16, ny=6, nz=5, n_modes=8)


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    require_cuda()


def _seconds(period):
    from paper_2205_02774_gb300.channel import Channel
    t = time.perf_counter()
    g = Channel.from_case(SMALL.with_(stats_every=period))
    g.set_tile(1, 4, 4)
    g.step(3)
    assert g.stats()["n_samples"] == 0
    s = time.perf_counter() - t
    g.close()
    return s


@pytest.mark.parametrize("period", [10 ** 9, 2 ** 31 - 1])
def test_create_and_set_tile_take_no_longer(period):
    _seconds(1000)
    assert _seconds(period) < _seconds(1000) + 1.0


# the phases where a period's first samples of each parity fall; blocks of 16, 18, 21, 256, 257 (none) steps
@pytest.mark.parametrize("period", [1, 2, 3, 4, 7, 256, 257, 1001])
def test_samples_fall_where_they_are_due(period):
    from paper_2205_02774_gb300.channel import Channel
    c = SMALL.with_(stats_every=period)
    g = Channel.from_case(c)
    one = Channel.from_case(c)
    n = 2 * period + 3
    g.step(n)
    for _ in range(n):
        one.step(1)
    a, b = g.stats(), one.stats()
    assert a["n_samples"] == b["n_samples"] == n // period
    assert np.array_equal(g.get_state(), one.get_state())
    assert np.array_equal(a["mean_sum"], b["mean_sum"]) and np.array_equal(a["rey_sum"], b["rey_sum"])
    assert (np.abs(a["mean_sum"]).max() > 0) == (a["n_samples"] > 0)
    g.close()
    one.close()
