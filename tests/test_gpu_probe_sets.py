"""Changing the probes is cheap (GPU, through the C ABI): a program that follows a
structure sets them anew every few steps."""
import time

import numpy as np
import pytest

from workloads import case

from gpu_helpers import require_cuda

pytestmark = pytest.mark.gpu

SMALL = case("channel_64x32x32").with_(n_modes=20)


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    require_cuda()


def test_set_probes_prepares_no_graph():
    """A copy of the table: 12 us, against 240 (one launch per step) to 540 with two graphs."""
    from paper_2205_02774_gb300.channel import Channel
    g = Channel.from_case(SMALL.with_(nx=128, ny=64, nz=76))
    times = []
    for k in range(31):
        xyz = np.array([[k, 1, 2], [3, k, 4]])
        t = time.perf_counter()
        g.set_probes(xyz)
        times.append(time.perf_counter() - t)
        g.step_probed(2)
    assert np.median(times) < 1e-4, times
    g.close()


# the graphs come with the call that completes two blocks of 20 steps, or not at all
@pytest.mark.parametrize("calls", [(20, 19, 20, 5), (5, 40, 21), (39, 1, 1, 60), (100,), (19, 19, 19)])
@pytest.mark.parametrize("streaming", ["pull", "aa"])
def test_series_however_it_is_called(calls, streaming):
    from paper_2205_02774_gb300.channel import Channel
    c = SMALL.with_(nx=64, ny=16, nz=12, stats_every=10, streaming=streaming)
    a, b = (Channel.from_case(c, check_every=13, mass_tol=0.5) for _ in range(2))
    for xyz in ([[0, 0, 0], [63, 15, 11], [5, 6, 7]], [[1, 2, 3]]):
        for g in (a, b):
            g.set_probes(np.array(xyz))
        for n in calls:
            one = np.concatenate([b.step_probed(1) for _ in range(n)])
            assert np.array_equal(a.step_probed(n), one), n
    assert np.array_equal(a.get_state(), b.get_state())
    a.close()
    b.close()
