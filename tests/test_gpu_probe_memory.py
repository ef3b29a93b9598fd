"""Probe sets that are refused (GPU, through the C ABI): a set_probes call that cannot
have its table, or names a cell outside the lattice, reports it and leaves the
earlier probes in place."""
import numpy as np
import pytest

from workloads import case

from gpu_helpers import require_cuda

pytestmark = pytest.mark.gpu

SMALL = case("channel_64x32x32").with_(nx=32, ny=8, nz=8, n_modes=8)


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    require_cuda()


class _Full:
    """torch whose allocator has no memory left."""

    class cuda:
        @staticmethod
        def caching_allocator_alloc(*args):
            raise MemoryError


def test_set_probes_without_memory_keeps_the_probes():
    from paper_2205_02774_gb300.capi import StgError, STG_ERR_NOMEM
    from paper_2205_02774_gb300.channel import Channel
    a, b = (Channel.from_case(SMALL) for _ in range(2))
    few = np.array([[3, 2, 1], [31, 7, 0]])
    many = np.stack([np.arange(20) % n for n in (32, 8, 8)], axis=1)
    for g in (a, b):
        g.set_probes(few)
        g.step_probed(60)  # the series buffer of the calls below
    real = a._allocator.torch
    a._allocator.torch = _Full
    try:
        with pytest.raises(StgError) as e:
            a.set_probes(many)
        assert e.value.code == STG_ERR_NOMEM
    finally:
        a._allocator.torch = real
    for n in (1, 45, 3):  # single steps, blocks and both
        assert np.array_equal(a.step_probed(n), b.step_probed(n))
    for g in (a, b):
        g.set_probes(many)
    assert np.array_equal(a.step_probed(21), b.step_probed(21))
    a.close()
    b.close()


def test_a_refused_set_keeps_the_series_shape():
    from paper_2205_02774_gb300.capi import StgError, STG_ERR_INVALID
    from paper_2205_02774_gb300.channel import Channel
    a, b = (Channel.from_case(SMALL) for _ in range(2))
    few = np.array([[3, 2, 1], [31, 7, 0]])
    for g in (a, b):
        g.set_probes(few)
    with pytest.raises(StgError) as e:
        a.set_probes(np.array([[32, 0, 0], [0, 0, 0], [0, 0, 0]]))
    assert e.value.code == STG_ERR_INVALID
    u, v = a.step_probed(5), b.step_probed(5)
    assert u.shape == (5, 2, 3) and np.array_equal(u, v)
    a.close()
    b.close()
