"""Inlet velocity planes of a block of steps (GPU, through the C ABI).

The planes are computed for several steps by one launch (4, then 16 at a time)
or for one step alone, over chunks of the modes; the sum over the modes is in
the same order in every form, so the planes must be bit-identical however the
steps are split, and match the oracle as a plane computed alone does."""
import numpy as np
import pytest

from workloads import case

from gpu_helpers import require_cuda, pair

pytestmark = pytest.mark.gpu

SMALL = case("channel_64x32x32").with_(nx=8)


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    require_cuda()


# mode counts at the edges of the chunks (32 and 96 modes), planes that are not
# whole 32-node tiles, blocks of 16, 21, 40 and 50 steps (the last chunks 12, 1, 4, 14)
@pytest.mark.parametrize("ny,nz,n_modes,stats_every", [(32, 32, 100, 0), (5, 33, 1, 7), (33, 7, 32, 40),
                                                       (31, 9, 33, 10), (64, 5, 96, 50), (40, 3, 97, 7)])
def test_planes_of_a_block(ny, nz, n_modes, stats_every):
    c = SMALL.with_(ny=ny, nz=nz, n_modes=n_modes, stats_every=stats_every, t_filter=4.0)
    gpu, orc = pair(c)
    one, _ = pair(c)
    done = 0
    for n in (1, 17, 70, 131):
        gpu.step(n - done)
        orc.step(n - done)
        for _ in range(n - done):
            one.step(1)
        done = n
        u, u_or = gpu.inlet(), orc.inlet()
        assert np.array_equal(u, one.inlet()), n
        assert np.abs(u - u_or).max() <= 1e-5 * np.abs(u_or).max(), n
    assert np.array_equal(gpu.get_state(), one.get_state())
    gpu.close()
    one.close()
