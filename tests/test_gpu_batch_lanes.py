"""Small FP32 lattices in a batch that fills the GPU (GPU, through the C ABI).

Alone such a lattice takes one cell per lane; whatever the batch's other members
make of its launches, its populations, planes and statistics must be those of
the same lattice alone, bit for bit, over whole blocks and a remainder."""
import numpy as np
import pytest

from workloads import case

from gpu_helpers import require_cuda

pytestmark = pytest.mark.gpu

SMALL = case("channel_64x32x32").with_(n_modes=20)
# 7 x 98 304 cells and one more: above the 622 592 cells up to which a lattice takes one cell per lane
CASES = [SMALL.with_(nx=96, ny=32, nz=32, stats_every=5, seed=1),
         SMALL.with_(nx=96, ny=32, nz=32, stats_every=10, collision="bgk", seed=2),
         SMALL.with_(nx=96, ny=32, nz=32, stats_every=5, sponge_len=6.4, seed=3),
         SMALL.with_(nx=96, ny=32, nz=32, stats_every=2, bc_x="periodic", force=(2e-6, -1e-6, 1e-6)),
         SMALL.with_(nx=96, ny=32, nz=32, stats_every=5, bc_x="periodic", bc_y="periodic", collision="bgk",
                     force=(2e-6, 0.0, 1e-6)),
         SMALL.with_(nx=98, ny=32, nz=32, stats_every=5, seed=6),
         SMALL.with_(nx=95, ny=33, nz=32, stats_every=5, seed=7),
         SMALL.with_(nx=64, ny=32, nz=33, stats_every=5, streaming="aa", seed=8)]


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    require_cuda()


def test_members_equal_the_lattices_alone():
    from paper_2205_02774_gb300.channel import Channel
    from paper_2205_02774_gb300.serving import Batch
    steps = (47, 20, 3)  # blocks of 20 and remainders
    chans = [Channel.from_case(c, check_every=6, mass_tol=0.5) for c in CASES]
    b = Batch()
    for ch in chans:
        b.add(ch)
    assert sum(c.nx * c.ny * c.nz for c in CASES) > 4 * 152 * 32 * 32
    for n in steps:
        b.step(n)
    b.sync()
    for c, ch in zip(CASES, chans):
        g = Channel.from_case(c, check_every=6, mass_tol=0.5)
        g.step(sum(steps))
        sa, sb = g.stats(), ch.stats()
        assert sa["rc"] == sb["rc"] == 0, sb["error"]
        assert np.array_equal(g.get_state(), ch.get_state()), c
        assert np.array_equal(sa["mean_sum"], sb["mean_sum"]) and np.array_equal(sa["rey_sum"], sb["rey_sum"]), c
        if c.bc_x == "stg":
            assert np.array_equal(g.inlet(), ch.inlet()), c
        g.close()
    b.close()
    for ch in chans:
        ch.close()
