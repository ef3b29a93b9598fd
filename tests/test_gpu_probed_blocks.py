"""Probed steps replayed in blocks (GPU, through the C ABI).

step_probed takes whole blocks of steps from graphs that sample the probes beside
the next step (in place: after their own); the series must be bit-identical to
the one taken a step at a time, whatever the first step index, call after call
and after the probes or the tile change."""
import numpy as np
import pytest

from workloads import case

from gpu_helpers import require_cuda

pytestmark = pytest.mark.gpu

SMALL = case("channel_64x32x32").with_(n_modes=20)


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    require_cuda()


# one launch of all rows, inner and wall rows apart (76 planes), odd rows; blocks of 20, 16 and 21 steps
@pytest.mark.parametrize("dims,kw", [((64, 16, 12), dict()), ((64, 16, 12), dict(streaming="aa", storage="fp16sr")),
                                     ((128, 64, 76), dict(stats_every=0)), ((65, 9, 8), dict(stats_every=7)),
                                     ((64, 8, 6), dict(streaming="aa", stats_every=7, bc_x="periodic", force=(1e-6, 0.0, 0.0)))])
def test_series_of_blocks(dims, kw):
    from paper_2205_02774_gb300.channel import Channel
    nx, ny, nz = dims
    c = SMALL.with_(nx=nx, ny=ny, nz=nz, **kw)
    a = Channel.from_case(c, check_every=13, mass_tol=0.5)
    b = Channel.from_case(c, check_every=13, mass_tol=0.5)
    r = np.random.default_rng(nx)
    for n_probes, n, tile in ((3, 47, None), (200, 64, None), (1, 21, (1, 4, 4)), (1, 50, None)):
        xyz = np.stack([r.integers(0, m, n_probes) for m in dims], axis=1)
        for g in (a, b):
            g.set_probes(xyz)
            if tile:
                g.set_tile(*tile)
        u = a.step_probed(n)
        one = np.concatenate([b.step_probed(1) for _ in range(n)])
        assert u.shape == (n, n_probes, 3) and np.isfinite(u).all()
        assert np.array_equal(u, one)
    assert np.array_equal(a.get_state(), b.get_state())
    a.close()
    b.close()
