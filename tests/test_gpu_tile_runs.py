"""The launch tile sets the runs of planes (GPU, through the C ABI): a tile takes effect,
and populations and statistics do not depend on it on lattices whose runs differ."""
import numpy as np
import pytest

from workloads import case, perturbed_equilibrium_field

from gpu_helpers import require_cuda

pytestmark = pytest.mark.gpu

SMALL = case("channel_64x32x32").with_(n_modes=20)


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    require_cuda()


@pytest.mark.parametrize("storage", ["fp32", "fp16s"])
def test_a_set_tile_takes_effect(storage):
    """64x32x1024: a warp that walks a whole column of 1024 planes takes many times as long
    as the many short runs of the default tile (30 and more times in FP32: the margin is 3)."""
    from paper_2205_02774_gb300.channel import Channel
    g = Channel.from_case(SMALL.with_(nx=64, ny=32, nz=1024, storage=storage, stats_every=0))
    ms = {}
    for tile in [(1, 8, 24), (1, 0, 0), (1, 0, 24), (1, 8, 0)]:
        g.set_tile(*tile)
        g.step_timed(3)
        ms[tile] = g.step_timed(20)[0]
    base = ms[1, 8, 24]
    assert ms[1, 0, 0] > 3 * base, ms
    g.close()


# runs by the lattice's size of 1, 2, 4 and 8 planes (binary16 quads), 1 and 2 (FP32, odd rows); 61 and 81 planes
# leave a last run that is not whole
@pytest.mark.parametrize("dims,storage,kw", [
    ((512, 64, 61), "fp16s", dict()), ((512, 64, 61), "fp16sr", dict(collision="bgk")),
    ((512, 96, 81), "fp16sr", dict()), ((512, 96, 81), "fp16s", dict(collision="bgk", streaming="aa")),
    ((1024, 96, 81), "fp16s", dict()), ((1024, 96, 81), "fp16sr", dict(streaming="aa")),
    ((1024, 96, 81), "fp16sr", dict(bc_x="periodic", force=(2e-6, 0.0, 1e-6))),
    ((512, 64, 61), "fp32", dict()), ((387, 65, 61), "fp32", dict(collision="bgk")), ((387, 65, 61), "fp16sr", dict())])
def test_runs_bit_identical(dims, storage, kw):
    from paper_2205_02774_gb300.channel import Channel
    nx, ny, nz = dims
    c = SMALL.with_(nx=nx, ny=ny, nz=nz, storage=storage, stats_every=4, **kw)
    f = perturbed_equilibrium_field(nx, ny, 3, seed=nx)  # three planes, repeated along z
    ref = None
    for tile in [(1, 8, 24), (1, 4, 4), (1, 5, 0), (1, 12, 24), (0, 0, 8), (1, 16, 7)]:
        g = Channel.from_case(c, check_every=3, mass_tol=0.5)
        g.set_tile(*tile)
        g.set_state(np.tile(g.encode(f), (1, nz // 3 + 1, 1, 1))[:, :nz], 0)
        g.step(5)
        st = g.stats()
        assert st["rc"] == 0, st["error"]
        got = (g.get_state(), st["mean_sum"], st["rey_sum"])
        g.close()
        if ref is None:
            ref = got
        for a, b in zip(got, ref):
            assert np.array_equal(a, b), tile


def test_autotune_where_the_candidates_differ():
    from paper_2205_02774_gb300.channel import Channel
    c = SMALL.with_(nx=512, ny=64, nz=61, storage="fp16s", stats_every=5)
    a = Channel.from_case(c, check_every=4, mass_tol=0.5)
    b = Channel.from_case(c, check_every=4, mass_tol=0.5)
    a.step(9)
    b.step(9)
    assert b.autotune(3) == b.tile()
    a.step(13)
    b.step(13)
    assert np.array_equal(a.get_state(), b.get_state())
    assert np.array_equal(a.stats()["mean_sum"], b.stats()["mean_sum"])
    a.close()
    b.close()
