"""Kernel choices by size, on the clock (GPU): forms that a rule must not give to a
lattice, shown by what it would cost against another form of the same work on the
same lattice.  The margins are a third and more of the difference between the forms."""
import pytest

from workloads import case

from gpu_helpers import require_cuda

pytestmark = pytest.mark.gpu

SMALL = case("channel_64x32x32").with_(n_modes=20, stats_every=0)


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    require_cuda()


def _us(tile=None, **kw):
    """Device time of a step in microseconds, the best of a few series."""
    import torch
    from paper_2205_02774_gb300.channel import Channel
    g = Channel.from_case(SMALL.with_(**kw))
    if tile:
        g.set_tile(*tile)
    best = 1e9
    g.step(96)
    for _ in range(7):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        with torch.cuda.stream(g.stream):
            a.record()
            g.step(96)
            b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b) / 96 * 1e3)
    g.close()
    return best


# quads on rows that leave a third to a half of their lanes idle: 1.13 and 1.12 times the
# regularized collision's time, pairs 0.93
@pytest.mark.parametrize("n", [140, 160])
def test_bgk_of_binary16_on_ragged_rows(n):
    kw = dict(nx=n, ny=n, nz=n, storage="fp16s")
    assert _us(collision="bgk", **kw) < 1.03 * _us(**kw)


# runs by the number of items alone came to 8 planes where 1 or 2 are the fastest: the same
# time as with a tile of 9, 0.90 to 0.93 of it with runs of 2
@pytest.mark.parametrize("dims", [(250, 125, 125), (770, 128, 192)])
def test_runs_of_binary16_pairs(dims):
    kw = dict(nx=dims[0], ny=dims[1], nz=dims[2], storage="fp16s")
    assert _us(**kw) < 0.97 * _us(tile=(1, 9, 24), **kw)


# four cells per lane of which one is in the row: 1.30 times the time of one cell per thread
def test_narrow_rows_of_binary16(monkeypatch):
    kw = dict(nx=5, ny=300, nz=300, storage="fp16sr")
    own = _us(**kw)
    monkeypatch.setenv("STG_LBM_INTERIOR", "scalar")
    assert own < 1.1 * _us(**kw)


# FP32 BGK, a last chunk of 8 of 64 cells: short runs in blocks of four warps that wait for
# each other took 1.06 times as long as runs of 9, runs of 4 in blocks of one 0.98 (the tile
# sets the run, not the block)
def test_fp32_bgk_on_ragged_rows():
    kw = dict(nx=200, ny=200, nz=200, collision="bgk")
    assert _us(**kw) < 1.02 * _us(tile=(1, 9, 24), **kw)


# a batch of many small channels: a graph branch of every member for its inlet planes made the
# step 1.56 times that of the same boxes without an inlet, planes in line 1.19
def test_inlet_planes_in_a_batch_of_many():
    import torch
    from paper_2205_02774_gb300.channel import Channel
    from paper_2205_02774_gb300.serving import Batch
    us = {}
    for bc_x in ("stg", "periodic"):
        s = torch.cuda.Stream()
        b = Batch(stream=s)
        c = SMALL.with_(nx=144, ny=24, nz=36, storage="fp16s", bc_x=bc_x, n_modes=60)
        chs = [Channel.from_case(c, stream=s) for _ in range(80)]
        for ch in chs:
            b.add(ch)
        for _ in range(6):
            b.step(32)
        best = 1e9
        for _ in range(8):
            t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            with torch.cuda.stream(s):
                t0.record()
                b.step(32)
                t1.record()
            t1.synchronize()
            best = min(best, t0.elapsed_time(t1))
        us[bc_x] = best
        b.close()
        for ch in chs:
            ch.close()
    assert us["stg"] < 1.35 * us["periodic"]


# rows that fill an eighth of a chunk count as what they hold: runs of 8 planes took 1.046
# times as long as runs of 2
def test_runs_of_narrow_binary16_rows():
    kw = dict(nx=16, ny=256, nz=256, storage="fp16sr", streaming="aa")
    assert _us(**kw) < 1.025 * _us(tile=(0, 16, 24), **kw)


# FP32 pairs on a few hundred thousand to two million cells: wall rows in runs of 4 planes
# outlasted the inner rows (1.20 times the time of runs of 1 or 2)
def test_wall_rows_of_small_fp32_lattices():
    kw = dict(nx=300, ny=50, nz=75)
    assert _us(**kw) < 0.93 * _us(tile=(1, 8, 32), **kw)


# binary16 pairs had FP32's line for one launch of all rows: 206x34x51 took longer than the
# same channel with 72 planes, which had two launches (1.05 times, 0.86 with two of its own)
def test_two_launches_of_binary16_pairs():
    kw = dict(nx=206, ny=34, storage="fp16s")
    assert _us(nz=51, **kw) < 0.97 * _us(nz=72, **kw)


# in place, periodic x: stores through shuffles beside the loads' own took 1.06 times as long
# (1.10 times the time of the channel, 1.03 without)
def test_in_place_stores_of_periodic_rows():
    kw = dict(nx=1536, ny=128, nz=192, storage="fp16sr", streaming="aa")
    assert _us(bc_x="periodic", **kw) < 1.065 * _us(**kw)


# in place, runs of 8 planes (1.05 times the time of runs of 4, runs of 9 no better than 8)
def test_runs_in_place():
    kw = dict(nx=512, ny=128, nz=128, storage="fp16s", streaming="aa")
    assert _us(**kw) < 0.985 * _us(tile=(1, 9, 24), **kw)
