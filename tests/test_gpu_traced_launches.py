"""Kernels that a call enqueues, as bench.py counts them (GPU): its count follows the
library's own rules (blocks, lane layouts, one launch per pass or two), so it is held
against the kernels that the device has run."""
import pytest

from workloads import case

from gpu_helpers import require_cuda

pytestmark = pytest.mark.gpu

SMALL = case("channel_64x32x32").with_(n_modes=8, stats_every=10)


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    require_cuda()
    import torch
    for _ in range(2):  # (the first trace of a process misses graph launches)
        names = _kernels(lambda: torch.zeros(8, device="cuda").add_(1))[1]
    if not names:
        pytest.skip("another profiler holds the tracing interface")


def _kernels(call):
    import torch
    from torch.profiler import profile, ProfilerActivity
    with profile(activities=[ProfilerActivity.CUDA]) as p:
        call()
        torch.cuda.synchronize()
    names = [e.name for e in p.events() if e.device_type == torch.autograd.DeviceType.CUDA]
    return sum("kernel" in n and "Memcpy" not in n and "Memset" not in n for n in names), names


# one launch and two by storage, lanes and collision, single steps before and after the blocks
@pytest.mark.parametrize("dims,kw", [
    ((64, 32, 32), dict()), ((128, 64, 38), dict()), ((128, 64, 76), dict()), ((385, 65, 26), dict()),
    ((240, 40, 60), dict(storage="fp16sr")), ((256, 48, 37), dict(storage="fp16s")),
    ((256, 48, 41), dict(storage="fp16s")), ((256, 48, 41), dict(storage="fp16s", collision="bgk")),
    ((256, 48, 41), dict(storage="fp16sr", collision="bgk", bc_x="periodic")),
    ((768, 48, 16), dict(storage="fp16sr", collision="bgk")), ((3, 190, 305), dict(storage="fp16sr")),
    ((256, 48, 41), dict(storage="fp16s", streaming="aa")), ((128, 64, 38), dict(streaming="aa")),
    ((64, 32, 32), dict(stats_every=0)), ((64, 2, 40), dict(stats_every=7))])
def test_of_a_channel(dims, kw):
    import bench
    from paper_2205_02774_gb300.channel import Channel
    c = SMALL.with_(nx=dims[0], ny=dims[1], nz=dims[2], **kw)
    g = Channel.from_case(c)
    g.step(3)
    for t0, n in ((3, 47), (50, 50), (100, 1)):
        got, names = _kernels(lambda: g.step(n))
        assert got == bench._launches_enqueued(c, t0, n), names
    g.close()


@pytest.mark.parametrize("n", [3, 20, 47])
def test_of_probed_steps(n):
    import bench
    from paper_2205_02774_gb300.channel import Channel
    g = Channel.from_case(SMALL)
    g.set_probes([[1, 2, 3], [4, 5, 6]])
    g.step_probed(n)
    got, names = _kernels(lambda: g.step_probed(n))
    assert got == bench._launches_enqueued(SMALL, n, n, probed=True), names
    g.close()


def test_of_a_batch():
    import bench
    from paper_2205_02774_gb300.channel import Channel
    from paper_2205_02774_gb300.serving import Batch
    c = SMALL.with_(nx=96, ny=32, nz=32)
    b = Batch()
    chs = [Channel.from_case(c) for _ in range(8)]
    for ch in chs:
        b.add(ch)
    b.step(20)
    got, names = _kernels(lambda: (b.step(40), b.sync()))
    assert got == 8 * bench._launches_enqueued(c, 20, 40, batch=True), names
    b.close()
    for ch in chs:
        ch.close()
