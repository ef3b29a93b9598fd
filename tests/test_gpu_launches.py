"""How a pass is cut into launches (GPU, through the C ABI).

Small lattices take one launch of all rows, larger ones a launch of the inner
rows beside one of the wall rows, with runs of 1 to 8 z planes per warp; on
sampling steps the runs are 1 to 32 planes long.  Each form must match the
oracle like the others, on both sides of the sizes where the rule changes."""
import numpy as np
import pytest

from workloads import case, perturbed_equilibrium_field

from gpu_helpers import require_cuda, pair, max_rel, normwise, fp16_bits, fp16_decode, fp16_half_ulp, W19

pytestmark = pytest.mark.gpu

SMALL = case("channel_64x32x32")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    require_cuda()


# (pairs: one launch below 9728 chunk rows of 64 cells x planes, binary16 quads below
# 3648 of 128; runs of 2 planes from 24320 (FP32) and 15200 (binary16) on)
@pytest.mark.parametrize("dims,storage", [((128, 64, 75), "fp32"), ((128, 64, 76), "fp32"), ((130, 2, 9), "fp32"),
                                          ((256, 40, 45), "fp16s"), ((256, 40, 46), "fp16s"), ((64, 3, 5), "fp16s"),
                                          ((192, 90, 91), "fp32"), ((260, 64, 80), "fp16s")])
@pytest.mark.parametrize("streaming", ["pull", "aa"])
def test_single_step_and_statistics(dims, storage, streaming):
    nx, ny, nz = dims
    c = SMALL.with_(nx=nx, ny=ny, nz=nz, storage=storage, stats_every=2, n_modes=20, streaming=streaming)
    gpu, orc = pair(c, streaming=streaming, check_every=1, mass_tol=0.5)
    f = perturbed_equilibrium_field(nx, ny, nz, seed=nx + nz)
    st = gpu.encode(f) if storage == "fp32" else fp16_bits(f)
    gpu.set_state(st, 0)
    orc.set_pops(gpu.decode(st) if storage == "fp32" else fp16_decode(st))
    gpu.step(1)
    orc.step(1)
    fo = orc.pops()
    if storage == "fp32":
        assert max_rel(gpu.populations(), fo) < 1e-5
    else:
        g = fo - W19.reshape(19, 1, 1, 1)
        err = np.abs(fp16_decode(gpu.get_state()) - fo)
        assert (err - (fp16_half_ulp(g) + 2e-6 * np.abs(fo))).max() <= 0
    gpu.step(1)  # a sampling step
    orc.step(1)
    s = gpu.stats()
    assert s["rc"] == 0, s["error"]
    m, r, n = orc.stats()
    assert s["n_samples"] == n == 1
    tol = 1e-4 if storage == "fp32" else 2e-3
    assert normwise(s["mean_sum"], m) < tol and normwise(s["rey_sum"], r) < tol
    assert abs(s["mass"] - orc.pops().sum()) <= (1e-6 if storage == "fp32" else 1e-4) * nx * ny * nz
    gpu.close()


@pytest.mark.parametrize("dims", [(64, 33, 31), (64, 32, 32), (96, 41, 50), (1000, 40, 60)])
def test_mass_check_of_many_blocks(dims):
    """The check's mass is added in groups of 1024 blocks (1023, 1024, a few and many
    groups here): in a closed box it stays the initial one to 1e-6."""
    from paper_2205_02774_gb300.channel import Channel
    nx, ny, nz = dims
    c = SMALL.with_(nx=nx, ny=ny, nz=nz, bc_x="periodic", stats_every=3)
    g = Channel.from_case(c, check_every=1, mass_tol=1e-6)
    g.set_state(g.encode(perturbed_equilibrium_field(nx, ny, nz, seed=3)), 0)
    for _ in range(4):
        g.step(1)
        st = g.stats()
        assert st["rc"] == 0, st["error"]
    g.close()
