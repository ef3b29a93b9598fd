"""Rows of odd length on lattices that fill the GPU (GPU, C ABI).

Lanes 32 cells apart with the inner rows and the wall rows in launches of their
own: FP32 with two cells per lane (from 622 592 cells on), binary16 with four,
runs of 1 and 2 planes with a ragged last one, the outlet node first of its 32
cells (nx = 1 mod 32) or beside its neighbour, walls and periodic rows, a
sampling step (the lanes' sums lie 32 cells apart as their cells do) and the
mass check of all blocks."""
import numpy as np
import pytest

from workloads import case, perturbed_equilibrium_field

from gpu_helpers import require_cuda, pair, max_rel, normwise, fp16_bits, fp16_decode, fp16_half_ulp, W19

pytestmark = pytest.mark.gpu

SMALL = case("channel_64x32x32").with_(stats_every=2, n_modes=20)


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    require_cuda()


# (runs of 2 planes from 24 320 items of 64 cells (FP32) and 15 200 of 128 (binary16) on)
@pytest.mark.parametrize("dims", [(385, 65, 26), (383, 65, 59), (129, 65, 75)])
@pytest.mark.parametrize("storage", ["fp32", "fp16s", "fp16sr"])
@pytest.mark.parametrize("kw", [dict(), dict(collision="bgk", sponge_len=12.0),
                                dict(bc_x="periodic", force=(2e-5, -1e-5, 3e-5)),
                                dict(bc_x="periodic", bc_y="periodic", collision="bgk", force=(0.0, 1e-5, 0.0))],
                         ids=["channel", "bgk_sponge", "force", "box_bgk"])
def test_step_and_statistics(dims, storage, kw):
    nx, ny, nz = dims
    c = SMALL.with_(nx=nx, ny=ny, nz=nz, storage=storage, **kw)
    gpu, orc = pair(c, check_every=1, mass_tol=0.5)
    f = perturbed_equilibrium_field(nx, ny, nz, seed=nx)
    st = gpu.encode(f) if storage == "fp32" else fp16_bits(f)
    gpu.set_state(st, 0)
    orc.set_pops(gpu.decode(st) if storage == "fp32" else fp16_decode(st))
    gpu.step(1)
    orc.step(1)
    fo = orc.pops()
    if storage == "fp32":
        assert max_rel(gpu.populations(), fo) < 1e-5
    else:
        err = np.abs(fp16_decode(gpu.get_state()) - fo)
        spacing = 2 * fp16_half_ulp(fo - W19.reshape(19, 1, 1, 1))
        assert (err - (spacing * (0.5 if storage == "fp16s" else 1.0) + 2e-6 * np.abs(fo))).max() <= 0
    gpu.step(1)
    orc.step(1)
    s = gpu.stats()
    assert s["rc"] == 0, s["error"]
    m, r, n = orc.stats()
    assert s["n_samples"] == n == 1
    tol = 1e-4 if storage == "fp32" else 4e-3
    assert normwise(s["mean_sum"], m) < tol and normwise(s["rey_sum"], r) < tol
    assert abs(s["mass"] - orc.pops().sum()) <= (1e-6 if storage == "fp32" else 1e-4) * nx * ny * nz
    gpu.close()


# rows of fewer than 32 cells change to one cell per thread at 57 760 (stochastic rounding) and
# 72 960 rows x planes
@pytest.mark.parametrize("dims", [(31, 190, 303), (31, 190, 305), (3, 190, 305), (5, 240, 303), (5, 240, 305)])
@pytest.mark.parametrize("storage", ["fp16s", "fp16sr"])
def test_narrow_rows(dims, storage):
    test_step_and_statistics(dims, storage, dict(collision="bgk"))
