"""Passes of inner rows and wall rows apart (GPU, C ABI).

One step from an identical state and a sampling step after it, against the
oracle, on lattices just large enough for two launches (and just too small):
binary16 BGK and forced quads (their inner-row kernels have register budgets of
their own) and pairs (nx = 2 mod 4), FP32 with one cell per lane and with pairs;
and the one-cell-per-thread kernels of lattices beyond 32-bit offsets, which the
environment override brings to small ones."""
import numpy as np
import pytest

from workloads import case, perturbed_equilibrium_field

from gpu_helpers import require_cuda, pair, max_rel, normwise, fp16_bits, fp16_decode, fp16_half_ulp, W19

pytestmark = pytest.mark.gpu

SMALL = case("channel_64x32x32").with_(stats_every=2, n_modes=20)
FORCE = dict(bc_x="periodic", force=(2e-5, -1e-5, 3e-5))


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    require_cuda()


def _step_and_sample(c, **kw):
    nx, ny, nz, storage = c.nx, c.ny, c.nz, c.storage
    gpu, orc = pair(c, check_every=1, mass_tol=0.5, **kw)
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


# quads: two launches from 3648 items of 128 cells on, runs of 2 planes from 15 200 on; pairs: 9728 items of 64
@pytest.mark.parametrize("dims", [(256, 48, 37), (256, 48, 41), (516, 64, 53), (130, 64, 51)])
@pytest.mark.parametrize("kw", [dict(collision="bgk"), dict(collision="bgk", **FORCE), dict(**FORCE),
                                dict(collision="bgk", sponge_len=6.4)], ids=["bgk", "bgk_force", "force", "bgk_sponge"])
@pytest.mark.parametrize("storage,streaming", [("fp16s", "pull"), ("fp16sr", "pull"), ("fp16s", "aa")])
def test_binary16(dims, kw, storage, streaming):
    nx, ny, nz = dims
    _step_and_sample(SMALL.with_(nx=nx, ny=ny, nz=nz, storage=storage, streaming=streaming, **kw), streaming=streaming)


# one cell per lane: two launches from 9728 items of 32 cells on; pairs from 622 592 cells on
@pytest.mark.parametrize("dims", [(128, 64, 37), (128, 64, 38), (128, 64, 75), (128, 64, 76), (128, 63, 38)])
@pytest.mark.parametrize("kw", [dict(), dict(collision="bgk", **FORCE), dict(sponge_len=6.4)],
                         ids=["channel", "bgk_force", "sponge"])
def test_fp32(dims, kw):
    nx, ny, nz = dims
    _step_and_sample(SMALL.with_(nx=nx, ny=ny, nz=nz, **kw))


@pytest.mark.parametrize("dims", [(101, 5, 7), (97, 9, 8), (128, 6, 5), (3, 2, 9), (40, 1, 6)])
@pytest.mark.parametrize("storage", ["fp32", "fp16s", "fp16sr"])
@pytest.mark.parametrize("kw", [dict(), dict(collision="bgk", **FORCE), dict(sponge_len=2.0)],
                         ids=["channel", "bgk_force", "sponge"])
def test_one_cell_per_thread(dims, storage, kw, monkeypatch):
    monkeypatch.setenv("STG_LBM_INTERIOR", "scalar")
    nx, ny, nz = dims
    _step_and_sample(SMALL.with_(nx=nx, ny=ny, nz=nz, storage=storage, **kw))
