"""Rows of any length (GPU, C ABI): lanes 32 cells apart.

Lattices with odd nx (every storage) and small FP32 ones take the loop whose
lanes own cells 32 apart.  One step from an identical state and a sampling step
after it must match the oracle for every remainder of the row: chunks of 32, 64
and 128 cells, the outlet node first of its 32 (nx = 1 mod 32) or beside its
neighbour, single cells, walls and periodic rows."""
import numpy as np
import pytest

from workloads import case, perturbed_equilibrium_field

from gpu_helpers import require_cuda, pair, max_rel, normwise, fp16_bits, fp16_decode, fp16_half_ulp, W19

pytestmark = pytest.mark.gpu

SMALL = case("channel_64x32x32").with_(stats_every=2, n_modes=20)


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    require_cuda()


@pytest.mark.parametrize("nx", [1, 2, 3, 5, 31, 32, 33, 64, 65, 97, 127, 129, 161, 257])
@pytest.mark.parametrize("storage", ["fp32", "fp16s", "fp16sr"])
@pytest.mark.parametrize("kw", [dict(), dict(collision="bgk", sponge_len=2.0),
                                dict(bc_x="periodic", force=(2e-5, -1e-5, 3e-5)),
                                dict(bc_x="periodic", bc_y="periodic", collision="bgk", force=(0.0, 1e-5, 0.0))],
                         ids=["channel", "bgk_sponge", "force", "box_bgk"])
def test_step_and_statistics(nx, storage, kw):
    if "bc_x" not in kw and nx < 3:
        pytest.skip("an inlet/outlet lattice has nx >= 3")
    if kw.get("sponge_len", 0.0) > nx - 1:
        pytest.skip("the sponge does not fit")
    c = SMALL.with_(nx=nx, ny=5, nz=6, storage=storage, **kw)
    gpu, orc = pair(c, check_every=1, mass_tol=0.5)
    f = perturbed_equilibrium_field(nx, 5, 6, seed=nx)
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
    gpu.close()
