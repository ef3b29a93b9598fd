"""Binary16 collisions in packed FP32, two and four cells per lane (GPU, C ABI).

Plain BGK and body-forced lattices of binary16 storage go through the packed
collision like the regularized one: a step from an identical state lies within
half a binary16 spacing of the oracle (one spacing with stochastic rounding)
plus the FP32 part, on rows of pairs (nx = 2 mod 4) and of quads, ragged or
whole chunks, with and without inlet and outlet nodes, pull and in place."""
import numpy as np
import pytest

from workloads import case, perturbed_equilibrium_field

from gpu_helpers import require_cuda, pair, fp16_bits, fp16_decode, fp16_half_ulp, W19

pytestmark = pytest.mark.gpu

SMALL = case("channel_64x32x32").with_(stats_every=0, n_modes=20)
FORCE = dict(bc_x="periodic", force=(2e-5, -1e-5, 3e-5))


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    require_cuda()


@pytest.mark.parametrize("nx", [8, 128, 130, 132, 260])
@pytest.mark.parametrize("kw", [dict(collision="bgk"), dict(collision="bgk", **FORCE), dict(**FORCE),
                                dict(collision="bgk", sponge_len=6.4)], ids=["bgk", "bgk_force", "force", "bgk_sponge"])
@pytest.mark.parametrize("storage,streaming", [("fp16s", "pull"), ("fp16sr", "pull"), ("fp16s", "aa")])
def test_two_steps(nx, kw, storage, streaming):
    c = SMALL.with_(nx=nx, ny=6, nz=7, storage=storage, streaming=streaming, **kw)
    gpu, orc = pair(c, streaming=streaming)
    bits = fp16_bits(perturbed_equilibrium_field(nx, 6, 7, seed=nx))
    W = W19.reshape(19, 1, 1, 1)
    for t in range(2):  # in place: a shifted and a local step
        gpu.set_state(bits, t)
        orc.set_pops(fp16_decode(bits))
        gpu.step(1)
        orc.step(1)
        fo = orc.pops()
        if c.bc_x == "stg" and t:  # the oracle's inlet goes on from its first step, set_state restarts the filter
            break
        spacing = 2 * fp16_half_ulp(fo - W)
        err = np.abs(fp16_decode(gpu.get_state()) - fo)
        assert (err - (spacing * (0.5 if storage == "fp16s" else 1.0) + 2e-6 * np.abs(fo))).max() <= 0, t
    gpu.close()
