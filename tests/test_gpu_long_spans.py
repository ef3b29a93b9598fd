"""Lattices of very many span nodes (GPU, through the C ABI): the launches take every
nz that the lattice's sizes allow, more blocks along z than a grid's 65 535 rows."""
import numpy as np
import pytest

from workloads import case, perturbed_equilibrium_field

from gpu_helpers import require_cuda, pair, max_rel, normwise

pytestmark = pytest.mark.gpu

SMALL = case("channel_64x32x32")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    require_cuda()


# planes by 4, 16 and 5 steps per launch (a block of 25 steps): 2, 2 and 1 span nodes per block
@pytest.mark.parametrize("nz", [65537, 131075])
def test_inlet_planes(nz):
    c = SMALL.with_(nx=3, ny=4, nz=nz, n_modes=5, stats_every=25, t_filter=4.0)
    gpu, orc = pair(c)
    gpu.step(26)
    orc.step(26)
    u, u_or = gpu.inlet(), orc.inlet()
    assert np.abs(u - u_or).max() <= 1e-5 * np.abs(u_or).max()
    gpu.close()


@pytest.mark.parametrize("nx", [1, 4])
def test_sampling_runs(nx):
    nz = 65535 * 32 + 3
    c = SMALL.with_(nx=nx, ny=1, nz=nz, bc_x="periodic", bc_y="periodic", stats_every=1)
    gpu, orc = pair(c)
    st = gpu.encode(perturbed_equilibrium_field(nx, 1, nz, seed=nx))
    gpu.set_state(st, 0)
    orc.set_pops(gpu.decode(st))
    gpu.step(1)
    orc.step(1)
    assert max_rel(gpu.populations(), orc.pops()) < 1e-5
    s = gpu.stats()
    m, r, n = orc.stats()
    assert s["n_samples"] == n == 1
    assert normwise(s["mean_sum"], m) < 1e-4 and normwise(s["rey_sum"], r) < 1e-4
    gpu.close()
