"""Device memory that a lattice needs beside its populations (CPU: the admission
estimate, which create() never exceeds)."""
import pytest


@pytest.fixture(scope="module")
def capi():
    from paper_2205_02774_gb300 import build
    build()
    from paper_2205_02774_gb300 import capi
    return capi


def _domain(capi, nx, ny, nz, storage, streaming=0):
    d = capi.stg_domain()
    d.nx, d.ny, d.nz, d.storage, d.streaming = nx, ny, nz, storage, streaming
    d.bc_x, d.tau0, d.c_smag = capi.STG_BC_X_PERIODIC, 0.6, 0.01
    return d


# narrow boxes and the largest lattices that there are (2^31 - 1 cells)
@pytest.mark.parametrize("dims,storage", [((1, 1, 2 ** 31 - 1), 1), ((1, 65535, 32767), 1), ((31, 1, 69273666), 2),
                                          ((1290, 1290, 1290), 1), ((1290, 1290, 1290), 2), ((640, 640, 640), 0)])
def test_a_periodic_box_needs_little_more_than_its_lattices(capi, dims, storage):
    """Populations, the filter state and one velocity plane at most per (y, z) node and
    the (x, y) statistics sums; block sums of the mass below 1 % of the populations."""
    nx, ny, nz = dims
    est = capi.stg_lbm_estimate_bytes(_domain(capi, nx, ny, nz, storage), None)
    pops = 2 * 19 * nx * ny * nz * (4 if storage == 0 else 2)
    assert pops < est <= 1.01 * pops + 24 * ny * nz + 72 * nx * ny + 1e6
