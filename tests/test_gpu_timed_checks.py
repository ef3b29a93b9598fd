"""Mass checks that run inside timed steps (GPU, through the C ABI).

stg_lbm_step_timed advances the same state by the same passes as stg_lbm_step,
its check steps among them: what such a check finds is reported like one of an
ordinary call, by the next step or statistics call."""
import numpy as np
import pytest

from workloads import case, perturbed_equilibrium_field

from gpu_helpers import require_cuda

pytestmark = pytest.mark.gpu

SMALL = case("channel_64x32x32").with_(nx=16, ny=6, nz=5, stats_every=0, n_modes=8)


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    require_cuda()


def test_drift_in_a_timed_call_reaches_stats():
    from paper_2205_02774_gb300.capi import STG_ERR_UNSTABLE
    from paper_2205_02774_gb300.channel import Channel
    ch = Channel.from_case(SMALL, check_every=10, mass_tol=1e-12)  # an open channel drifts by far more
    ch.step_timed(15)
    st = ch.stats()
    assert st["rc"] == STG_ERR_UNSTABLE and "drift" in st["error"]
    ch.close()


def test_nan_in_a_timed_call_stops_the_next_step():
    from paper_2205_02774_gb300.capi import StgError, STG_ERR_UNSTABLE
    from paper_2205_02774_gb300.channel import Channel
    ch = Channel.from_case(SMALL, check_every=5, mass_tol=0.5)
    bad = ch.encode(perturbed_equilibrium_field(ch.nx, ch.ny, ch.nz, seed=1))
    bad[3, 1, 2, 3] = np.nan
    ch.set_state(bad, 0)
    ch.step(3)  # no check step yet
    ch.step_timed(4)
    with pytest.raises(StgError) as e:
        ch.step(1)
    assert e.value.code == STG_ERR_UNSTABLE
    ch.close()


def test_a_check_is_read_once_and_a_reset_forgets_it():
    from paper_2205_02774_gb300.channel import Channel
    ch = Channel.from_case(SMALL, check_every=4, mass_tol=0.5)
    for n in (3, 1, 9, 2):
        ch.step_timed(n)
        ch.step(n)
    assert ch.stats()["rc"] == 0
    good = ch.get_state()
    ch.set_state(good, 2)
    ch.step_timed(1)
    ch.step(1)
    assert ch.stats()["rc"] == 0 and ch.stats()["step"] == 4
    ch.close()
