"""Exponential clocks of one long call without records in between: 1.57e9
steps of a domain (lane groups) and of a trajectory (partitions), whose
product of clock variates has a binary exponent below -2^31.

The clock is a sum of N = 1.57e9 independent waiting times of mean and
standard deviation 1 / Lambda, so it is N / Lambda to a relative standard
deviation of N^-1/2 = 2.5e-5; the bound is eight of them."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

K, N_SCHED = 65535, 24000  # one visit of K steps per domain and fixed schedule
STEPS = K * N_SCHED
BOUND = 8.0 / STEPS ** 0.5


@pytest.fixture(autouse=True, scope="module")
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def test_lane_groups():
    import paper_1403_4674_gb300 as kmc
    lat = kmc.Lattice([64], 32, K, [3], init=kmc.KMC_INIT_ALL_UP)
    lat.set_rates(3.0)
    rec = lat.run(N_SCHED, schedule=kmc.KMC_SCHEDULE_FIXED, obs_every=N_SCHED)
    lat.sync()
    want = STEPS / (32 * 32)
    np.testing.assert_allclose(lat.domain_state()[2], want, rtol=BOUND, atol=0)
    np.testing.assert_allclose(lat.observables()["t"], want, rtol=BOUND, atol=0)
    np.testing.assert_allclose(rec[0, 0, 3].item(), want, rtol=BOUND, atol=0)
    lat.close()


def test_partitions():
    import paper_1403_4674_gb300 as kmc
    part = kmc.Partitioned(12, kmc.KMC_PART_BLOCKS, 1, K, [5])
    part.set_rates(3.0)
    part.run(N_SCHED, schedule=kmc.KMC_SCHEDULE_FIXED)
    np.testing.assert_allclose(part.state()[3], STEPS / 144.0, rtol=BOUND, atol=0)
    part.close()
