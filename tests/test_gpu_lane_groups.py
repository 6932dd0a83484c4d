"""Lane groups per domain (the thread plans' kernel for moderate numbers of
domains): every number of lanes per domain and sets per warp that the library
picks, against the warp kernel decision for decision.  The sizes walk the
plan's rule: few domains take 32 (L_d = 16: 16) lanes, more of them 16 or 8,
visits of k >= 8 steps two sets per warp; a replica with an odd number of
domains per colour leaves sets partly empty, and k > 16 fills chunks of 32
steps and goes past them."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

GRID, THREADS = 2, 3


@pytest.fixture(autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _run(L, Ld, ks, plan, n, time_mode, schedule, per_pass, interleave_init):
    import paper_1403_4674_gb300 as kmc
    m = len(L)
    lat = kmc.Lattice(L, Ld, 1, list(range(71, 71 + m)))
    lat.set_replica_params(k=ks, init=[i % 2 if interleave_init else 0 for i in range(m)])
    lat.reset(kmc.KMC_INIT_PER_REPLICA)
    if plan is not None:
        lat.set_launch(*plan)
    lat.set_rates([0.30 + 0.05 * (i % 5) for i in range(m)], [0.02 * (i % 3) for i in range(m)])
    if per_pass:
        lat.set_observation(kmc.KMC_OBS_PASS)
    obs = [lat.run(c, schedule=schedule, time_mode=time_mode, obs_every=2).cpu().numpy() for c in n]
    lat.sync()
    out = (lat.spins.cpu().numpy(), *lat.domain_state(), np.concatenate(obs), lat.launch())
    lat.close()
    return out


@pytest.mark.parametrize("L,Ld,ks", [
    ([32, 96, 64], 16, [3, 1, 2]),              # 16 lanes, one set per warp; 1, 9 and 4 domains per colour
    ([32, 96, 64], 16, [16, 9, 40]),            # 16 lanes, two sets per warp
    ([512, 480], 16, [4, 3]),                   # 8 lanes, one set per warp
    ([512, 480], 16, [16, 20]),                 # 8 lanes, two sets per warp
    ([64, 192], 32, [1, 4]),                    # 32 lanes, one set
    ([64, 192, 128], 32, [33, 8, 70]),          # 32 lanes, two sets, past two chunks
    ([1024, 704], 32, [2, 1]),                  # 16 lanes, one set
    ([2048], 32, [2]),                          # 8 lanes, one set
    ([2048], 32, [9]),                          # 8 lanes, two sets
    ([128, 384], 64, [5, 2]),                   # 32 lanes, one set
    ([128, 384], 64, [20, 33]),                 # 32 lanes, two sets
    ([2048, 1152], 64, [3, 2]),                 # 16 lanes, one set
    ([3072], 64, [8]),                          # 16 lanes, two sets
])
@pytest.mark.parametrize("mode", ["plain", "fixed_expected", "per_pass"])
def test_lane_groups_equal_the_warp_kernel(L, Ld, ks, mode):
    args = dict(time_mode=1 if mode == "fixed_expected" else 0, schedule=1 if mode == "fixed_expected" else 0,
                per_pass=mode == "per_pass", interleave_init=True)
    n = [2, 3]
    want = _run(L, Ld, ks, (GRID, 152, 8), n, **args)
    for plan in (None, (THREADS, 2, 4), (THREADS, 1, 3)):
        got = _run(L, Ld, ks, plan, n, **args)
        assert got[-1][0] == THREADS and want[-1][0] == GRID
        assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1]) and np.array_equal(got[2], want[2])
        np.testing.assert_allclose(got[3], want[3], rtol=1e-12, atol=0)
        assert np.array_equal(got[4][..., :3], want[4][..., :3])
        np.testing.assert_allclose(got[4][..., 3], want[4][..., 3], rtol=1e-12, atol=0)


@pytest.mark.parametrize("L,Ld,ks", [
    ([32, 96, 64], 16, [3, 1, 40]),   # 16 lanes
    ([256, 192, 256], 16, [9, 8, 16]),  # two sets per warp, of different replicas
    ([64, 192], 32, [4, 9]),          # 32 lanes
    ([2048], 32, [9]),                # 8 lanes
    ([128, 256], 64, [5, 20]),        # 32 lanes, 64 columns
])
@pytest.mark.parametrize("per_pass,time_mode", [(False, 0), (True, 1)])
def test_random_orders_equal_the_warp_kernel(L, Ld, ks, per_pass, time_mode):
    """Each replica's own order of the colours, run after run, on the grid of
    lane groups that a random-order run takes by itself."""
    args = dict(time_mode=time_mode, schedule=2, per_pass=per_pass, interleave_init=True)
    n = [4, 3]
    want = _run(L, Ld, ks, (GRID, 152, 8), n, **args)
    got = _run(L, Ld, ks, None, n, **args)
    assert got[-1][0] == GRID
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1]) and np.array_equal(got[2], want[2])
    np.testing.assert_allclose(got[3], want[3], rtol=1e-12, atol=0)
    assert np.array_equal(got[4][..., :3], want[4][..., :3])
    np.testing.assert_allclose(got[4][..., 3], want[4][..., 3], rtol=1e-12, atol=0)


def test_fixed_time_and_scores_after_a_random_order():
    """A fixed-time run (also captured in a graph) and scores after a
    random-order run leave the lane groups for a kernel that has them."""
    import torch
    import paper_1403_4674_gb300 as kmc
    out = []
    for plan in (None, (GRID, 152, 8)):
        lat = kmc.Lattice([64, 96], 16, 8, [5, 6])
        if plan:
            lat.set_launch(*plan)
        lat.set_rates([0.4, 0.3], [0.01, 0.0])
        lat.run(2, schedule=kmc.KMC_SCHEDULE_RANDOM_PERM)
        lat.set_horizon(0.02)
        g = torch.cuda.CUDAGraph()
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            with torch.cuda.graph(g, stream=side):
                lat.run(2, time_mode=kmc.KMC_TIME_HORIZON)
        torch.cuda.current_stream().wait_stream(side)
        g.replay()
        torch.cuda.synchronize()
        lat.run(2, schedule=kmc.KMC_SCHEDULE_RANDOM_PERM)
        lat.enable_grad(True)
        lat.run(2)
        lat.sync()
        out.append((lat.spins.cpu().numpy(), *lat.domain_state()[:2]))
        lat.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("Ld,ks", [(32, [2, 8, 5]), (32, [16, 9, 1]), (16, [17, 3, 16]), (32, [16, 33, 40]), (16, [8, 16, 12])])
@pytest.mark.parametrize("per_pass", [False, True])
def test_scores_after_the_visit_equal_the_warp_kernels(Ld, ks, per_pass):
    """Scores worked off after a visit's edges (k <= 16: lists of 16 steps, a
    null run going on past a list's end unless at a multiple of 32 steps) or
    event by event (longer visits): the same terms in the same order as the
    warp kernel's, hence the same numbers."""
    import paper_1403_4674_gb300 as kmc
    L, out = [4 * Ld, 8 * Ld, 2 * Ld], []
    for plan in ((THREADS, 0, 4), (GRID, 152, 8)):
        lat = kmc.Lattice(L, Ld, 1, [41, 42, 43])
        lat.set_replica_params(k=ks)
        lat.set_launch(*plan)
        lat.enable_grad(True)
        lat.set_rates([0.42, 0.35, 0.5], [0.02, 0.01, -0.02])
        if per_pass:
            lat.set_observation(kmc.KMC_OBS_PASS)
        obs = np.concatenate([lat.run(n, obs_every=3).cpu().numpy() for n in (7, 8)])
        assert lat.launch()[0] == plan[0]
        out.append((lat.spins.cpu().numpy(), lat.score().cpu().numpy(), obs))
        lat.close()
    (s0, g0, o0), (s1, g1, o1) = out
    assert np.array_equal(s0, s1) and np.array_equal(g0, g1)
    assert np.array_equal(o0[..., :3], o1[..., :3])
    np.testing.assert_allclose(o0[..., 4:6], o1[..., 4:6], rtol=1e-12, atol=1e-12)
