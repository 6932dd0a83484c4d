"""Launch plans that change under a context: scores on and off, random orders,
work still queued on a side stream, graphs captured with an earlier plan."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
GRID, THREADS = 2, 3
WARP = (GRID, 152, 8)


@pytest.fixture(autouse=True, scope="module")
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _state(lat):
    lat.sync()
    out = (lat.spins.cpu().numpy(), *lat.domain_state())
    lat.close()
    return out


def _same(a, b):
    for x, y in zip(a[:3], b[:3]):
        assert np.array_equal(x, y)
    np.testing.assert_allclose(a[3], b[3], rtol=1e-12, atol=0)


def _captured(side, lat, n, **kw):
    import torch
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(side):
        with torch.cuda.graph(g, stream=side):
            lat.run(n, **kw)
    return g


OFF_AGAIN = """
import sys
import numpy as np
sys.path.insert(0, %r)
import paper_1403_4674_gb300 as kmc
Ld, plan = int(sys.argv[1]), [int(x) for x in sys.argv[2:]]
out = []
for p in (plan, (2, 152, 8)):
    lat = kmc.Lattice([8 * Ld, 4 * Ld], Ld, 8, [3, 4])
    if p:
        lat.set_launch(*p)
    lat.set_rates([0.42, 0.3], [0.01, 0.0])
    for on in (True, False, True, False):
        lat.enable_grad(on)
        lat.run(3)
        lat.run(2, time_mode=kmc.KMC_TIME_EXPECTED)
    lat.sync()
    out.append((lat.spins.cpu().numpy(), *lat.domain_state()[:2], lat.score().cpu().numpy()))
    lat.close()
assert all(np.array_equal(a, b) for a, b in zip(*out))
"""


@pytest.mark.parametrize("args", [(32,), (16,), (16, THREADS, 0, 2), (16, THREADS, 0, 4), (32, THREADS, 2, 4), (64,)])
def test_scores_turned_off_again(args):
    """In a process of its own: shared-memory limits belong to the process's kernels."""
    res = subprocess.run([sys.executable, "-c", OFF_AGAIN % ROOT, *map(str, args)], capture_output=True, text=True,
                         timeout=300)
    assert res.returncode == 0, res.stderr[-2000:]


def _queued(plan):
    """Runs queued on a non-blocking stream while the plan changes twice."""
    import torch
    import paper_1403_4674_gb300 as kmc
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        lat = kmc.Lattice([256], 32, 8, [11])
        if plan:
            lat.set_launch(*plan)
        lat.set_rates([0.42], [0.01])
        for _ in range(4):
            lat.run(500)
        lat.enable_grad(True)
        for _ in range(4):
            lat.run(500)
        if not plan:
            lat.set_launch(THREADS, 2, 2)
        for _ in range(2):
            lat.run(500)
        lat.enable_grad(False)
        lat.run(100)
        return _state(lat)


def test_plans_change_while_runs_are_queued():
    _same(_queued(None), _queued(WARP))


def _graphs(plan):
    """Graphs captured with a plan that is then replaced."""
    import torch
    import paper_1403_4674_gb300 as kmc
    side = torch.cuda.Stream()
    lat = kmc.Lattice([256], 32, 8, [11])
    if plan:
        lat.set_launch(*plan)
    lat.set_rates([0.42], [0.01])
    torch.cuda.synchronize()
    a = _captured(side, lat, 20)
    lat.enable_grad(True)
    lat.run(5)
    torch.cuda.synchronize()
    b = _captured(side, lat, 7)
    if not plan:
        lat.set_launch(GRID, 76, 4)
    lat.run(3)
    lat.enable_grad(False)
    if not plan:
        lat.set_launch()
    lat.run(3)
    torch.cuda.synchronize()
    fill = [torch.full((1 << 16,), -1, dtype=torch.int32, device="cuda") for _ in range(8)]  # (into freed memory)
    for g in (a, b, a):
        g.replay()
        torch.cuda.synchronize()
    del fill
    return _state(lat)


def test_graphs_outlive_their_plan():
    _same(_graphs(None), _graphs(WARP))


@pytest.mark.parametrize("Ld", [16, 32, 64])
def test_random_orders_with_scores_captured(Ld):
    """After a random-order run every run has its plan at hand, also while capturing."""
    import torch
    import paper_1403_4674_gb300 as kmc
    out, RANDOM = [], kmc.KMC_SCHEDULE_RANDOM_PERM
    for plan in (None, WARP):
        side = torch.cuda.Stream()
        lat = kmc.Lattice([4 * Ld, 2 * Ld], Ld, 4, [3, 4])
        if plan:
            lat.set_launch(*plan)
        lat.set_rates([0.42, 0.3], [0.01, 0.0])
        lat.set_horizon(0.02)
        lat.run(2, schedule=RANDOM)
        lat.enable_grad(True)
        torch.cuda.synchronize()
        graphs = [_captured(side, lat, 3, schedule=RANDOM), _captured(side, lat, 2)]
        lat.enable_grad(False)
        graphs += [_captured(side, lat, 3, schedule=RANDOM), _captured(side, lat, 2, time_mode=kmc.KMC_TIME_HORIZON),
                   _captured(side, lat, 1)]
        for g in graphs:
            g.replay()
            torch.cuda.synchronize()
        lat.run(2, schedule=RANDOM)
        lat.sync()
        out.append((lat.spins.cpu().numpy(), *lat.domain_state()[:2], lat.score().cpu().numpy()))
        lat.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("Ld", [16, 32])
def test_lane_groups_again_after_scores(Ld):
    import paper_1403_4674_gb300 as kmc
    lat = kmc.Lattice([8 * Ld], Ld, 4, [3])
    before = lat.launch()
    lat.enable_grad(True)
    assert lat.launch() != before
    lat.run(1)
    lat.enable_grad(False)
    assert lat.launch() == before
    lat.close()


@pytest.mark.parametrize("Ld", [16, 32])
@pytest.mark.parametrize("ks", [[1, 2], [3, 5], [7, 8], [15, 16], [17, 33], [32, 40]])
@pytest.mark.parametrize("scores", [False, True])
def test_one_thread_per_domain_chunks(Ld, ks, scores):
    """Visits that end inside, at and past a chunk of drawn steps, replicas of
    both lengths in one warp, on the kernel of one thread per domain (a plan
    made while scores are on keeps it when they go off)."""
    import paper_1403_4674_gb300 as kmc
    out = []
    for plan in ((THREADS, 2, 2), WARP):
        lat = kmc.Lattice([4 * Ld, 2 * Ld], Ld, 1, [8, 9])
        lat.set_replica_params(k=ks)
        lat.enable_grad(True)
        lat.set_launch(*plan)
        lat.enable_grad(scores)
        assert lat.launch()[3] == plan[2]
        lat.set_rates([0.25, 0.4], [0.02, -0.01])
        obs = [lat.run(5, obs_every=2), lat.run(4, obs_every=2, schedule=kmc.KMC_SCHEDULE_FIXED,
                                                time_mode=kmc.KMC_TIME_EXPECTED)]
        lat.sync()
        out.append((lat.spins.cpu().numpy(), *lat.domain_state()[:2], lat.score().cpu().numpy(),
                    *[o[..., :3].cpu().numpy() for o in obs]))
        lat.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
