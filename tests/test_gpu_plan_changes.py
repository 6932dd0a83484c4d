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
