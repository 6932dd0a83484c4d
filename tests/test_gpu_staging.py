"""How a call takes its spins in and gives them back, and how the 8x8 kernel
deals a colour's domains to its threads: a spin buffer that is 8- but not
16-byte aligned, and grids whose threads visit one, a few or many domains per
phase, give the results of the aligned buffer and of the warp kernel, every
spin, hash and record bit for bit (clocks to 1e-12 relative)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True, scope="module")
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _run(L, Ld, shift=0, plan=None, init=None, ks=None, schedule=0, time_mode=0):
    import torch
    import paper_1403_4674_gb300 as kmc
    n = sum(x * x for x in L)
    buf = torch.full((n + 16,), 1, dtype=torch.int8, device="cuda")
    at = (-buf.data_ptr()) % 16 + shift
    sp = buf[at:at + n]
    lat = kmc.Lattice(L, Ld, 3, list(range(5, 5 + len(L))), spins=sp)
    if init is not None:
        sp.copy_(init)
        lat.reset(kmc.KMC_INIT_KEEP)
    if ks is not None:
        lat.set_replica_params(k=ks)
        lat.reset(0)
    start = sp.cpu().numpy()
    if plan is not None:
        lat.set_launch(*plan)
    lat.set_rates([0.35 + 0.1 * i for i in range(len(L))], [0.05] * len(L))
    obs = lat.run(6, schedule=schedule, time_mode=time_mode, obs_every=2).cpu().numpy()
    lat.sync()
    out = (start, sp.cpu().numpy(), *lat.domain_state(), obs, buf.cpu().numpy(), at, n)
    lat.close()
    return out


def _same(a, b):
    for x, y in zip(a[:4], b[:4]):
        assert np.array_equal(x, y)
    np.testing.assert_allclose(a[4], b[4], rtol=1e-12, atol=0)
    assert np.array_equal(a[5][..., :3], b[5][..., :3])
    np.testing.assert_allclose(a[5][..., 3], b[5][..., 3], rtol=1e-12, atol=0)


@pytest.mark.parametrize("L,Ld", [([16, 48], 8), ([32, 96], 16), ([64, 192], 32), ([128], 64)])
@pytest.mark.parametrize("keep", [False, True])
def test_spin_buffer_on_an_8_byte_boundary(L, Ld, keep):
    import torch
    init = None
    if keep:
        n = sum(x * x for x in L)
        init = torch.from_numpy(np.where(np.random.default_rng(1).random(n) < 0.5, 1, -1).astype(np.int8)).cuda()
    a, b = _run(L, Ld, 0, init=init), _run(L, Ld, 8, init=init)
    _same(a, b)
    for r in (a, b):  # nothing beside the buffer's own bytes is written
        assert (r[6][:r[7]] == 1).all() and (r[6][r[7] + r[8]:] == 1).all()


@pytest.mark.parametrize("ctas", [1, 2, 3, 8])
def test_rounds_of_the_8x8_kernel(ctas):
    """64 + 100 domains per colour on grids of 32 to 256 threads: one round to six."""
    L = [128, 160]
    _same(_run(L, 8, plan=(3, ctas, 1)), _run(L, 8, plan=(2, 8, 8)))


@pytest.mark.parametrize("ks", [[1, 2], [3, 4], [15, 16], [17, 5], [32, 33], [1, 40]])
@pytest.mark.parametrize("schedule,time_mode", [(0, 0), (1, 1)])
def test_chunks_of_the_8x8_kernel(ks, schedule, time_mode):
    """Visits that end inside, at and past a chunk of 32 drawn steps, replicas
    of both lengths side by side in one warp."""
    L = [48, 32]
    a = _run(L, 8, plan=(3, 1, 2), ks=ks, schedule=schedule, time_mode=time_mode)
    _same(a, _run(L, 8, plan=(2, 4, 8), ks=ks, schedule=schedule, time_mode=time_mode))
