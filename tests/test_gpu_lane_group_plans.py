"""Which lane groups the library picks: lanes per domain, sets per warp and
warps per CTA of the batches whose trajectories test_gpu_lane_groups.py
compares with the warp kernel, told apart by the CTAs and the shared memory
that the plan reports.  A batch that stopped taking the kernel named here
would leave that comparison without it."""
import pytest

pytestmark = pytest.mark.gpu

GRID, THREADS = 2, 3
SM = 152  # the expectations are those of this many SMs


@pytest.fixture(autouse=True, scope="module")
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if torch.cuda.get_device_properties(0).multi_processor_count != SM:
        pytest.skip("expectations for %d SMs" % SM)


def _domain_bytes(Ld, G):
    row = 8 if Ld > 32 else 4
    raw = (16 * G + 80 + 80 + 16 * G + 16 + 16 + 16 + 16 + 16      # counts above, A, 1/A, clocks, totals, meta, halo, columns, ring
           + (Ld + 1) * row + (0 if Ld == 64 else 8 - row)         # rows
           + 64 + 40 + 16 + 32 + 8 + 128)                          # edges, counters, record, neighbours, seed, events
    return ((raw + 15) // 16 | 1) * 16


def _shape(L, Ld, G, ns, wpb):
    """(CTAs, warps per CTA, shared-memory bytes) of lane groups of G lanes, ns sets per warp."""
    dpw = 32 // G
    sets = sum(((x // Ld) ** 2 // 4 + dpw - 1) // dpw for x in L)
    warps = 4 * sets if ns == 1 else 2 * ((sets + ns // 2 - 1) // (ns // 2))
    return (warps + wpb - 1) // wpb, wpb, 31 * 16 + wpb * ns * dpw * _domain_bytes(Ld, G)


CASES = [  # L, L_d, k, lanes per domain, sets per warp, warps per CTA by default
    ([32, 96, 64], 16, [3, 1, 2], 16, 1, 4),
    ([32, 96, 64], 16, [16, 9, 40], 16, 2, 4),
    ([512, 480], 16, [4, 3], 16, 1, 4),
    ([512, 480], 16, [16, 20], 16, 2, 4),
    ([1024], 16, [4], 8, 1, 4),
    ([1024], 16, [9], 8, 2, 4),
    ([64, 192], 32, [1, 4], 32, 1, 4),
    ([64, 192, 128], 32, [33, 8, 70], 32, 2, 4),
    ([1024, 704], 32, [2, 1], 16, 1, 4),
    ([1536], 32, [9], 16, 2, 4),
    ([2048], 32, [2], 8, 1, 4),
    ([2048], 32, [9], 8, 2, 4),
    ([128, 384], 64, [5, 2], 32, 1, 4),
    ([128, 384], 64, [20, 33], 32, 2, 4),
    ([2048, 1152], 64, [3, 2], 16, 1, 4),
    ([3072], 64, [8], 16, 2, 4),
    ([64] * 100, 16, [2] * 100, 16, 1, 8),    # small replicas, short visits
    ([64] * 100, 16, [3] * 100, 16, 1, 4),
    ([64] * 16, 16, [1] * 16, 16, 1, 4),      # ... but few of them
    ([128] * 140, 16, [4] * 140, 8, 2, 8),    # two sets per warp for want of room
    ([128] * 140, 16, [8] * 140, 8, 2, 4),
]


@pytest.mark.parametrize("L,Ld,ks,G,ns,wpb", CASES)
def test_lanes_sets_and_warps(L, Ld, ks, G, ns, wpb):
    import paper_1403_4674_gb300 as kmc
    lat = kmc.Lattice(L, Ld, 1, list(range(1, 1 + len(L))))
    lat.set_replica_params(k=ks)
    assert lat.launch()[0] == THREADS and lat.launch()[2:] == _shape(L, Ld, G, ns, wpb)
    lat.set_launch(THREADS, 2, 3)
    assert lat.launch()[0] == THREADS and lat.launch()[2:] == _shape(L, Ld, G, ns, 3)
    lat.set_launch()
    lat.run(1, schedule=kmc.KMC_SCHEDULE_RANDOM_PERM)
    lat.sync()
    assert lat.launch()[0] == GRID and lat.launch()[2:] == _shape(L, Ld, G, ns, wpb)
    lat.close()


@pytest.mark.parametrize("L,Ld,ks", [([1024], 16, [4]), ([1024], 16, [9]), ([1536], 32, [9]), ([64] * 100, 16, [1, 2] * 50),
                                     ([128] * 140, 16, [4, 2] * 70)])
@pytest.mark.parametrize("schedule", [0, 2])
def test_lane_groups_equal_the_warp_kernel(L, Ld, ks, schedule):
    import numpy as np
    import paper_1403_4674_gb300 as kmc
    out = []
    for plan in (None, (GRID, 2 * SM, 8)):
        lat = kmc.Lattice(L, Ld, 1, list(range(1, 1 + len(L))))
        lat.set_replica_params(k=ks)
        if plan:
            lat.set_launch(*plan)
        lat.set_rates([0.3 + 0.02 * (i % 8) for i in range(len(L))], [0.01] * len(L))
        obs = lat.run(6, schedule=schedule, obs_every=2).cpu().numpy()
        lat.sync()
        out.append((lat.spins.cpu().numpy(), *lat.domain_state(), obs))
        lat.close()
    a, b = out
    assert all(np.array_equal(a[i], b[i]) for i in range(3)) and np.array_equal(a[4][..., :3], b[4][..., :3])
    np.testing.assert_allclose(a[3], b[3], rtol=1e-12, atol=0)
    np.testing.assert_allclose(a[4][..., 3], b[4][..., 3], rtol=1e-12, atol=0)


@pytest.mark.parametrize("L,Ld,k", [([1600], 16, 1), ([3200], 32, 8), ([4608], 64, 4)])
def test_more_domains_take_a_thread_each(L, Ld, k):
    import paper_1403_4674_gb300 as kmc
    lat = kmc.Lattice(L, Ld, k, [1])
    mode, _, ctas, wpb, _ = lat.launch()
    assert mode == THREADS and wpb == 1 and ctas == 4 * (((L[0] // Ld) ** 2 // 4 + 31) // 32)
    lat.close()
