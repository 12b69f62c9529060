"""The tile kernel (overlapping warp tiles) against the block and cluster kernels, which a
mailbox keeps a rod on: every element takes the same arithmetic, so the states are the same
bit for bit, whatever the length, the iteration count and the steps per launch."""
import numpy as np
import pytest

from paper_2509_04277_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def corde(cuda):
    from paper_2509_04277_gb300 import build, corde as C

    build.build()
    C.load()
    return C


def _bits(a, b):
    return all(np.array_equal(a[k].view(np.uint32), b[k].view(np.uint32)) for k in a)


def _pair(corde, rods, plan=None, tube=None):
    """The same rods on the tile kernel and, under a mailbox, on the others."""
    out = []
    for box in (False, True):
        b = corde.RodBatch(rods)
        if plan is not None:
            (b.set_plan if len(plan) == 2 else b.set_plan_cluster)(*plan)
        if tube is not None:
            b.set_tube(0, tube)
        if box:
            corde.rod_mailbox_enable(b.handle, 1 << 20)
        out.append(b)
    return out


def _check(corde, rods, calls, plan=None, tube=None):
    import torch

    g = W.rng(sum(r.n_nodes for r in rods))
    drive = torch.zeros((len(rods), 8), device="cuda")
    drive[:, 0:3] = torch.as_tensor(g.uniform(-0.1, 0.1, (len(rods), 3)))
    drive[:, 6] = 2.0
    a, b = _pair(corde, rods, plan, tube)
    for steps in calls:
        a.step(steps, drive=drive)
        b.step(steps, drive=drive)
        assert _bits(a.state_numpy(), b.state_numpy())
    a.close()
    b.close()


# the tiles' edges: one warp of 2 (4) elements a lane holds 64 (128) nodes, a further tile 20 (80)
@pytest.mark.parametrize("n", [2, 3, 63, 64, 65, 84, 85, 128, 129, 333, 512, 1205, 2048])
@pytest.mark.parametrize("plan", [None, (2, 512)])
def test_lengths(corde, n, plan):
    if plan is not None and n > 1024:
        plan = (2, 256, 8)
    _check(corde, [W.guidewire(n, seed=900 + n)], (1, 10), plan)


# 2304 nodes: the last length at two elements a lane; 10384: the last of a cluster's tiles
@pytest.mark.parametrize("n", [2304, 2305, 5001, 10384, 10385, 32768])
def test_long_rods(corde, n):
    _check(corde, [W.guidewire(n, seed=900 + n)], (1, 3))


# more than eight warps on every SM (half the registers): the grid kernel, which several rods keep to
def test_longest_rods(corde):
    import torch

    n = 100_001
    rod = W.guidewire(n, seed=6)
    a, b = corde.RodBatch([rod]), corde.RodBatch([rod, W.guidewire(n, seed=7)])
    for steps in (1, 3):
        a.step(steps)
        b.step(steps)
    sa, sb = a.state_numpy(), b.state_numpy()
    assert all(np.array_equal(sa[k][:n].view(np.uint32), sb[k][:n].view(np.uint32)) for k in sa)
    torch.cuda.synchronize()
    a.close()
    b.close()


# iterations per exchange (10 and 11 fill the ghosts), velocity exchanges within a step beyond
@pytest.mark.parametrize("iters", [0, 1, 2, 4, 5, 9, 10, 11, 12, 21, 22, 37])
@pytest.mark.parametrize("n,plan", [(300, None), (300, (2, 256)), (4000, None)])
def test_iteration_counts(corde, iters, n, plan):
    rod = W.guidewire(n, seed=iters)
    rod.n_iters = iters
    _check(corde, [rod], (1, 12), plan)


# an extensible rod runs up to 22 (24) steps between two exchanges
@pytest.mark.parametrize("n", [64, 500, 3001])
def test_extensible(corde, n):
    _check(corde, [W.extensible_pendulum(n, seed=n)], (1, 22, 23, 50))


@pytest.mark.parametrize("n,iters", [(100, 10), (512, 10), (512, 25), (3000, 10)])
def test_vessel(corde, n, iters):
    rod, tube = W.vessel_guidewire(n, seed=n)
    rod.n_iters = iters
    _check(corde, [rod], (1, 10), tube=tube)


def test_uneven_rods_in_one_handle(corde):
    _check(corde, W.batched_rods(12, seed=77), (1, 10))


# more rods than SMs: one tile per rod (64 and 128 nodes; 1300 rods fill the SMs), two and three tiles in a
# block, and too many for either
@pytest.mark.parametrize("n,count,plan", [(64, 200, None), (64, 200, (4, 32)), (100, 200, None), (128, 1300, None),
                                          (100, 200, (2, 64)), (200, 300, None), (270, 200, (2, 256)), (200, 700, None)])
def test_many_rods(corde, n, count, plan):
    rod = W.guidewire(n, seed=n)
    _check(corde, [rod] * count, (1, 10), plan)


def test_free_base(corde):
    rod = W.guidewire(200, seed=5)
    rod.clamp = 0
    rod.gravity = (0.0, 0.0, -9.81)
    _check(corde, [rod], (1, 10))


# a rod of tiles on a cooperative grid beside bins of other rods: the step is a graph of parallel branches
@pytest.mark.parametrize("ns", [(20000, 300), (20000, 300, 300, 700), (11000, 20000, 5000)])
def test_grid_of_tiles_beside_other_rods(corde, ns):
    _check(corde, [W.guidewire(n, seed=n) for n in ns], (1, 10, 10))


# tiles on a grid wait for their neighbours' data: several exchanges a step, one in several steps, call after call
@pytest.mark.parametrize("n,iters", [(12000, 0), (12000, 4), (12000, 25), (32768, 12)])
def test_grid_exchanges(corde, n, iters):
    rod = W.guidewire(n, seed=iters)
    rod.n_iters = iters
    _check(corde, [rod], (1, 12, 1, 7, 30))
