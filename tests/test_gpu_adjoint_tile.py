"""The adjoint on warp tiles against the one-block reverse kernel: the same gradients bit for bit
for lengths at the tiles' edges, every iteration count the ghosts hold, short last segments,
extensible rods and several rods of different lengths; beyond (more iterations, a budget that
the records do not fit) the block kernels run."""
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


def _grads(corde, rods, n_steps, every, tiles, budget=None):
    import torch

    b = corde.RodBatch(rods)
    b.set_adjoint_pipeline(tiles)
    if budget is not None:
        b.set_adjoint_record_budget(budget)
    drive = np.zeros((len(rods), 8), np.float32)
    drive[:, 0], drive[:, 6] = 0.02, 1.0
    b.set_input(drive)
    traj = b.rollout(n_steps, every)
    g = torch.zeros_like(traj)
    g[:, :, :3] = 1e-2 * torch.cos(traj[:, :, :3] * 23.0)
    out = {k: v.cpu().numpy() for k, v in b.adjoint(g).items()}
    out["traj"] = traj.cpu().numpy()
    info = corde.rod_adjoint_info(b.handle)
    b.close()
    return out, info


def _same(corde, rods, n_steps=7, every=3):
    (a, ia), (c, ic) = (_grads(corde, rods, n_steps, every, t) for t in (True, False))
    assert ia["pipelined"] and not ic["pipelined"]
    for k in a:
        assert np.isfinite(a[k]).all(), k
        np.testing.assert_array_equal(a[k], c[k], err_msg=k)


@pytest.mark.parametrize("n", [2, 3, 63, 64, 65, 84, 85, 104, 144, 145, 256, 511, 512])
def test_lengths(corde, n):
    rod = W.adjoint_rod(n, seed=n) if n > 2 else W.guidewire(2, seed=2)
    _same(corde, [rod])


@pytest.mark.parametrize("iters", [0, 1, 2, 9, 10])
def test_iterations(corde, iters):
    rod = W.adjoint_rod(150, seed=iters)
    rod.n_iters = iters
    _same(corde, [rod])


@pytest.mark.parametrize("n_steps,every", [(1, 1), (4, 1), (5, 9), (9, 4)])
def test_segments(corde, n_steps, every):
    _same(corde, [W.adjoint_rod(100, seed=1)], n_steps, every)


def test_uneven_and_extensible_rods(corde):
    rods = [W.adjoint_rod(n, seed=n) for n in (40, 300, 90, 301, 512)]
    rods[2].n_iters = 4
    _same(corde, rods)
    _same(corde, [W.extensible_pendulum(100, seed=3)])


def test_where_the_tiles_end(corde):
    rod = W.adjoint_rod(100, seed=5)
    rod.n_iters = 11
    a, ia = _grads(corde, [rod], 6, 3, True)
    c, _ = _grads(corde, [rod], 6, 3, False)
    assert all(np.array_equal(a[k], c[k]) for k in a)
    assert ia["blocks"] == 2  # the two-block pipeline
    rod.n_iters = 10
    a, _ = _grads(corde, [rod], 6, 3, True)
    c, ic = _grads(corde, [rod], 6, 3, True, budget=100000)  # one segment's records fit, all six steps' do not
    assert ic["mode"] == "recompute" or ic["blocks"] <= 2
    assert all(np.array_equal(a[k], c[k]) for k in a)


def test_scratch_that_held_other_values(corde):
    """Records and states live in scratch that is not cleared: a reverse pass after one that left
    NaN there (a non-finite loss gradient and state) gives the gradients of a fresh handle."""
    import torch

    n_steps, every = 6, 3
    rod = W.adjoint_rod(101, seed=8)
    want, _ = _grads(corde, [rod], n_steps, every, True)
    b = corde.RodBatch([rod])
    drive = np.zeros((1, 8), np.float32)
    drive[:, 0], drive[:, 6] = 0.02, 1.0
    b.set_input(drive)
    start = [torch.as_tensor(v, device="cuda") for v in b.state_numpy().values()]
    corde.rod_set_state(b.handle, torch.full_like(start[0], float("nan")))
    b.adjoint(torch.full_like(b.rollout(n_steps, every), float("nan")))
    corde.rod_set_state(b.handle, *start)
    traj = b.rollout(n_steps, every)
    g = torch.zeros_like(traj)
    g[:, :, :3] = 1e-2 * torch.cos(traj[:, :, :3] * 23.0)
    got = {k: v.cpu().numpy() for k, v in b.adjoint(g).items()}
    for k in got:
        np.testing.assert_array_equal(got[k], want[k], err_msg=k)
    b.close()


def test_without_memory_for_the_whole_rollout(corde):
    """8 rods of 512 nodes over 700 steps: 0.9 GB of states and records, within the default budget but beyond
    what the device has left.  The segment-wise modes run instead, with the same gradients."""
    import torch

    rods = [W.adjoint_rod(512, seed=k) for k in range(8)]
    a, b = corde.RodBatch(rods), corde.RodBatch(rods)
    g = None
    for h in (a, b):
        traj = h.rollout(700, 20)
        if g is None:
            g = torch.zeros_like(traj)
            g[:, :, :3] = 1e-3 * torch.cos(traj[:, :, :3] * 23.0)
        del traj
    want = a.adjoint(g)
    assert corde.rod_adjoint_kernels(a.handle)["tiles"] == 1
    a.close()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    hold = []
    for keep, piece in ((3 << 30, None), (600 << 20, 256 << 20)):
        while torch.cuda.mem_get_info()[0] > keep + (piece or 0):
            hold.append(torch.empty(piece or torch.cuda.mem_get_info()[0] - keep, dtype=torch.uint8, device="cuda"))
    assert torch.cuda.mem_get_info()[0] < 900 << 20
    for _ in range(2):
        got = b.adjoint(g)
        ran = corde.rod_adjoint_kernels(b.handle)
        assert ran["tiles"] == 0 and sum(ran.values()) == 1, ran
        for k in want:
            assert torch.equal(got[k], want[k]), k
    hold.clear()
    torch.cuda.empty_cache()
    b.set_adjoint_record_budget(1 << 30)
    got = b.adjoint(g)
    assert corde.rod_adjoint_kernels(b.handle)["tiles"] == 1
    for k in want:
        assert torch.equal(got[k], want[k]), k
    b.close()
