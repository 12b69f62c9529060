"""Which kernel steps a rod, and the block, cluster, grid, pair and pipelined kernels with the warp
tiles switched off: against the oracle, against each other and against the tiles, bit for bit."""
import dataclasses

import numpy as np
import pytest

import oracle
from paper_2509_04277_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def corde(cuda):
    from paper_2509_04277_gb300 import build, corde as C

    build.build()
    C.load()
    return C


def _states(corde, rods, calls, kind, tiles=True, setup=None):
    """States after the calls on a handle whose rods all run on kernels of the named kinds."""
    import torch

    b = corde.RodBatch(rods)
    b.set_tiles(tiles)
    if setup is not None:
        setup(b)
    kinds = [k[0] for k in b.kernels()]
    assert kinds == ([kind] * len(rods) if isinstance(kind, str) else list(kind)), kinds
    drive = torch.zeros((len(rods), 8), device="cuda")
    drive[:, 0], drive[:, 1], drive[:, 4], drive[:, 6] = 0.02, -0.01, 0.1, 2.0
    for n in calls:
        b.step(n, drive=drive)
    out = b.state_numpy()
    b.close()
    return out


def _same(a, b):
    for k in a:
        np.testing.assert_array_equal(a[k].view(np.uint32), b[k].view(np.uint32), err_msg=k)


# position error over the rod's length after up to 30 steps, and that of the quaternions, as in the parity tests
ROLL_TOL, QUAT_TOL = 1e-4, 1e-4


def _oracle(rods, st, steps):
    drive = np.array([0.02, -0.01, 0, 0, 0.1, 0, 2.0, 0])
    off = 0
    for rod in rods:
        n = rod.n_nodes
        ref = oracle.step(rod, oracle.state_of(rod), steps, drive=drive)
        assert np.abs(st["pos4"][off:off + n, :3] - ref["pos"]).max() <= ROLL_TOL * rod.length
        assert np.abs(st["quat4"][off:off + n - 1] - ref["quat"]).max() <= QUAT_TOL
        off += n


@pytest.mark.parametrize("n,kind,off", [(64, "tiles", "block"), (512, "tiles", "block"), (2049, "tiles", "cluster"),
                                        (12000, "tiles_grid", "cluster"), (40000, "tiles_grid", "grid")])
def test_default_kernels(corde, n, kind, off):
    rod = W.guidewire(n, seed=n)
    a = _states(corde, [rod], (1, 10), kind)
    b = _states(corde, [rod], (1, 10), off, tiles=False)
    _same(a, b)


@pytest.mark.parametrize("ept,nt,C", [(2, 256, 8), (4, 256, 4), (4, 512, 3)])
def test_cluster_and_grid_kernels(corde, ept, nt, C):
    """Both kernels on the same blocks, one rod and two of uneven lengths: the oracle's states, and
    the same bits as each other and as the tiles."""
    full = min(ept * nt * C, 4096)
    for lengths in ((full - 5,), (full, full // 2 + 3)):
        rods = [W.guidewire(n, seed=540 + n) for n in lengths]
        c = _states(corde, rods, (10, 10), "cluster", False, lambda b: b.set_plan_cluster(ept, nt, C))
        g = _states(corde, rods, (10, 10), "grid", False, lambda b: b.set_plan_grid(ept, nt, C))
        t = _states(corde, rods, (10, 10), "tiles", True, lambda b: b.set_plan_cluster(ept, nt, C))
        _same(c, g)
        _same(c, t)
        _oracle(rods, c, 20)


def test_cluster_kernel_of_16_blocks(corde):
    import torch

    rod = W.guidewire(8192, seed=520)
    try:
        c = _states(corde, [rod], (5,), "cluster", False, lambda b: b.set_plan_cluster(2, 256, 16))
    except corde.CordeError as e:
        torch.cuda.synchronize()
        pytest.skip(f"16-block cluster not schedulable: {e}")
    _oracle([rod], c, 5)


@pytest.mark.parametrize("mode", [0, 1, 2])
def test_pair_kernels(corde, mode):
    rods = W.catheter_guidewire(300, seed=31, beta0=-40.25)
    a = _states(corde, rods, (1, 10), "pair_tiles", True, lambda b: b.bind(0, 1, mode))
    b = _states(corde, rods, (1, 10), "pair", False, lambda b: b.bind(0, 1, mode))
    _same(a, b)


def test_reverse_kernels(corde):
    """One block per rod, the two-block pipeline and the tiles: the same gradients bit for bit for rods of
    three lengths and iteration counts, with one segment, and several with a short last one."""
    import torch

    rods = [dataclasses.replace(W.adjoint_rod(n, seed=1500 + n), n_iters=it) for n, it in ((64, 4), (200, 10), (256, 7))]
    for n_steps, every in ((47, 10), (12, 20), (21, 7)):
        out = {}
        for kind, tiles, pipe in (("block", False, False), ("pipelined", False, True), ("tiles", True, True)):
            b = corde.RodBatch(rods)
            b.set_tiles(tiles)
            b.set_adjoint_pipeline(pipe)
            traj = b.rollout(n_steps, every)
            g = torch.zeros_like(traj)
            g[:, :, :3] = 1e-2 * torch.cos(traj[:, :, :3] * 23.0)
            out[kind] = {k: v.cpu().numpy() for k, v in b.adjoint(g).items()}
            out[kind]["traj"] = traj.cpu().numpy()
            ran = corde.rod_adjoint_kernels(b.handle)
            assert ran[kind] > 0 and sum(ran.values()) == ran[kind], ran
            b.close()
        for kind in ("pipelined", "tiles"):
            for k in out["block"]:
                assert np.isfinite(out["block"][k]).all(), k
                np.testing.assert_array_equal(out["block"][k], out[kind][k], err_msg=f"{n_steps} steps, {kind}: {k}")


def test_switch(corde):
    """The switch takes effect between steps, also for the reverse pass, and refuses other values."""
    rod = W.adjoint_rod(200, seed=3)
    b = corde.RodBatch([rod])
    assert b.kernels()[0][0] == "tiles"
    corde.rod_mailbox_enable(b.handle, 1 << 20)
    assert b.kernels()[0][0] == "block"
    corde.rod_mailbox_disable(b.handle)
    for tiles, kind, rev in ((False, "block", "pipelined"), (True, "tiles", "tiles")):
        b.set_tiles(tiles)
        assert b.kernels()[0][0] == kind
        b.rollout(8, 4)
        b.adjoint(None)
        assert corde.rod_adjoint_kernels(b.handle)[rev] == 1
    with pytest.raises(corde.CordeError):
        corde.rod_set_tiles(b.handle, 2)
    b.close()
