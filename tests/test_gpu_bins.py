"""Rods of one plan stay one launch wherever launches cannot overlap: under a mailbox (whose rods run
together), in a rollout, in a caller's capture; split by block size only in the graph of a repeated step."""
import numpy as np
import pytest

from paper_2509_04277_gb300 import workloads as W

pytestmark = pytest.mark.gpu

LENGTHS = (600, 900, 700, 1000)  # one plan, <4, 256>; blocks of 160, 256, 192 and 256 threads


@pytest.fixture(scope="module")
def corde(cuda):
    from paper_2509_04277_gb300 import build, corde as C

    build.build()
    C.load()
    return C


def _rods(times=1):
    return [W.guidewire(n, seed=n) for n in LENGTHS] * times


def _same(a, b):
    for k in a:
        np.testing.assert_array_equal(a[k].view(np.uint32), b[k].view(np.uint32), err_msg=k)


def test_lockstep_rods_of_one_plan_run_together(corde):
    """Each tick waits for the snapshots of every rod before it writes the next input."""
    import torch

    rods = _rods()
    a, b = corde.RodBatch(rods), corde.RodBatch(rods)
    assert len({tuple(p) for p in a.plan()}) == 1
    corde.rod_mailbox_enable(a.handle, 10, 256)
    corde.rod_mailbox_positions_enable(a.handle)
    corde.rod_mailbox_lockstep(a.handle, True, 300_000)
    drives = np.zeros((5, len(rods), 8), np.float32)
    drives[:, :, 0] = 0.01 * np.arange(1, 6)[:, None]
    snaps = np.zeros((5, a.n_elem, 4), np.float32)
    a.step(50)
    assert a.last_launch_count() == 1
    for k in range(5):
        corde.rod_mailbox_write(a.handle, drives[k])
        for r, off in enumerate(a.offsets[:-1]):
            out = snaps[k, off:off + LENGTHS[r]]
            assert corde.rod_mailbox_exchange(a.handle, None, r, 10 * (k + 1), out, 200_000) == 10 * (k + 1)
    torch.cuda.synchronize()
    assert corde.rod_mailbox_status(a.handle) == 0
    corde.rod_mailbox_disable(a.handle)
    for k in range(5):
        b.step(10, drive=torch.as_tensor(drives[k], device="cuda"))
        np.testing.assert_array_equal(snaps[k], b.state_numpy()["pos4"])
    a.close()
    b.close()


@pytest.mark.parametrize("lengths", [LENGTHS, (300, 600, 900, 40), (12000, 300, 5000)])
def test_caller_capture(corde, lengths):
    """A step in a caller's capture, the first of its handle or a repeated one, replays like direct steps."""
    import torch

    rods = [W.guidewire(n, seed=n) for n in lengths]
    for before in (0, 3):
        a, b = corde.RodBatch(rods), corde.RodBatch(rods)
        pos_out = torch.zeros((a.n_elem, 4), device="cuda")
        for _ in range(before):
            corde.rod_step_io(a.handle, 7, None, pos_out)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            corde.rod_step_io(a.handle, 7, None, pos_out)
        for _ in range(3):
            g.replay()
        torch.cuda.synchronize()
        for _ in range(before + 3):
            b.step(7)
        sb = b.state_numpy()
        _same(a.state_numpy(), sb)
        np.testing.assert_array_equal(pos_out.cpu().numpy(), sb["pos4"])
        a.close()
        b.close()


def test_launches(corde):
    """Once per plan directly, in a rollout and with graphs off; split in the graph of a repeated step,
    which takes up a changed output, drive and step count; the same bits throughout.  240 rods of
    6.75 warps fill the GPU; four do not, and stay one launch."""
    import torch

    c = corde.RodBatch(_rods())
    for _ in range(3):
        c.step(2)
        assert c.last_launch_count() == 1
    c.close()
    rods = _rods(60)
    a, b = corde.RodBatch(rods), corde.RodBatch(rods)
    b.set_graph_mode(0)
    outs = [torch.zeros((a.n_elem, 4), device="cuda") for _ in range(2)]
    drive = torch.zeros((len(rods), 8), device="cuda")
    count = []
    for n, o, v in ((5, 0, 0.0), (5, 0, 0.01), (5, 0, 0.02), (5, 1, 0.03), (5, 0, 0.0), (6, 0, 0.01), (6, 0, 0.0), (5, 0, 0.0)):
        drive[:, 0] = v
        corde.rod_step_io(a.handle, n, drive, outs[o])
        count.append(a.last_launch_count())
        b.step(n, drive=drive)
        assert b.last_launch_count() == 1
        sb = b.state_numpy()
        _same(a.state_numpy(), sb)
        np.testing.assert_array_equal(outs[o].cpu().numpy(), sb["pos4"])
    assert count == [1, 3, 3, 1, 1, 1, 3, 1]
    a.rollout(6, 3)
    assert a.last_launch_count() == 2
    b.rollout(6, 3)
    _same(a.state_numpy(), b.state_numpy())
    a.close()
    b.close()


def test_concurrent_launches_of_a_first_step(corde):
    """Several plans: a step unlike the one before it launches them on branches that its stream waits for."""
    import torch

    rods = [W.guidewire(n, seed=n) for n in (40, 200, 600, 900, 3000, 12000)]
    a, b = corde.RodBatch(rods), corde.RodBatch(rods)
    b.set_graph_mode(0)
    s = torch.cuda.Stream()
    drive = torch.zeros((len(rods), 8), device="cuda")
    drive[:, 0] = 0.02
    out = {k: torch.zeros((a.n_elem, 4), device="cuda") for k in ("pos4", "quat4", "vel4", "omega4")}
    torch.cuda.synchronize()
    for n in (1, 2, 3, 4):
        a.step(n, drive=drive, stream=s)
        b.step(n, drive=drive)
    corde.rod_get_state(a.handle, *out.values(), stream=s)
    s.synchronize()
    sb = b.state_numpy()
    for k in ("pos4", "vel4"):
        np.testing.assert_array_equal(out[k].cpu().numpy(), sb[k], err_msg=k)
    a.close()
    b.close()
