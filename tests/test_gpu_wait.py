"""A wait for a neighbouring tile that runs out: no finite value of that launch is left to be taken
for a result, the host can read what happened, and the handle goes on once its state is set again."""
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


# two tiles a block, and six; with a limit of no polls at all, some tile finds its neighbour late
@pytest.mark.parametrize("n", [12000, 65536])
def test_wait_that_runs_out(corde, n):
    import torch

    rod = W.guidewire(n, seed=n)
    ref, b = corde.RodBatch([rod]), corde.RodBatch([rod])
    assert b.kernels()[0][0] == "tiles_grid"
    start = [torch.as_tensor(x).cuda() for x in b.state_numpy().values()]
    ref.step(20)
    want = ref.state_numpy()
    ref.close()

    corde.rod_set_wait_limit(b.handle, 0)
    pos_out = torch.zeros((n, 4), device="cuda")
    corde.rod_step_io(b.handle, 20, None, pos_out)
    st = b.state_numpy()
    for k in ("pos4", "vel4", "omega4"):
        assert np.isnan(st[k][:, :3]).all(), k
    assert np.isnan(st["quat4"][:-1]).all()
    assert torch.isnan(pos_out[:, :3]).all()
    assert np.isfinite(st["pos4"][:, 3]).all()  # the masses stay
    assert b.diagnostics()[0] == corde.CORDE_ERR_NONFINITE
    assert corde.rod_wait_status(b.handle) == 1
    assert corde.rod_wait_status(b.handle) == 0

    # trajectory rows
    corde.rod_set_state(b.handle, *start)
    traj = b.rollout(20, 10)
    assert torch.isnan(traj[:, :, :3]).all()

    # with time to wait the same handle steps as any other, also where the status was not read
    corde.rod_set_wait_limit(b.handle, 1 << 22)
    corde.rod_set_state(b.handle, *start)
    b.step(20)
    st = b.state_numpy()
    for k in want:
        np.testing.assert_array_equal(st[k].view(np.uint32), want[k].view(np.uint32), err_msg=k)
    b.close()


def test_nothing_lost_without_a_cause(corde):
    b = corde.RodBatch([W.guidewire(20000, seed=1), W.guidewire(300, seed=2)])
    assert [k[0] for k in b.kernels()] == ["tiles_grid", "tiles"]
    b.step(50)
    assert corde.rod_wait_status(b.handle) == 0
    b.close()


@pytest.mark.parametrize("n", [20000, 65536])
def test_grid_beside_a_running_launch(corde, n):
    """A lock-step launch of another handle holds its SM until its wait for the host runs out, after 1 s; the
    grid's steps start and end meanwhile."""
    import time

    import torch

    a, b, c = corde.RodBatch([W.guidewire(512, seed=1)]), corde.RodBatch([W.guidewire(n, seed=2)]), corde.RodBatch([W.guidewire(n, seed=2)])
    c.step(10)
    c.step(10)
    want = c.state_numpy()
    a.step(10)
    corde.rod_mailbox_enable(a.handle, 10, 64)
    corde.rod_mailbox_lockstep(a.handle, True, 1_000_000)
    sa, sb = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    t0 = time.time()
    a.step(50, stream=sa)
    for _ in range(2):
        b.step(10, stream=sb)
    sb.synchronize()
    took = time.time() - t0
    sa.synchronize()
    assert corde.rod_mailbox_status(a.handle) & 1  # it did run, and waited
    assert took < 0.5 <= time.time() - t0
    st = b.state_numpy()
    for k in want:
        np.testing.assert_array_equal(st[k].view(np.uint32), want[k].view(np.uint32), err_msg=k)
    for h in (a, b, c):
        h.close()
