"""rod_autotune times what runs: the block variants for nt, also where tiles step the rod, since a
mailbox launch runs on the block; the state is as it was."""
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


# 512 nodes: <2, 256> steps 2.50 us as a block, <2, 512> 3.62; tiles step both in 1.88
def test_same_plan_every_time(corde):
    plans = set()
    for k in range(10):
        b = corde.RodBatch([W.guidewire(512, seed=k)])
        b.set_tiles(k % 5 != 4)
        if k % 5 == 3:
            corde.rod_mailbox_enable(b.handle, 1 << 20)
        before = b.state_numpy()
        b.autotune(10)
        after = b.state_numpy()
        for key in before:
            np.testing.assert_array_equal(before[key], after[key])
        plans.add(tuple(b.plan()[0]))
        b.close()
    assert plans == {(2, 256, 0)}


@pytest.mark.parametrize("count", [40, 700])
def test_uneven_rods(corde, count):
    """Classes whose rods share bins, tiles and trimmed blocks with others; the results are the plan's."""
    rods = W.batched_rods(count, seed=45) + list(W.catheter_guidewire(64, seed=1, beta0=-6.5))
    a, b = corde.RodBatch(rods), corde.RodBatch(rods)
    for h in (a, b):
        h.bind(count, count + 1, 2)
    a.step(3)
    before = a.state_numpy()
    a.autotune(10)
    after = a.state_numpy()
    for k in before:
        np.testing.assert_array_equal(before[k], after[k], err_msg=k)
    plan = a.plan()
    assert all(p[2] != 0 or p[0] * p[1] >= n for p, n in zip(plan, a.n_nodes[:count]))
    b.step(3)
    for _ in range(3):
        a.step(5)
        b.step(5)
    sa, sb = a.state_numpy(), b.state_numpy()
    assert np.abs(sa["pos4"] - sb["pos4"]).max() < 1e-5
    a.close()
    b.close()
