"""The arrays hold one frame and two joints more than a rod has (the last element's frame, the last
two elements' joints).  Whatever stands there, NaN and infinities included, neither reaches the
step nor is changed by it, on every stepping kernel."""
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


def _rods(kind):
    if kind == "pair":
        return list(W.catheter_guidewire(64, seed=3, beta0=-6.5))
    if kind == "knot":
        return [W.torus_knot(130, seed=4)]
    if kind == "extensible":
        return [W.extensible_pendulum(65, seed=4)]
    return [W.guidewire(n, seed=n) for n in {"short": (2, 3), "block": (300,), "long": (2500,), "many": (66,) * 200}[kind]]


@pytest.mark.parametrize("box", [False, True])  # with a mailbox: the block, cluster and pair kernels
@pytest.mark.parametrize("kind", ["short", "block", "long", "many", "extensible", "pair", "knot"])
@pytest.mark.parametrize("junk", [float("nan"), float("inf")])
def test_step_ignores_padding(corde, kind, box, junk):
    import torch

    if kind == "knot" and box:
        pytest.skip("self-collision runs without a mailbox")
    rods = _rods(kind)
    a, b = corde.RodBatch(rods), corde.RodBatch(rods)
    last = torch.as_tensor(a.offsets[1:] - 1, device="cuda")
    state = {k: torch.as_tensor(v, device="cuda") for k, v in b.state_numpy().items()}
    joints = torch.as_tensor(b.per_joint(), device="cuda")
    for k in ("quat4", "omega4"):
        state[k][last] = junk
    joints[last] = junk
    joints[(last - 1).clamp_min(0)] = junk
    corde.rod_set_state(b.handle, *state.values())
    corde.rod_set_material(b.handle, joints)
    for h in (a, b):
        if kind == "pair":
            h.bind(0, 1, 2)
        if kind == "knot":
            h.set_self_collision(0, 0.1)
        if box:
            corde.rod_mailbox_enable(h.handle, 1 << 20)
        h.step(7)
    sa, sb = a.state_numpy(), b.state_numpy()
    keep = np.ones(a.n_elem, bool)
    keep[last.cpu().numpy()] = False
    for k in ("pos4", "vel4"):
        assert np.isfinite(sa[k]).all()
        np.testing.assert_array_equal(sa[k], sb[k], err_msg=k)
    for k in ("quat4", "omega4"):
        np.testing.assert_array_equal(sa[k][keep], sb[k][keep], err_msg=k)
    np.testing.assert_array_equal(sb["quat4"][~keep], np.full((len(rods), 4), junk, np.float32))
    a.close()
    b.close()
