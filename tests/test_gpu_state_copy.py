"""rod_get_state and rod_set_state between device buffers (one copy kernel), host buffers and
device buffers that are not 16-byte aligned (a copy each): the same bytes, arrays that are
not given untouched, and the inverse masses kept."""
import numpy as np
import pytest

from paper_2509_04277_gb300 import workloads as W

pytestmark = pytest.mark.gpu
KEYS = ("pos4", "quat4", "vel4", "omega4")


@pytest.fixture(scope="module")
def corde(cuda):
    from paper_2509_04277_gb300 import build, corde as C

    build.build()
    C.load()
    return C


@pytest.mark.parametrize("given", [(1, 1, 1, 1), (0, 1, 1, 1), (1, 0, 0, 0), (0, 0, 0, 1)])
@pytest.mark.parametrize("shift", [0, 1])  # floats off a 16-byte boundary
@pytest.mark.parametrize("n", [2, 127, 128, 129, 700])
def test_device_buffers(corde, n, shift, given):
    import torch

    b = corde.RodBatch([W.guidewire(n, seed=n), W.guidewire(3, seed=1)])
    b.step(5)
    host = b.state_numpy()
    E = b.n_elem

    def buffers(fill):
        return [torch.full((4 * E + 4,), fill, device="cuda")[shift:shift + 4 * E] for _ in KEYS]

    out = buffers(-7.0)
    corde.rod_get_state(b.handle, *[o if g else None for o, g in zip(out, given)])
    for o, g, k in zip(out, given, KEYS):
        got = o.cpu().numpy().reshape(E, 4)
        assert np.array_equal(got, host[k] if g else np.full((E, 4), -7.0, np.float32))
    new = buffers(0.0)
    gen = torch.Generator(device="cuda").manual_seed(n)
    for t in new:
        t.copy_(torch.rand(4 * E, generator=gen, device="cuda"))
    corde.rod_set_state(b.handle, *[t if g else None for t, g in zip(new, given)])
    after = b.state_numpy()
    for t, g, k in zip(new, given, KEYS):
        want = t.cpu().numpy().reshape(E, 4) if g else host[k]
        if k == "pos4":
            want = np.concatenate([want[:, :3], host[k][:, 3:]], axis=1)
        assert np.array_equal(after[k], want)
    b.close()


# one element per thread up to 65536, four above; the arrays not given leave no gap
@pytest.mark.parametrize("given", [(1, 1, 1, 1), (1, 0, 1, 0), (0, 1, 0, 1), (0, 0, 1, 0)])
@pytest.mark.parametrize("extra", [None, 2, 3, 1027])
def test_many_elements(corde, extra, given):
    import torch

    rods = [W.guidewire(512, seed=1)] * 128 + ([W.guidewire(extra, seed=2)] if extra else [])
    b = corde.RodBatch(rods)
    b.step(2)
    host, E = b.state_numpy(), b.n_elem
    out = [torch.full((E + 1, 4), -7.0, device="cuda") for _ in KEYS]
    corde.rod_get_state(b.handle, *[o if g else None for o, g in zip(out, given)])
    for o, g, k in zip(out, given, KEYS):
        got = o.cpu().numpy()
        assert np.array_equal(got[:E], host[k] if g else np.full((E, 4), -7.0, np.float32)), k
        assert (got[E] == -7.0).all()
    new = [torch.rand((E, 4), device="cuda") for _ in KEYS]
    corde.rod_set_state(b.handle, *[t if g else None for t, g in zip(new, given)])
    after = b.state_numpy()
    for t, g, k in zip(new, given, KEYS):
        want = t.cpu().numpy() if g else host[k]
        if k == "pos4":
            want = np.concatenate([want[:, :3], host[k][:, 3:]], axis=1)
        assert np.array_equal(after[k], want), k
    b.close()


@pytest.mark.parametrize("which", [0, 2])
def test_buffer_that_ends_too_early(corde, which):
    """A device buffer up to the end of its allocation serves; one that is shorter is refused on the host."""
    import torch

    E = 65536
    b = corde.RodBatch([W.guidewire(512, seed=1)] * 128)
    # torch hands allocations above 10 MB out whole, in multiples of 2 MB
    big = torch.empty(32 << 20, dtype=torch.uint8, device="cuda")
    assert big.untyped_storage().nbytes() % (2 << 20) == 0
    rest = [torch.zeros((E, 4), device="cuda") for _ in KEYS]

    def given(spare):
        args = list(rest)
        args[which] = big.data_ptr() + big.numel() - 16 * (E - spare)
        return args

    corde.rod_get_state(b.handle, *given(0))
    want = b.state_numpy()[KEYS[which]]
    assert np.array_equal(big[-16 * E:].view(torch.float32).cpu().numpy().reshape(E, 4), want)
    corde.rod_set_state(b.handle, *given(0))
    for spare in (1, E // 2):
        for call in (corde.rod_get_state, corde.rod_set_state):
            with pytest.raises(corde.CordeError):
                call(b.handle, *given(spare))
    torch.cuda.synchronize()
    b.close()
