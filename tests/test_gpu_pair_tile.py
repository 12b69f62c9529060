"""The pair's tile kernel against its block kernel, which a mailbox keeps a pair on: the same
states bit for bit for every mode, binding offsets of both parities (the two layouts of the
colors), rods that only partly or never overlap, and both arithmetic layouts."""
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


def _same(corde, n, mode, betas, iters=10, n_in=None):
    import torch

    cat, gw = W.catheter_guidewire(n, seed=n + mode, beta0=betas[0])
    if n_in is not None:  # a shorter inner rod with the same segment length
        gw = W.straight_rod(n_in, gw.length * (n_in - 1) / (n - 1), base=gw.pos[0], seg_sigma=1e-3, ang_sigma=1e-3,
                            seed=n_in, radius=gw.radius, E_bend=gw.E_bend, E_stretch=gw.E_stretch, G=gw.G,
                            density=gw.density, dt=gw.dt, n_iters=gw.n_iters, inextensible=True, clamp=1,
                            damping_alpha=0.0)
    cat.n_iters = gw.n_iters = iters
    a, b = corde.RodBatch([cat, gw]), corde.RodBatch([cat, gw])
    for h in (a, b):
        h.bind(0, 1, mode)
    corde.rod_mailbox_enable(b.handle, 1 << 20)
    for k, beta in enumerate(betas):
        d = torch.zeros((2, 8), device="cuda")
        d[0, 0], d[1, 0], d[1, 6], d[1, 3] = 0.01, 0.05, 1.0, beta
        for h in (a, b):
            h.step(1 + 6 * (k % 2), drive=d)
        sa, sb = a.state_numpy(), b.state_numpy()
        assert all(np.array_equal(sa[q].view(np.uint32), sb[q].view(np.uint32)) for q in sa), (k, beta)
    a.close()
    b.close()


@pytest.mark.parametrize("mode", [0, 1, 2])
@pytest.mark.parametrize("n", [20, 64, 150, 512, 600, 1024])
def test_offsets(corde, n, mode):
    _same(corde, n, mode, [-0.2 * n - 0.25, -0.2 * n - 1.25, -3.0, 0.5, 1.5, 0.3 * n + 0.75])


@pytest.mark.parametrize("mode", [1, 2])
def test_no_overlap(corde, mode):
    _same(corde, 128, mode, [-128.5, -127.5, 127.25, 126.25, -1e6, 1e6 + 1])


@pytest.mark.parametrize("mode", [1, 2])
@pytest.mark.parametrize("iters", [1, 5, 6, 11, 20, 23])
def test_iteration_counts(corde, iters, mode):
    _same(corde, 300, mode, [-40.25, -41.25], iters)


@pytest.mark.parametrize("n,n_in", [(300, 100), (100, 300)])
def test_uneven_rods(corde, n, n_in):
    _same(corde, n, 2, [-10.25, -9.5, 20.0], n_in=n_in)
