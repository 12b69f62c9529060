"""Tiles that the device does not hold all at once: large clusters, several bins of pairs and rods beside
them, always with the results of the kernels without tiles."""
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


def _run(corde, rods, pairs, tiles):
    b = corde.RodBatch(rods)
    b.set_tiles(tiles)
    for p in pairs:
        b.bind(*p)
    for n in (1, 6, 6):
        b.step(n)
    out, kernels = b.state_numpy(), b.kernels()
    b.close()
    return out, kernels


def _same(a, b):
    for k in a:
        np.testing.assert_array_equal(a[k].view(np.uint32), b[k].view(np.uint32), err_msg=k)


# a cluster of 16 blocks needs 16 SMs of one GPC: eight rods of 2048 or 10000 nodes find the SMs, not the GPCs
@pytest.mark.parametrize("n,count,kinds", [(2048, 1, {"tiles"}), (2048, 8, {"tiles"}), (10000, 1, {"tiles"}),
                                           (10000, 8, {"cluster"}), (1500, 9, {"tiles"})])
def test_rods_of_large_clusters(corde, n, count, kinds):
    rods = [W.guidewire(n, seed=k) for k in range(count)]
    a, ka = _run(corde, rods, (), True)
    b, _ = _run(corde, rods, (), False)
    assert {k[0] for k in ka} == kinds
    if count == 8 and n == 2048:
        assert {k[1:] for k in ka} == {(7, 128, 4)}  # four elements per lane, half the blocks
    _same(a, b)


# pairs of several layouts and rods beside them, with more blocks than SMs; more pairs than clusters of 13 (16) blocks
@pytest.mark.parametrize("pair_lengths,lengths,blocks", [([512] * 6 + [700] * 6, [], 13), ([512] * 11, [], 8),
                                                         ([300] * 8 + [600] * 3, [512] * 4 + [2048] * 2, 8),
                                                         ([1024] * 8, [], 16), ([64, 200, 512, 1024], [3000, 40, 700], 2)])
def test_pairs(corde, pair_lengths, lengths, blocks):
    rods, pairs = [], []
    for k, n in enumerate(pair_lengths):
        pairs.append((len(rods), len(rods) + 1, k % 3))
        rods += list(W.catheter_guidewire(n, seed=k, beta0=-0.2 * n - 0.25))
    rods += [W.guidewire(n, seed=n) for n in lengths]
    a, ka = _run(corde, rods, pairs, True)
    b, kb = _run(corde, rods, pairs, False)
    assert ka[0][:2] == ("pair_tiles", blocks) and {k[0] for k in ka[:2 * len(pairs)]} == {"pair_tiles"}
    assert not {"pair_tiles", "tiles"} & {k[0] for k in kb}
    _same(a, b)
