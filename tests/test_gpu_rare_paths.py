"""Branches that ordinary runs reach rarely or not at all: a tile's full queue, the automatic tiles of large lattices, and
the exact half-integer quadrants of XY angles."""
import numpy as np
import pytest

import oracle
import paper_2402_06415_gb300 as ising

pytestmark = pytest.mark.gpu

BITS, HALF, TILED = ising.ISING_LAYOUT_BITS, ising.ISING_KERNEL_HALF, ising.ISING_KERNEL_TILED


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ising.lib()


def _chain(L, beta, kernel, calls):
    with ising.Lattice(L, beta, BITS, seed=11) as lat:
        if kernel:
            lat.set_kernel(*kernel)
        for n, every in calls:
            lat.sweep(n, every)
        return (lat.bits(), *lat.series())


# 512 rows x 32 words a tile: 16,000 words a half sweep, of which a cold lattice leaves 10 % undecided (lanes that do
# not flip outright, 28 of 32, are undecided with probability 2^-8), more than the queue's 1536
@pytest.mark.parametrize("k", [1, 2])
def test_tiles_with_a_full_queue(k):
    calls = [(12, 0), (5, 1)]
    for a, b in zip(_chain(2048, 1.2, (TILED, k, 4, 32), calls), _chain(2048, 1.2, (HALF,), calls)):
        assert np.array_equal(a, b)


# four sweeps a launch and calls that leave one to three, records at their ends
@pytest.mark.parametrize("L", [6144, 8192])
def test_automatic_tiles(L):
    calls = [(1, 1), (3, 2), (9, 3)]
    with ising.Lattice(L, 0.44, BITS) as lat:
        assert lat.kernel()["kernel"] == TILED
    for a, b in zip(_chain(L, 0.44, None, calls), _chain(L, 0.44, (HALF,), calls)):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("seed", [1, 8])
def test_xy_angles_on_quadrant_edges(seed):
    """Start angles of 4096 x 4096 spins, bit for bit the oracle's; among them are words whose angle is exactly half way
    between two quadrants (m = 2^21 + k 2^22), in all four places, where the integer quadrant is not used."""
    ref = oracle.xy_init(4096, seed)
    c, s = ref[..., 0], ref[..., 1]
    tie = np.abs(np.abs(c) - np.abs(s)) < 1e-9
    assert len(set(zip(np.sign(c[tie]), np.sign(s[tie])))) == 4
    with ising.XY(4096, 1.0, 64, seed=seed) as x:
        assert np.array_equal(x.spins(), ref)
