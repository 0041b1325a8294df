"""Resident strips (the automatic kernel of lattices up to a few thousand sites a side): bit for bit the
one-launch-per-half-sweep kernel, whose own parity with the CPU oracle test_gpu_sweep.py pins."""
import numpy as np
import pytest

import oracle
import paper_2402_06415_gb300 as ising

pytestmark = pytest.mark.gpu

BITS, I8 = ising.ISING_LAYOUT_BITS, ising.ISING_LAYOUT_I8


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ising.lib()


def _run(L, beta, layout, calls, kernel=None):
    with ising.Lattice(L, beta, layout, seed=40 + L) as lat:
        if kernel is not None:
            lat.set_kernel(kernel)
        n = 0
        for sweeps, every in calls:
            lat.sweep(sweeps, every)
            n += sweeps
        E, M = lat.series()
        return lat.spins(), E, M


# one CTA (L <= 64), strips of one to several words a row, full and ragged last words (L / 2 = 1, 31, 32, 33 ... mod 32),
# four threads and one thread per word, uneven strips; sweep counts below, at and above a group of sweeps
@pytest.mark.parametrize("L", [4, 6, 62, 64, 66, 94, 128, 130, 190, 258, 510, 512, 514, 1000, 1022, 1536, 2050])
@pytest.mark.parametrize("layout", [BITS, I8])
def test_strips_equal_half_sweeps(L, layout):
    calls = [(1, 1), (2, 0), (7, 3), (20, 1)]
    got = _run(L, 0.4406868, layout, calls)
    ref = _run(L, 0.4406868, BITS, calls, ising.ISING_KERNEL_HALF)
    for a, b in zip(got, ref):
        assert np.array_equal(a, b)


# strips without a halo: one word a thread and a loop over more, edge words that share a warp with inner ones, ragged last
# words, uneven strips, and calls of a single sweep (the first exchange only)
@pytest.mark.parametrize("L", [900, 1300, 2046, 2306, 3074])
@pytest.mark.parametrize("layout", [BITS, I8])
def test_edge_strips_equal_half_sweeps(L, layout):
    calls = [(1, 0), (1, 1), (3, 2), (10, 1)]
    got = _run(L, 0.4406868, layout, calls)
    ref = _run(L, 0.4406868, BITS, calls, ising.ISING_KERNEL_HALF)
    for a, b in zip(got, ref):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("L,beta", [(64, 0.9), (256, 0.05), (258, 0.6), (1026, 0.3)])
def test_strips_equal_oracle(L, beta):
    ref = oracle.init(L, 40 + L)
    E, M = oracle.sweep(ref, beta, 40 + L, 12)
    got = _run(L, beta, BITS, [(12, 1)])
    assert np.array_equal(got[0], ref) and np.array_equal(got[1], E) and np.array_equal(got[2], M)


# one CTA and strips, odd and even row lengths L / 2, one site per thread and loops; calls of one sweep, fewer half
# sweeps than an exchange group, and records at both ends of a call
@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("L", [2, 6, 8, 16, 32, 34, 62, 130, 256, 514])
def test_xy_strips_equal_half_sweeps(precision, L):
    out = []
    for mode in (0, 1):
        with ising.XY(L, 1.0 / 0.85, precision, seed=7 + L) as x:
            x.set_mode(mode)
            for n, every in [(1, 1), (2, 0), (5, 2), (12, 1)]:
                x.sweep(n, every)
            out.append((x.spins(), x.accepted(), x.series(15)))
    assert np.array_equal(out[0][0], out[1][0]) and out[0][1] == out[1][1]
    # the same terms (at most 1.5 L^2 of them, each within 4) in another order, in double
    for a, b in zip(out[0][2], out[1][2]):
        np.testing.assert_allclose(a, b, rtol=0, atol=6 * L * L * 1.2e-16 * (2 + np.log2(L * L)))


def test_xy_angles_of_quadrant_edges():
    """The double path takes the quadrant of an angle from its 24-bit word; at every word within two of a
    quadrant edge it must give the same integer as rounding the angle (the recipe the oracle follows)."""
    m = np.concatenate([(1 << 21) * k + np.arange(-2, 3) for k in range(1, 8)]).astype(np.int64)
    x = 6.283185307179586 * (m * 2.0 ** -24)
    assert np.array_equal(x, (6.283185307179586 / 16777216.0) * m)
    tie = (m & 0x3FFFFF) == 0x200000
    assert np.array_equal(np.rint(x * 0.6366197723675814)[~tie], ((m + (1 << 21)) >> 22)[~tie])


# sizes that take strips (and 40, which stays in one CTA), one and several words a row, ragged last words, all three
# numbers of distinct thresholds; calls of one sweep, groups without a record, and records at both ends of a group
@pytest.mark.parametrize("lattice,J1,J2", [(ising.ISING_QUAD_SQOCT, 1.0, 1.0), (ising.ISING_QUAD_SQOCT, 0.7, 1.9),
                                           (ising.ISING_QUAD_SQUARE, 1.0, 0.0), (ising.ISING_QUAD_SQUARE, 0.75, 1.25)])
@pytest.mark.parametrize("Lc", [40, 64, 97, 200, 257, 640])
def test_quad_strips_equal_oracle(lattice, J1, J2, Lc):
    seed = 90 + Lc
    s = oracle.quad_init(Lc, seed)
    with ising.Quad(lattice, Lc, 0.4406868, J1, J2, seed=seed) as x:
        for n, every in [(1, 1), (2, 0), (6, 4), (5, 1)]:
            x.sweep(n, every)
        got = x.spins()
        B1, B2, M = x.series(7)  # after sweeps 1; 4, 8; 10 ... 14 (the last seven: 4, 8, 10 ... 14)
    R1, R2, RM = oracle.quad_sweep(lattice, s, 0.4406868, J1, J2, seed, 14)
    assert np.array_equal(got, s)
    at = [3, 7, 9, 10, 11, 12, 13]
    assert np.array_equal(B1, R1[at]) and np.array_equal(B2, R2[at]) and np.array_equal(M, RM[at])


# a shared forest per CTA (L <= 160) and the global one, uneven strips of 2 to 10 rows, rows that are no multiple of a
# 64-site block; one step, records, and a hot, critical and cold lattice
@pytest.mark.parametrize("wolff", [False, True])
@pytest.mark.parametrize("L", [66, 158, 160, 162, 330, 446, 450, 766, 1030])
@pytest.mark.parametrize("beta", [0.2, 0.4406868, 1.5])
def test_cluster_strips_equal_kernels(wolff, L, beta):
    out = []
    for mode in (ising.ISING_CLUSTER_PERSISTENT, ising.ISING_CLUSTER_KERNELS):
        with ising.Lattice(L, beta, BITS, seed=3 + L) as lat:
            lat.cluster_set_mode(mode)
            step = lat.wolff_step if wolff else lat.sw_step
            for n, every in [(1, 1), (2, 0), (6, 2)]:
                step(n, every)
            lat.sweep(1)
            step(3, 1)
            out.append((lat.spins(), *lat.series(), lat.wolff_stats()["flipped"] if wolff else 0))
    for x, y in zip(*out):
        assert np.array_equal(x, y)
