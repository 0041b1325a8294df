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


@pytest.mark.parametrize("L,beta", [(64, 0.9), (256, 0.05), (258, 0.6), (1026, 0.3)])
def test_strips_equal_oracle(L, beta):
    ref = oracle.init(L, 40 + L)
    E, M = oracle.sweep(ref, beta, 40 + L, 12)
    got = _run(L, beta, BITS, [(12, 1)])
    assert np.array_equal(got[0], ref) and np.array_equal(got[1], E) and np.array_equal(got[2], M)
