"""Two contexts on two streams: a long call of one does not hold up a short call of the other, and a call that is
split into several launches gives what one launch gave."""
import time

import numpy as np
import pytest

import paper_2402_06415_gb300 as ising

pytestmark = pytest.mark.gpu

BITS, I8 = ising.ISING_LAYOUT_BITS, ising.ISING_LAYOUT_I8


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ising.lib()


LONG = {  # each about 0.6 to 0.9 s of one context's work
    "one CTA": (lambda s: ising.Lattice(64, 0.44, I8, stream=s, seed=1), "sweep", 2_000_000),
    "halo": (lambda s: ising.Lattice(512, 0.44, BITS, stream=s, seed=1), "sweep", 600_000),
    "edge": (lambda s: ising.Lattice(2048, 0.44, BITS, stream=s, seed=1), "sweep", 300_000),
    "sw": (lambda s: ising.Lattice(512, 0.44, BITS, stream=s, seed=1), "sw_step", 30_000),
    "xy": (lambda s: ising.XY(32, 1.1, 64, stream=s, seed=1), "sweep", 200_000),
    "quad": (lambda s: ising.Quad(ising.ISING_QUAD_SQOCT, 512, 0.44, 1.0, 1.0, stream=s, seed=1), "sweep", 250_000),
}


@pytest.mark.parametrize("name", sorted(LONG))
def test_a_long_call_leaves_room(name):
    """A call is launched in pieces of about 20 ms, so the other context's strips start within a few of them."""
    import torch

    make, step, n = LONG[name]
    a = make(torch.cuda.Stream())
    with ising.Lattice(2048, 0.44, BITS, stream=torch.cuda.Stream(), seed=2) as b:
        getattr(a, step)(10)
        b.sweep(20)
        b.measure(), a.spins()
        t0 = time.perf_counter()
        getattr(a, step)(n)
        time.sleep(0.02)
        t1 = time.perf_counter()
        b.sweep(20)
        b.measure()
        waited = time.perf_counter() - t1
        a.spins()
        whole = time.perf_counter() - t0
        a.close()
    assert whole > 0.4  # the long call was still running
    assert waited < 0.2, (waited, whole)


def test_pieces_are_one_chain():
    """20003 sweeps of a 512 x 512 lattice with records (more than a launch takes): the oracle-checked half sweeps' chain."""
    out = []
    for kernel in (ising.ISING_KERNEL_AUTO, ising.ISING_KERNEL_HALF):
        with ising.Lattice(512, 0.44, BITS, seed=9) as x:
            x.set_kernel(kernel)
            x.sweep(20003, 7)
            assert ising.ising_launch_count(x.ctx) > 2
            out.append((x.spins(), *x.series()))
    for p, q in zip(*out):
        assert np.array_equal(p, q)


def test_pieces_of_xy_and_quad_are_one_chain():
    with ising.XY(32, 1.1, 64, seed=9) as x, ising.XY(32, 1.1, 64, seed=9) as y:
        x.sweep(20003, 7)
        for _ in range(7):
            y.sweep(2857, 7)
        y.sweep(4, 7)
        assert np.array_equal(x.spins(), y.spins()) and x.accepted() == y.accepted()
        assert x.series(2857)[0].shape == y.series(2857)[0].shape
    with ising.Quad(ising.ISING_QUAD_SQOCT, 128, 0.44, 1.0, 1.0, seed=9) as x, \
            ising.Quad(ising.ISING_QUAD_SQOCT, 128, 0.44, 1.0, 1.0, seed=9) as y:
        x.sweep(20003, 7)
        for _ in range(7):
            y.sweep(2857, 7)
        y.sweep(4, 7)
        assert np.array_equal(x.spins(), y.spins())
        for p, q in zip(x.series(2857), y.series(2857)):
            assert np.array_equal(p, q)
