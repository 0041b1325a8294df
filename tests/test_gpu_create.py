"""Creating a context: no more for strips than for other kernels, and status words that contexts do not share."""
import time

import numpy as np
import pytest

import paper_2402_06415_gb300 as ising

pytestmark = pytest.mark.gpu

BITS, I8, OCT = ising.ISING_LAYOUT_BITS, ising.ISING_LAYOUT_I8, ising.ISING_QUAD_SQOCT


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ising.lib()


def _us(make):
    import torch

    best = 1e30
    for _ in range(25):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        make().close()
        best = min(best, time.perf_counter() - t0)
    return best * 1e6


# without strips: one CTA; with them, a status block and an exchange buffer (allocated one by one: three times as long)
@pytest.mark.parametrize("plain,strips", [
    (lambda: ising.Lattice(64, 0.44, BITS, seed=1), lambda: ising.Lattice(256, 0.44, BITS, seed=1)),
    (lambda: ising.Lattice(64, 0.44, I8, seed=1), lambda: ising.Lattice(512, 0.44, I8, seed=1)),
    (lambda: ising.XY(16, 1.1, 32, seed=1), lambda: ising.XY(128, 1.1, 32, seed=1)),
    (lambda: ising.Quad(OCT, 48, 0.44, 1.0, 1.0, seed=1), lambda: ising.Quad(OCT, 400, 0.44, 1.0, 1.0, seed=1)),
])
def test_strips_cost_no_more_to_create(plain, strips):
    a, b = _us(plain), _us(strips)
    assert b < 1.6 * a, (a, b)


def test_status_words_of_many_contexts(monkeypatch):
    """More contexts than a slab has blocks: a wait that gave up in some is reported by those alone, and a block that is
    given back and taken again is clear."""
    xs = [ising.Lattice(256, 0.44, BITS, seed=3) for _ in range(70)]
    bad = set(range(0, 70, 9))
    monkeypatch.setenv("ISING_FAULT", "wait")
    for k in bad:
        xs[k].seed(4)
    monkeypatch.delenv("ISING_FAULT")
    for x in xs:
        x.sweep(60)
    for k, x in enumerate(xs):
        if k in bad:
            with pytest.raises(ising.IsingError) as e:
                x.measure()
            assert e.value.status == ising.ISING_ETIMEOUT
        else:
            x.measure()
    for x in xs:
        x.close()
    again = [ising.Lattice(256, 0.44, BITS, seed=3) for _ in range(70)]
    ref = None
    for x in again:
        x.sweep(20)
        s = x.spins()
        ref = s if ref is None else ref
        assert np.array_equal(s, ref)
        x.close()


# lattice, records, status and exchange buffer lie in one allocation: each is where the others are not
@pytest.mark.parametrize("L,layout", [(4, BITS), (6, I8), (66, BITS), (1000, I8), (1300, BITS), (6144, BITS)])
def test_buffers_do_not_overlap(L, layout):
    with ising.Lattice(L, 0.44, layout, seed=7) as x, ising.Lattice(L, 0.44, layout, seed=7) as ref:
        ref.set_kernel(ising.ISING_KERNEL_HALF)
        for c in (x, ref):
            c.sweep(7, 1)
        assert x.measure() == ref.measure()
        for a, b in zip(x.series(), ref.series()):
            assert np.array_equal(a, b)
        assert np.array_equal(x.spins(), ref.spins())


def test_strips_asked_for_later_have_a_buffer_of_their_own():
    with ising.Lattice(6144, 0.44, BITS, seed=7) as x, ising.Lattice(6144, 0.44, BITS, seed=7) as ref:
        x.set_kernel(ising.ISING_KERNEL_STRIP)
        for c in (x, ref):
            c.sweep(3, 1)
        x.set_kernel(ising.ISING_KERNEL_AUTO)
        for c in (x, ref):
            c.sweep(3, 1)
        assert np.array_equal(x.bits(), ref.bits())
