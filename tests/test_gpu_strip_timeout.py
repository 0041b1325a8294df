"""A wait between strips that runs out: the status reaches the caller, the context stays usable, and setting the
lattice again (in stream order) clears it.  A lattice set under ISING_FAULT=wait gives the waits no time, so some give up
at once; nothing hangs and nothing is read out of range: the strips set the status and return."""
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


def _lattice(L, layout):
    return lambda: ising.Lattice(L, 0.44, layout, seed=3)


# four threads a word, one thread a word, edge words, both layouts; XY in both precisions; four sublattices; and
# the cluster steps' flag barrier with either forest
CASES = {
    "split": (_lattice(256, BITS), "sweep"),
    "split_i8": (_lattice(256, I8), "sweep"),
    "halo": (_lattice(768, BITS), "sweep"),
    "edge": (_lattice(1300, BITS), "sweep"),
    "edge_i8": (_lattice(1300, I8), "sweep"),
    "xy64": (lambda: ising.XY(128, 1.1, 64, seed=3), "sweep"),
    "xy32": (lambda: ising.XY(512, 1.1, 32, seed=3), "sweep"),
    "quad": (lambda: ising.Quad(ising.ISING_QUAD_SQOCT, 256, 0.44, 1.0, 1.0, seed=3), "sweep"),
    "sw_128": (_lattice(128, BITS), "sw_step"),
    "sw_512": (_lattice(512, BITS), "sw_step"),
    "wolff_256": (_lattice(256, BITS), "wolff_step"),
}


def _read(x):
    if hasattr(x, "measure"):
        return x.measure()
    return x.series(0), x.spins().sum()


def _hurry(x, monkeypatch):
    monkeypatch.setenv("ISING_FAULT", "wait")
    x.seed(4)
    monkeypatch.delenv("ISING_FAULT")


def _give_up(x, step, monkeypatch):
    _hurry(x, monkeypatch)
    getattr(x, step)(60)


def _times_out(x):
    with pytest.raises(ising.IsingError) as e:
        _read(x)
    return e.value.status == ising.ISING_ETIMEOUT


@pytest.mark.parametrize("case", sorted(CASES))
def test_reported_and_cleared_by_the_seed(case, monkeypatch):
    make, step = CASES[case]
    with make() as x, make() as ref:
        _give_up(x, step, monkeypatch)
        assert _times_out(x) and _times_out(x)  # until the lattice is set again
        for c in (x, ref):
            c.seed(5)
            getattr(c, step)(7)
        assert np.array_equal(x.spins(), ref.spins())


@pytest.mark.parametrize("case", sorted(CASES))
def test_cleared_by_setting_the_spins(case, monkeypatch):
    make, step = CASES[case]
    with make() as x, make() as ref:
        start = ref.spins()
        _give_up(x, step, monkeypatch)
        assert _times_out(x)
        x.set_spins(start)
        assert np.array_equal(x.spins(), start)


@pytest.mark.parametrize("case", ["split", "edge", "xy32", "quad"])
def test_a_seed_clears_what_is_still_queued(case, monkeypatch):
    """The call that gives up is still behind a long one on the stream when the host seeds its context again."""
    make, step = CASES[case]
    with make() as x, _lattice(256, BITS)() as other:  # both on the default stream
        _read(x), other.measure()
        _hurry(x, monkeypatch)
        _read(x)
        other.sweep(20000)
        getattr(x, step)(60)
        x.seed(5)
        _read(x)


def test_bits_and_device_forms_clear_it_too(monkeypatch):
    import torch

    with ising.Lattice(256, 0.44, BITS, seed=3, stream=torch.cuda.current_stream()) as x:
        words, spins = x.bits(), x.spins()
        dev_w = torch.from_numpy(words.view(np.int32)).cuda()
        dev_s = torch.from_numpy(spins).cuda()
        for put in (lambda: x.set_bits(words), lambda: ising.ising_set_bits_device(x.ctx, dev_w),
                    lambda: ising.ising_set_spins_device(x.ctx, dev_s)):
            _give_up(x, "sweep", monkeypatch)
            assert _times_out(x)
            put()
            assert np.array_equal(x.bits(), words)


def test_a_status_word_that_is_used_again_is_clear(monkeypatch):
    """The context has 1024 status words, one after the other for each lattice that is set."""
    with ising.Lattice(256, 0.44, BITS, seed=3) as x:
        _give_up(x, "sweep", monkeypatch)
        assert _times_out(x)
        for k in range(1024):
            x.seed(k)
        _read(x)
        x.sweep(20)
        _read(x)
