"""Where a stream's SMs are too few for the strips' cooperative launch (ISING_FAULT=coop answers as the driver does), a
call goes on with the kernels that run where strips do not fit: same chain, no error."""
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


def _same(make, run, read, monkeypatch):
    out = []
    for refused in (False, True):
        if refused:
            monkeypatch.setenv("ISING_FAULT", "coop")
        with make() as x:
            monkeypatch.delenv("ISING_FAULT", raising=False)
            run(x)
            run(x)
            out.append(read(x))
    for a, b in zip(*out):
        assert np.array_equal(a, b)


# fallbacks: half sweeps, tiles (whose second buffer strips do without), one CTA (int8) and half sweeps (int8)
@pytest.mark.parametrize("L,layout", [(130, BITS), (256, BITS), (2048, BITS), (128, I8), (512, I8)])
def test_sweeps(L, layout, monkeypatch):
    def run(x):
        x.sweep(5, 2)

    _same(lambda: ising.Lattice(L, 0.44, layout, seed=3), run, lambda x: (x.spins(), *x.series()), monkeypatch)
    monkeypatch.setenv("ISING_FAULT", "coop")
    with ising.Lattice(L, 0.44, layout, seed=3) as x:
        run(x)
        assert x.kernel()["kernel"] != ising.ISING_KERNEL_STRIP


@pytest.mark.parametrize("mode", [ising.ISING_CLUSTER_AUTO, ising.ISING_CLUSTER_PERSISTENT])
@pytest.mark.parametrize("step,L", [("sw_step", 128), ("sw_step", 800), ("wolff_step", 256)])
def test_cluster_steps(step, L, mode, monkeypatch):
    def make():
        x = ising.Lattice(L, 0.44, BITS, seed=3)
        x.cluster_set_mode(mode)
        return x

    _same(make, lambda x: getattr(x, step)(4, 1), lambda x: (x.spins(), *x.series()), monkeypatch)


@pytest.mark.parametrize("precision,L", [(64, 64), (32, 256)])
def test_xy(precision, L, monkeypatch):
    _same(lambda: ising.XY(L, 1.1, precision, seed=3), lambda x: x.sweep(4, 0), lambda x: (x.spins(), x.accepted()),
          monkeypatch)


# fallbacks: one CTA up to 256, quarter launches above; ragged last words
@pytest.mark.parametrize("lattice,J2", [(ising.ISING_QUAD_SQOCT, 1.0), (ising.ISING_QUAD_SQUARE, 0.5),
                                        (ising.ISING_QUAD_SQUARE, 0.0)])
@pytest.mark.parametrize("Lc", [97, 300, 641])
def test_quad(lattice, J2, Lc, monkeypatch):
    _same(lambda: ising.Quad(lattice, Lc, 0.44, 1.0, J2, seed=3), lambda x: x.sweep(5, 2),
          lambda x: (x.spins(), *x.series(5)), monkeypatch)
