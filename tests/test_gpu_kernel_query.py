"""ising_get_kernel names the kernel that runs, and ising_set_kernel takes its answer back."""
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


def _launches(lat, n):
    lat.sweep(n)
    before = ising.ising_launch_count(lat.ctx)
    lat.sweep(n)
    return ising.ising_launch_count(lat.ctx) - before


# one strip, strips with a halo, strips that exchange edge words, and int8 spins
@pytest.mark.parametrize("L,layout", [(64, BITS), (64, I8), (256, BITS), (256, I8), (1000, BITS), (2048, BITS)])
def test_strips_are_named_and_kept(L, layout):
    with ising.Lattice(L, 0.44, layout, seed=1) as lat:
        k = lat.kernel()
        assert k["kernel"] == ising.ISING_KERNEL_STRIP and k["tile_rows"] >= 1
        assert _launches(lat, 12) == 1  # one launch a call: strips
        lat.set_kernel(**k)
        assert lat.kernel() == k and _launches(lat, 12) == 1
        lat.set_kernel(ising.ISING_KERNEL_HALF)
        assert lat.kernel()["kernel"] == ising.ISING_KERNEL_HALF and _launches(lat, 12) == 24
        lat.set_kernel(ising.ISING_KERNEL_AUTO)
        assert lat.kernel() == k


def test_other_kernels_are_named_as_before():
    with ising.Lattice(8192, 0.44, BITS, seed=1) as lat:
        k = lat.kernel()
        assert k["kernel"] == ising.ISING_KERNEL_TILED and k["sweeps_per_launch"] == 4 and k["tile_words"] == 32
        lat.set_kernel(**k)
        assert lat.kernel() == k
        lat.set_kernel(ising.ISING_KERNEL_STRIP)  # they fit, if not chosen
        assert lat.kernel()["kernel"] == ising.ISING_KERNEL_STRIP and _launches(lat, 8) == 1


def test_refused_buffers_leave_the_choice_as_it_was(monkeypatch):
    with ising.Lattice(8192, 0.44, BITS, seed=1) as lat:
        lat.set_kernel(ising.ISING_KERNEL_HALF)
        before = lat.kernel()
        monkeypatch.setenv("ISING_FAULT", "alloc")
        with pytest.raises(ising.IsingError) as e:
            lat.set_kernel(ising.ISING_KERNEL_STRIP)
        monkeypatch.delenv("ISING_FAULT")
        assert e.value.status == ising.ISING_ENOMEM and lat.kernel() == before and _launches(lat, 2) == 4


def test_strips_that_do_not_fit_are_refused():
    with ising.Lattice(16384, 0.44, BITS) as lat:
        before = lat.kernel()
        with pytest.raises(ising.IsingError) as e:
            lat.set_kernel(ising.ISING_KERNEL_STRIP)
        assert e.value.status == ising.ISING_EINVAL and lat.kernel() == before
