"""Tensor-core training on many windows: the sums over a call's windows are no less exact than the mean of calls on parts of them."""
import numpy as np
import pytest

import paper_2402_06415_gb300 as ising
from paper_2402_06415_gb300 import learned

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ising.lib()


def test_sums_over_16384_windows_are_rounded_and_not_cut():
    """n is a power of two, so every product has the same BF16 operands as in calls on 512 windows and only sums differ.  A
    thread's sum of dW1 and db1 takes about 600 additions (16384 windows x 1196 rows / (152 CTAs x 16 warps x 16 rows)): rounded
    ones leave at most 2^-24 sqrt(600) = 1.5e-6 of it, cut ones up to 2^-24 600 / 2 = 1.8e-5 to one side."""
    import torch

    n, part = 16384, 512
    rng = np.random.default_rng(7)
    f = np.fft.ifft2(np.fft.fft2(rng.standard_normal((512, 512))) / (1.0 + np.hypot(*np.meshgrid(*[
        np.abs(np.fft.fftfreq(512, 1 / 512))] * 2)))).real  # clusters of all sizes
    w = torch.from_numpy(learned.extract_windows(np.where(f > 0, 1, -1).astype(np.int8), n, 16, rng)).cuda()
    with learned.Trainer(16, seed=3, proposal=ising.ISING_PROPOSAL_STAGED, precision=ising.ISING_NN_TRAIN_BF16_TC) as tr:
        ref = np.mean([ising.ising_nn_loss_grad(tr.h, w[k:k + part].contiguous(), part)[1].astype(np.float64)
                       for k in range(0, n, part)], axis=0)
        got = ising.nn_unflatten(ising.ising_nn_loss_grad(tr.h, w, n)[1])
    ref = ising.nn_unflatten(ref)
    for k in ("W1", "b1"):
        d = got[k].astype(np.float64) - ref[k]
        assert np.sqrt((d ** 2).mean() / (ref[k] ** 2).mean()) < 2e-6, k
