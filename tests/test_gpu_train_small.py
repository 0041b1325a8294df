"""Tensor-core training on few windows: a CTA takes one window of one stage, and the gradients are the FP32 kernel's."""
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


def _windows(block, n):
    import torch

    rng = np.random.default_rng(block)
    return torch.from_numpy(np.where(rng.random((n, block + 2, block + 2)) < 0.5, 1, -1).astype(np.int8)).cuda()


def _trainer(block, proposal):
    return learned.Trainer(block, seed=1, proposal=proposal, precision=ising.ISING_NN_TRAIN_BF16_TC)


# fewer samples (window, stage) than SMs, about as many, and more; n a power of two, so that 1 / n is exact and BF16
# operands round alike however the windows are packed: only the order of the FP32 sums differs
@pytest.mark.parametrize("block", [2, 4, 8, 16])
@pytest.mark.parametrize("proposal", [ising.ISING_PROPOSAL_ONESHOT, ising.ISING_PROPOSAL_STAGED])
def test_gradients_are_the_mean_of_single_windows(block, proposal):
    w = _windows(block, 64)
    with _trainer(block, proposal) as tr:
        one = [ising.ising_nn_loss_grad(tr.h, w[k:k + 1].contiguous(), 1) for k in range(64)]
        for n in (1, 2, 8, 16, 32, 64):
            loss, g = ising.ising_nn_loss_grad(tr.h, w, n)
            assert abs(loss - np.mean([v for v, _ in one[:n]])) < 1e-5 * loss
            ref = ising.nn_unflatten(np.mean([v.astype(np.float64) for _, v in one[:n]], axis=0))
            size = ising.nn_unflatten(np.mean([np.abs(v) for _, v in one[:n]], axis=0))
            for k, v in ising.nn_unflatten(g).items():
                assert np.abs(v - ref[k]).max() <= 1e-4 * size[k].max(), (n, k)


def test_few_staged_windows_take_no_longer_than_one_shot_ones():
    """A staged sample has fewer positions than a one-shot sample, and with fewer samples than SMs each has an SM of its
    own (with as many CTAs as samples, some took samples of two stages and set up twice: 1.18 times as long)."""
    import time

    us = []
    for proposal in (ising.ISING_PROPOSAL_ONESHOT, ising.ISING_PROPOSAL_STAGED):
        with _trainer(8, proposal) as tr:
            w = _windows(8, 8)
            best = 1e30
            for _ in range(300):
                t0 = time.perf_counter()
                ising.ising_nn_loss_grad(tr.h, w, 8)
                best = min(best, time.perf_counter() - t0)
            us.append(best * 1e6)
    assert us[1] < 1.08 * us[0], us
