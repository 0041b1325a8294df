"""Batches of replicas above 128 x 128: results against the oracle, and the work decomposition's speed."""
import numpy as np
import pytest

import oracle
import paper_2402_06415_gb300 as ising

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ising.lib()


def _ms(b, n, reps=5):
    """Best time of b.run(n) in ms."""
    import torch

    b.run(n)
    best = 1e30
    for _ in range(reps):
        torch.cuda.synchronize()
        e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        e0.record()
        b.run(n)
        e1.record()
        e1.synchronize()
        best = min(best, e0.elapsed_time(e1))
    return best


def _batch(L, n_rep, kernel=None, betas=None):
    import torch

    b = ising.Batch([L] * n_rep, betas if betas is not None else [0.44], 10, stream=torch.cuda.current_stream(),
                    seed=5)
    if kernel:
        ising.ising_batch_set_kernel(b.h, *kernel)
    return b


# one replica an item, more undecided words per half sweep than the queue takes, several passes of the queue with a
# ragged last one (640: 3200 pairs, 1024: 8192), rows of a ragged last word (514), and a cold lattice, where nearly
# every word draws in all its lanes and a single pass overfills the queue now and then
@pytest.mark.parametrize("L", [514, 640, 1024])
@pytest.mark.parametrize("threads", [32, 256])
def test_large_replicas_bit_exact(L, threads):
    betas, seed, n, pt = [0.40, 1.2], 21, 7, 3
    ref = oracle.run_ladders([L], betas, seed, n, pt)
    with ising.Batch([L], betas, pt) as b:
        ising.ising_batch_set_kernel(b.h, 512, threads)
        ising.ising_batch_seed(b.h, seed)
        b.run(n)
        assert ising.ising_batch_status(b.h) == (0, n)
        p, E, M = b.state()
        assert np.array_equal(p[0], ref[1][0]) and np.array_equal(E[0], ref[2][0]) and np.array_equal(M[0], ref[3][0])
        for i in range(2):
            assert np.array_equal(b.spins(0, i), ref[0][0][i])


def test_cold_replicas_cost_no_more_than_the_words_they_queue():
    """A half sweep of a cold 1024 x 1024 replica queues 12 % of its words, of a hot one 4 %, each for one to two Philox
    blocks after the two that every word draws: at most 1.15 times the time.  Far above it where the queue fills up and
    lanes finish words alone."""
    ms = []
    for beta in (0.02, 1.2):
        with _batch(1024, 64, (512, 256), [beta]) as b:
            b.run(200)  # domains
            ms.append(_ms(b, 120) - _ms(b, 20))
    assert ms[1] < 1.25 * ms[0], ms


# one replica an SM, three, a few items more than CTAs of either size, uneven replicas
@pytest.mark.parametrize("Ls", [[256] * 64, [512] * 64, [1024] * 64, [256] * 456, [64] * 8192, [96] * 1024, [64, 512] * 16,
                                [16, 32, 64, 128, 256] * 64])
def test_default_decomposition_loses_to_no_other(Ls):
    """The automatic decomposition is within 15 % of every one it chooses from (a fixed 128 threads a CTA took 1.2 to
    1.6 times as long on replicas above 128 x 128)."""
    import torch

    with ising.Batch(Ls, [0.44], 10, stream=torch.cuda.current_stream(), seed=5) as b:
        auto = _ms(b, 20)
        other = {}
        for words in (256, 512):
            for threads in (128, 256):
                ising.ising_batch_set_kernel(b.h, words, threads)
                other[words, threads] = _ms(b, 20)
    assert auto < 1.15 * min(other.values()), (auto, other)


def test_a_small_batch_does_not_take_a_large_one_its_shared_memory():
    with _batch(1024, 2) as large:
        large.run(1)
        with _batch(16, 2) as small:
            small.run(1)
            large.run(1)
            assert ising.ising_batch_status(large.h) == (0, 2) and ising.ising_batch_status(small.h) == (0, 1)


def test_of_equal_plans_the_one_with_fewer_items():
    """64 ladders of 64 replicas of 16 .. 128 squared: items of 512 words are one for a CTA, those of 256 up to two (5 % slower)."""
    from paper_2402_06415_gb300 import workloads

    with ising.Batch(workloads.batch_ladder_sizes(64, 6), workloads.batch_betas(64), workloads.BATCH_PT_EVERY) as b:
        info = ising.ising_batch_info(b.h)
        assert info["items"] == info["grid"]
