"""Threads that each run lattices of their own: the first calls of a process at the same time, small and large shared-memory
needs of one kernel side by side."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = """
import threading
import numpy as np, torch
import paper_2402_06415_gb300 as ising

BITS, I8, OCT = ising.ISING_LAYOUT_BITS, ising.ISING_LAYOUT_I8, ising.ISING_QUAD_SQOCT
sizes = [(lambda s, L=L: ising.Lattice(L, 0.44, BITS, stream=s, seed=3), "sweep") for L in (128, 512, 1300, 4000)]
sizes += [(lambda s, L=L: ising.Lattice(L, 0.44, I8, stream=s, seed=3), "sweep") for L in (32, 1300, 2600)]
sizes += [(lambda s, L=L: ising.Lattice(L, 0.44, BITS, stream=s, seed=3), "sw_step") for L in (200, 1500)]
sizes += [(lambda s, L=L: ising.XY(L, 1.1, 32, stream=s, seed=3), "sweep") for L in (128, 1024)]
sizes += [(lambda s, L=L: ising.Quad(OCT, L, 0.44, 1.0, 1.0, stream=s, seed=3), "sweep") for L in (128, 3000)]

def chain(make, step, stream):
    with make(stream) as x:
        getattr(x, step)(5)
        return x.spins()

got = [None] * len(sizes)
start = threading.Barrier(len(sizes))

def work(k):
    make, step = sizes[k]
    torch.cuda.set_device(0)
    stream = torch.cuda.Stream()
    start.wait()
    got[k] = chain(make, step, stream)

threads = [threading.Thread(target=work, args=(k,)) for k in range(len(sizes))]
for t in threads: t.start()
for t in threads: t.join()
for k, (make, step) in enumerate(sizes):
    assert got[k] is not None and np.array_equal(got[k], chain(make, step, torch.cuda.current_stream())), k

# a batch of small replicas made by another thread while one of large replicas runs
large = ising.Batch([1024, 1024], [0.44], 10, stream=torch.cuda.current_stream(), seed=5)
def small():
    for _ in range(20):
        with ising.Batch([16, 16], [0.44], 10, stream=torch.cuda.Stream(), seed=5) as b:
            b.run(1)
t = threading.Thread(target=small)
t.start()
for _ in range(20):
    large.run(1)
t.join()
assert ising.ising_batch_status(large.h) == (0, 20)
print("threads ok")
"""


def test_first_calls_from_several_threads():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    r = subprocess.run([sys.executable, "-c", CODE], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "threads ok" in r.stdout, r.stdout + r.stderr
