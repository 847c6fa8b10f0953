"""Initial conditions of two contexts from two host threads at once: the shared
memory that a launch may ask for belongs to the kernel and the device, so what
one call sets up must hold for the other's launches too."""
import threading

import pytest

from paper_2303_05599_gb300 import _binding as B
from paper_2303_05599_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_contexts_of_two_sizes_at_once():
    """Both take more shared memory than a launch gets by default, 50 and 64 KB."""
    barrier = threading.Barrier(2)
    errors = []

    def run(N):
        ev = B.Event(W.Workload("t", N=N, L_fm=0.02 * N, Ns=12, precision=W.FP32_2ROW, species=[]),
                     stream=torch.cuda.Stream())
        for _ in range(12):
            barrier.wait()
            try:
                ev.glasma_init()
            except B.GlasmaError as e:
                errors.append((N, str(e)))
        ev.close()

    threads = [threading.Thread(target=run, args=(N,)) for N in (800, 1024)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert errors == []
