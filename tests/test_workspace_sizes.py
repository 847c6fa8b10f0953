"""The device memory a context asks for beside its state: the initial conditions
take no more scratch than 576 bytes a site, or 4 MB on a small lattice."""
import pytest

from paper_2303_05599_gb300 import _binding as B
from paper_2303_05599_gb300 import workloads as W


def up(n):
    return (n + 255) // 256 * 256


@pytest.mark.parametrize("prec", [W.FP64, W.FP32_2ROW])
@pytest.mark.parametrize("Ns", [1, 10, 50, 400])
@pytest.mark.parametrize("N", [4, 5, 8, 16, 32, 45, 64, 86, 90, 128, 200, 256, 500, 512, 1024, 2048, 3072])
def test_scratch_of_the_initial_conditions(N, Ns, prec):
    V = N * N
    w = W.Workload("size", N=N, L_fm=0.04 * N, Ns=Ns, precision=prec, species=[])
    fields, site = (544 * V, 384 * V) if prec == W.FP64 else (224 * V, 192 * V)
    rows = B.GL_MAX_SPECIES * 7 + 7  # values of the observables' rows
    state = 2 * up(fields) + 2 * up(site) + up(1024 * rows * 8) + up(rows * 8) + 256
    assert B.gl_workspace_bytes(w) - state <= up(max(576 * V, 4 << 20))
