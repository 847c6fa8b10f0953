"""The length of a charge over many rapidity rotations: the truncated series of
the FP32 push is not orthogonal, so what it adds to |Q|^2 has one sign."""
import numpy as np
import pytest

from paper_2303_05599_gb300 import _binding as B
from paper_2303_05599_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

STEPS = 300


# below the limits of one to five terms, and between them
@pytest.mark.parametrize("angle", [3.0e-5, 2.3e-4, 5.5e-3, 1.0e-2, 2.8e-2, 6.2e-2, 7.9e-2])
def test_mean_length_is_kept(angle):
    N, n = 32, 8
    w = W.Workload("length", N=N, L_fm=1.5, precision=W.FP32_2ROW, reunit_every=0, sort_every=0,
                   species=[W.Species(0.0, 0.0, N * N, W.REP_F, W.MOM_FIXED_PT, 0.5)])
    rng = np.random.default_rng(5)
    phi = rng.normal(size=(N * N, 8))
    phi *= angle * n / np.linalg.norm(phi, axis=1)[:, None]  # angle dt / t v_w |phi|, dt / t = 1 / n, v_w = 1
    links = np.zeros((2, N * N, 18))
    links[:, :, [0, 8, 16]] = 1.0
    zero = np.zeros((N * N, 8))
    ev = B.Event(w)
    ev.glasma_init()
    ev.wong_init()
    part = ev.download(B.GL_BUF_PARTICLES)
    part[:, 0], part[:, 1] = np.arange(N * N) % N, np.arange(N * N) // N
    part[:, 2:5], part[:, 5] = 0.0, 1e4  # at rest on their cells, moving in rapidity
    ev.upload(B.GL_BUF_PARTICLES, part)

    def length():
        return (ev.download(B.GL_BUF_PARTICLES)[:, 6:14] ** 2).sum(1)

    start = length()
    for _ in range(STEPS):
        for buf, a in ((B.GL_BUF_LINKS, links), (B.GL_BUF_PHI, phi), (B.GL_BUF_E, np.stack([zero, zero])),
                       (B.GL_BUF_PI, zero)):
            ev.upload(buf, a)
        ev.set_step(n)
        ev.step(1)
    # an eighth of a unit in the last place of |Q|^2 = 4 a step; the roundings of
    # 1024 charges, turned about as many axes, average out well below it
    assert abs((length() - start).mean()) < STEPS * 4.0 * 2.0 ** -27
