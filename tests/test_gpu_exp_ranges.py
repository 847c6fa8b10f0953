"""The link update's exponential over the norms its branches divide: on unit
links with phi = pi = 0 every plaquette vanishes, so one field step multiplies
each link by exp(i dt/t_{n+1/2} e) of its own momentum.  The norms |dt/t e| run
over the FP64 series lengths (0.01, 0.25, 1, 2) and their scaling and squaring
beyond, and the FP32 series' limit (0.2) and its squarings."""
import numpy as np
import pytest

import oracle as O
from paper_2303_05599_gb300 import _binding as B
from paper_2303_05599_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("prec", [W.FP64, W.FP32_2ROW])
def test_link_update_over_the_norms(prec):
    N, n = 16, 8
    w = W.Workload("exp", N=N, L_fm=1.5, precision=prec, reunit_every=0, species=[])
    rng = np.random.default_rng(5)
    norm = np.geomspace(1e-3, 8.0, 2 * N * N).reshape(2, N * N)     # |X|_F of each link's exponent
    norm[0, :8] = [0.0099, 0.0101, 0.19, 0.21, 0.249, 0.251, 0.999, 1.001]
    x = rng.normal(size=(2, N * N, 8))
    x *= (norm * np.sqrt(2.0) / np.linalg.norm(x, axis=-1))[..., None]  # |X|_F^2 = x.x / 2
    th = (n + 0.5) * w.dt
    e = x * th / w.dt
    if prec == W.FP32_2ROW:
        e = e.astype(np.float32).astype(np.float64)
    st = O.FieldState(N, O.unit_links(N), np.zeros((N * N, 8)), e, np.zeros((N * N, 8)))
    ev = B.Event(w)
    for buf, a in ((B.GL_BUF_LINKS, st.U), (B.GL_BUF_PHI, st.phi), (B.GL_BUF_E, st.e), (B.GL_BUF_PI, st.pi)):
        ev.upload(buf, a)
    ev.set_step(n)
    ev.glasma_step(1)
    got = ev.download(B.GL_BUF_LINKS)
    want = O.field_step(st, n * w.dt, w.dt).U
    err = np.abs(got - want.reshape(got.shape)).max(-1)
    # the series' rounding is a few units in the last place of 1; each of the
    # log2(|X| / limit) squarings doubles it
    eps, limit = (2.0 ** -53, 2.0) if prec == W.FP64 else (2.0 ** -24, 0.2)
    bound = 32 * eps * np.maximum(1.0, 4 * norm / limit)
    assert (err <= bound).all(), (err / bound).max()
