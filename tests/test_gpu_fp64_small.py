"""The FP64 field step on both sides of the size that takes the small tiles (a
quarter more large tiles than SMs): against the oracle, with ragged and wrapping tiles;
and batches that take the large tiles, bitwise as their events alone in the
small ones, and the reverse, on two streams and as one fused launch."""
import numpy as np
import pytest

import oracle as O
from paper_2303_05599_gb300 import _binding as B
from paper_2303_05599_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

BUFS = (B.GL_BUF_LINKS, B.GL_BUF_E, B.GL_BUF_PI, B.GL_BUF_PHI, B.GL_BUF_SITE, B.GL_BUF_PARTICLES)


def wl(N, seed=2):
    return W.Workload("small", N=N, L_fm=0.06 * N, Ns=2, precision=W.FP64, seed=seed, sort_every=3,
                      species=[W.Species(W.M_CHARM, 0.0, 60, W.REP_F, W.MOM_FIXED_PT, 0.5)])


def rel(a, b):
    return np.abs(np.asarray(a).ravel() - np.asarray(b).ravel()).max() / max(1e-300, np.abs(b).max())


@pytest.mark.parametrize("N", [4, 5, 7, 33, 128, 140, 160, 165])
def test_fields_against_the_oracle(N):
    w = wl(N)
    st, bad = O.mv_init(w.N, w.Ns, w.g2mu_a, w.m_a, w.Lambda_a, w.seed)
    assert bad == 0
    ev = B.Event(w)
    for buf, a in ((B.GL_BUF_LINKS, st.U), (B.GL_BUF_PHI, st.phi), (B.GL_BUF_E, st.e), (B.GL_BUF_PI, st.pi)):
        ev.upload(buf, a)
    ev.wong_init()
    ev.step(3)
    for n in range(3):
        old = st
        st = O.field_step(st, n * w.dt, w.dt)
    # a few hundred roundings of values of order 1 a step
    tol = 1e-13
    for buf, b in ((B.GL_BUF_LINKS, st.U), (B.GL_BUF_PHI, st.phi), (B.GL_BUF_E, st.e), (B.GL_BUF_PI, st.pi)):
        assert rel(ev.download(buf), b) < tol, buf
    assert rel(ev.download(B.GL_BUF_SITE), O.site_fields(old, st, 2 * w.dt)) < 10 * tol


@pytest.mark.parametrize("fused", [False, True])
@pytest.mark.parametrize("sizes", [[33, 132, 5, 64, 160, 128], [33, 5, 64, 16]])
def test_batches_of_both_kinds(sizes, fused):
    ws = [wl(N, e) for e, N in enumerate(sizes)]
    batch = B.Batch(ws)
    with torch.cuda.stream(batch.stream):
        batch.init()
        batch.set_launch("32x4", 128, 512, fused)
        batch.step(5)
        for w, be in zip(ws, batch.events):
            one = B.Event(w, stream=batch.stream)
            one.glasma_init()
            one.wong_init()
            one.step(5)
            for buf in BUFS:
                assert np.array_equal(be.download(buf), one.download(buf)), (w.N, buf)
