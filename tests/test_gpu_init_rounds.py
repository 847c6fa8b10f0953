"""FP32 initial conditions whose sheets take several rounds, the last one partial,
on lattices with one and with several groups of sheets; events of a batch that
finish in different rounds; and a context that starts again in the middle of a
run, whichever of its field slices is current."""
import numpy as np
import pytest

import oracle as O
from paper_2303_05599_gb300 import _binding as B
from paper_2303_05599_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

STATE = (B.GL_BUF_LINKS, B.GL_BUF_PI, B.GL_BUF_PHI, B.GL_BUF_E, B.GL_BUF_PARTICLES)


def wl(N, Ns, prec=W.FP32_2ROW, seed=9):
    return W.Workload("rounds", N=N, L_fm=0.05 * N, Ns=Ns, precision=prec, seed=seed,
                      species=[W.Species(W.M_CHARM, 0.0, 50, W.REP_F, W.MOM_FIXED_PT, 0.5)])


@pytest.mark.parametrize("N,Ns", [(32, 50), (48, 47), (64, 50), (90, 33), (100, 20), (128, 40)])
def test_fields_against_the_oracle(N, Ns):
    w = wl(N, Ns)
    ev = B.Event(w)
    ev.glasma_init()
    st, bad = O.mv_init(w.N, w.Ns, w.g2mu_a, w.m_a, w.Lambda_a, w.seed)
    assert bad == 0
    U, pi = ev.download(B.GL_BUF_LINKS)[:, :, :12], ev.download(B.GL_BUF_PI)
    # the rounding of the stored entries beside 48-bit lines
    assert np.abs(U - st.U.reshape(2, N * N, 18)[:, :, :12]).max() < 2.0 ** -25 + 1e-10
    assert (np.abs(pi - st.pi.reshape(pi.shape)) <= np.abs(st.pi.reshape(pi.shape)) * 2.0 ** -24 + 1e-10).all()


@pytest.mark.parametrize("prec", [W.FP32_2ROW, W.FP64])
def test_batch_of_uneven_rounds_equals_single_events(prec):
    ws = [wl(N, Ns, prec, seed=40 + e)
          for e, (N, Ns) in enumerate([(128, 40), (16, 50), (64, 50), (90, 33), (32, 2), (32, 50), (128, 1)])]
    batch = B.Batch(ws)
    with torch.cuda.stream(batch.stream):
        batch.init()
        for w, be in zip(ws, batch.events):
            one = B.Event(w, stream=batch.stream)
            one.glasma_init()
            one.wong_init()
            for buf in STATE:
                assert np.array_equal(be.download(buf), one.download(buf)), (w.N, w.Ns, buf)


@pytest.mark.parametrize("prec", [W.FP32_2ROW, W.FP64])
@pytest.mark.parametrize("steps", [1, 2])
def test_a_second_start_is_the_first(prec, steps):
    w = wl(64, 30, prec)
    ev = B.Event(w)
    first = []
    for _ in range(2):
        ev.glasma_init()
        ev.wong_init()
        with pytest.raises(B.GlasmaError) as err:
            ev.download(B.GL_BUF_SITE)
        assert err.value.status == B.GL_ERR_STATE
        got = [ev.download(b) for b in STATE]
        ev.step(steps)
        got += [ev.download(b) for b in STATE + (B.GL_BUF_SITE,)]
        first = first or got
    assert all(np.array_equal(a, b) for a, b in zip(first, got))
