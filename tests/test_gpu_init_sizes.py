"""MV initial conditions over the line transforms and the work split: powers of
two with an even and an odd number of factors, composite and prime sizes,
lattices whose sheets are multiplied in groups and ones that take several
rounds; and uneven events started together against the same events alone."""
import numpy as np
import pytest

import oracle as O
from paper_2303_05599_gb300 import _binding as B
from paper_2303_05599_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def wl(N, Ns, prec=W.FP64, seed=9):
    return W.Workload("init", N=N, L_fm=0.05 * N, Ns=Ns, precision=prec, seed=seed,
                      species=[W.Species(W.M_CHARM, 0.0, 50, W.REP_F, W.MOM_FIXED_PT, 0.5)])


# (128, 16) takes several rounds of sheets; an FP32 event below 128 sites a side
# takes one and multiplies groups of sheets apart
@pytest.mark.parametrize("N,Ns", [(4, 3), (5, 1), (8, 50), (12, 7), (32, 50), (45, 4), (53, 2), (64, 6), (90, 2),
                                  (128, 16)])
def test_initial_fields_against_the_oracle(N, Ns):
    w = wl(N, Ns)
    ev = B.Event(w)
    ev.glasma_init()
    st, bad = O.mv_init(w.N, w.Ns, w.g2mu_a, w.m_a, w.Lambda_a, w.seed)
    assert bad == 0
    U, pi = ev.download(B.GL_BUF_LINKS), ev.download(B.GL_BUF_PI)
    # a few hundred roundings of values of order 1 a link, amplified by at most
    # the norm of the inverse Jacobian (order 10)
    assert np.abs(U - st.U.reshape(U.shape)).max() < 1e-11
    assert np.abs(pi - st.pi.reshape(pi.shape)).max() < 1e-11 * max(1.0, np.abs(st.pi).max())
    assert ev.observables().unitarity_max < 1e-13


@pytest.mark.parametrize("N,Ns", [(4, 3), (32, 50), (45, 4), (53, 2), (64, 6), (128, 16)])
def test_fp32_initial_fields_are_the_rounded_fp64_ones(N, Ns):
    """An FP32 event's sheets run on pairs of FP32 values (48 bits), so that
    its links and E_eta(0) are off by the rounding of their storage alone:
    half a unit in the last place of an entry below 1 is 2^-25."""
    w = wl(N, Ns, W.FP32_2ROW)
    ev = B.Event(w)
    ev.glasma_init()
    st, bad = O.mv_init(w.N, w.Ns, w.g2mu_a, w.m_a, w.Lambda_a, w.seed)
    assert bad == 0
    U, pi = ev.download(B.GL_BUF_LINKS)[:, :, :12], ev.download(B.GL_BUF_PI)
    assert np.abs(U - st.U.reshape(2, N * N, 18)[:, :, :12]).max() < 2.0 ** -25 + 1e-10
    assert (np.abs(pi - st.pi.reshape(pi.shape)) <= np.abs(st.pi.reshape(pi.shape)) * 2.0 ** -24 + 1e-10).all()


@pytest.mark.parametrize("prec", [W.FP64, W.FP32_2ROW])
def test_batch_init_equals_single_events(prec):
    ws = [wl(N, Ns, prec, seed=20 + e) for e, (N, Ns) in enumerate([(64, 3), (16, 5), (37, 2), (128, 16), (8, 1)])]
    batch = B.Batch(ws)
    with torch.cuda.stream(batch.stream):
        batch.init()
        for w, be in zip(ws, batch.events):
            one = B.Event(w, stream=batch.stream)
            one.glasma_init()
            one.wong_init()
            for buf in (B.GL_BUF_LINKS, B.GL_BUF_PI, B.GL_BUF_PHI, B.GL_BUF_E, B.GL_BUF_PARTICLES):
                assert np.array_equal(be.download(buf), one.download(buf)), (w.N, buf)


def test_init_beyond_the_longest_line_is_an_error():
    """N = 4096 was never within the transforms' shared memory."""
    w = W.Workload("big", N=4096, L_fm=10.0, Ns=1, precision=W.FP32_2ROW, species=[])
    ev = B.Event(w)
    with pytest.raises(B.GlasmaError) as err:
        ev.glasma_init()
    assert err.value.status == B.GL_ERR_CUDA


@pytest.mark.parametrize("N,Ns,value", [(8, 50, "0x1.94a390714d34ap-47"), (33, 1, "0x1.6ea1164352606p-48"),
                                        (64, 6, "0x1.63c18e857b809p-47")])
def test_fp64_links_keep_their_roundings(N, Ns, value):
    """The unitarity a check reports for an FP64 event right after its initial
    conditions is the sum of their roundings, so it is the same number as long
    as the order of the operations is."""
    ev = B.Event(wl(N, Ns))
    ev.glasma_init()
    assert ev.observables(B.GL_OBS_FIELDS).unitarity_max.hex() == value
