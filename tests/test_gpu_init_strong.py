"""Link matching in strong fields on coarse lattices (g^2 mu a of order 1), where
a few links take many damped Newton steps: an FP32 event accepts what an FP64
event accepts and finds the same solutions."""
import numpy as np
import pytest

import oracle as O
from paper_2303_05599_gb300 import _binding as B
from paper_2303_05599_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("N,Ns,a,g2mu,seed", [(32, 10, 0.09, 3.5, 1), (48, 3, 0.2, 2.0, 8), (24, 5, 0.15, 3.0, 8),
                                             (24, 5, 0.15, 3.0, 11)])
def test_fp32_links_of_a_strong_field(N, Ns, a, g2mu, seed):
    w = W.Workload("strong", N=N, L_fm=a * N, Ns=Ns, precision=W.FP32_2ROW, seed=seed, g2mu_GeV=g2mu, species=[])
    st, bad = O.mv_init(w.N, w.Ns, w.g2mu_a, w.m_a, w.Lambda_a, w.seed)
    assert bad == 0
    ev = B.Event(w)
    ev.glasma_init()
    U = ev.download(B.GL_BUF_LINKS)[:, :, :12]
    # the rounding of the stored entries, and 48-bit lines through as many steps
    assert np.abs(U - st.U.reshape(2, w.N * w.N, 18)[:, :, :12]).max() < 2.0 ** -25 + 1e-8


@pytest.mark.parametrize("precision", [W.FP64, W.FP32_2ROW])
@pytest.mark.parametrize("g2mu", [1e6, 1e20, 1e37, 1e160, 1e300])
def test_charges_beyond_any_range_end(g2mu, precision):
    """Infinite and undefined residuals end the matching, with an error or with
    fields that are not finite; the context is usable afterwards."""
    w = W.Workload("huge", N=8, L_fm=0.4, Ns=2, precision=precision, seed=1, g2mu_GeV=g2mu, species=[])
    ev = B.Event(w)
    try:
        ev.glasma_init()
    except B.GlasmaError as err:
        assert err.status == B.GL_ERR_NUMERIC
    assert ev.download(B.GL_BUF_LINKS).shape == (2, 64, 18)
