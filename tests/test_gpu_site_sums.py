"""The sums of squares of the site fields of an FP32 state against exact sums:
beyond the range of FP32, and over lattices on which a thread has many sites."""
import numpy as np
import pytest

from paper_2303_05599_gb300 import _binding as B
from paper_2303_05599_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def event(N, scale, precision=W.FP32_2ROW):
    w = W.Workload("sums", N=N, L_fm=0.04 * N, Ns=1, precision=precision,
                   species=[W.Species(W.M_CHARM, 0.0, 64, W.REP_F, W.MOM_FIXED_PT, 0.5)])
    ev = B.Event(w)
    ev.glasma_init()
    ev.wong_init()
    ev.upload(B.GL_BUF_PI, scale)
    ev.step(1)
    return ev


@pytest.mark.parametrize("N", [32, 300])
def test_sums_beyond_fp32(N):
    """A square of 1e36 fits FP32, the sum of a few hundred does not."""
    ev = event(N, np.full((N * N, 8), 1e18))
    s = ev.download(B.GL_BUF_SITE)[2].astype(np.longdouble)
    want = float(0.5 * (s * s).sum() / (N * N))
    assert ev.observables(B.GL_OBS_FIELDS).mean_trE_L2 == pytest.approx(want, rel=1e-12)


@pytest.mark.parametrize("precision", [W.FP32_2ROW, W.FP64])
@pytest.mark.parametrize("N", [24, 256, 512])
def test_sums_of_uneven_fields(N, precision):
    rng = np.random.default_rng(N)
    ev = event(N, rng.standard_normal((N * N, 8)) * 10.0 ** rng.uniform(-6, 2, size=(N * N, 1)), precision)
    s = ev.download(B.GL_BUF_SITE).astype(np.longdouble)
    h = 0.5 * (s * s).sum((1, 2)) / (N * N)
    o = ev.observables(B.GL_OBS_FIELDS)
    # FP32: a site's 16 squares as pairs, 2^-48 for each addition, halved on
    # average over a sum that grows; then FP64 sums: up to eight sites a thread, 8
    # threads and three levels of a block, 16 rows a lane and five levels.  FP64: a
    # thread's 128 squares in one chain, then the same
    tol = 8 * 2.0 ** -48 + 64 * 2.0 ** -53 if precision == W.FP32_2ROW else 192 * 2.0 ** -53
    for got, want in ((o.mean_trE_T2, h[0] + h[1]), (o.mean_trE_L2, h[2]), (o.mean_trB_T2, h[3] + h[4]),
                      (o.mean_trB_L2, h[5])):
        assert abs(got - float(want)) <= tol * float(want)
