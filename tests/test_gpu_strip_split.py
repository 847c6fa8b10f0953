"""The split of the FP32 strips: the same events alone (short segments in
4-warp blocks on as many SMs as there are) and in a batch that fills the chip
(the launch shape's own blocks) evolve bitwise alike, and a segment length set
between two steps takes effect in the next one without changing anything."""
import numpy as np
import pytest

from paper_2303_05599_gb300 import _binding as B
from paper_2303_05599_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

BUFS = (B.GL_BUF_LINKS, B.GL_BUF_E, B.GL_BUF_PI, B.GL_BUF_PHI, B.GL_BUF_SITE, B.GL_BUF_PARTICLES)


def wl(N, seed):
    return W.Workload("split", N=N, L_fm=0.04 * N, Ns=1, precision=W.FP32_2ROW, reunit_every=3, sort_every=4,
                      seed=seed, species=[W.Species(W.M_CHARM, 0.0, 500, W.REP_F, W.MOM_FIXED_PT, 0.5)])


def test_alone_and_in_a_full_batch():
    ws = [wl(N, e) for e, N in enumerate([31, 64, 200, 256] + [512] * 8)]
    batch = B.Batch(ws)
    with torch.cuda.stream(batch.stream):
        batch.init()
        batch.set_launch("strip12", 128, 256)
        batch.step(5)
        for e in range(5):
            one = B.Event(ws[e], stream=batch.stream)
            one.glasma_init()
            one.wong_init()
            one.step(5)
            for buf in BUFS:
                assert np.array_equal(batch.events[e].download(buf), one.download(buf)), (ws[e].N, buf)


def test_segment_length_set_between_steps():
    ws = [wl(N, e) for e, N in enumerate([40, 64, 100])]
    got = []
    for rows in ([0, 0], [7, 30]):
        batch = B.Batch(ws)
        with torch.cuda.stream(batch.stream):
            batch.init()
            for r in rows:
                batch.set_segment_rows(r)
                batch.step(3)
            got.append([[ev.download(buf) for buf in BUFS] for ev in batch.events])
        batch.close()
    for a, b in zip(*got):
        for x, y in zip(a, b):
            assert np.array_equal(x, y)
