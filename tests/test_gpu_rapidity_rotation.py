"""The push's rapidity rotation over its angles: FP32 sums one to four terms of
its series up to an angle of 0.08 and takes the exponential beyond."""
import numpy as np
import pytest

import oracle as O
from paper_2303_05599_gb300 import _binding as B
from paper_2303_05599_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("prec", [W.FP64, W.FP32_2ROW])
def test_rotation_over_the_angles(prec):
    N, n = 32, 8
    w = W.Workload("rapidity", N=N, L_fm=1.5, precision=prec, reunit_every=0,
                   species=[W.Species(0.0, 0.0, N * N, W.REP_F, W.MOM_FIXED_PT, 0.5)])
    rng = np.random.default_rng(11)
    f32 = (lambda a: a.astype(np.float32).astype(np.float64)) if prec == W.FP32_2ROW else (lambda a: a)
    # angle dt / t v_w |phi| with dt / t = 1/8 and v_w near 1, across the lattice and on both sides of each limit
    angle = np.geomspace(1e-6, 0.6, N * N)
    for k, limit in enumerate((2.4e-4, 5.6e-3, 2.9e-2, 8.1e-2)):
        angle[8 * k:8 * k + 8] = limit * np.linspace(0.97, 1.03, 8)
    phi = rng.normal(size=(N * N, 8))
    phi = f32(phi * (angle / (w.dt / (n * w.dt)) / np.linalg.norm(phi, axis=1))[:, None])
    st = O.FieldState(N, O.unit_links(N), phi, np.zeros((2, N * N, 8)), np.zeros((N * N, 8)))
    part = O.sample_species(N, 3, 0, W.REP_F, W.MOM_FIXED_PT, 0.5, 0.0, N * N)
    part[:, 0], part[:, 1] = np.arange(N * N) % N, np.arange(N * N) // N
    part[:, 2] = 0.0
    part[:, 5] = 20.0 * np.where(np.arange(N * N) % 2, 1, -1)
    part = f32(part)
    ev = B.Event(w)
    for buf, a in ((B.GL_BUF_LINKS, st.U), (B.GL_BUF_PHI, st.phi), (B.GL_BUF_E, st.e), (B.GL_BUF_PI, st.pi)):
        ev.upload(buf, a)
    ev.upload(B.GL_BUF_PARTICLES, part)
    ev.set_step(n)
    ev.step(1)
    got = ev.download(B.GL_BUF_PARTICLES)[:, 6:14]
    run = O.Run(st, part.copy(), [0.0], [0.0], [W.REP_F], w.dt, step=n)
    run.step()
    want = run.part[:, 6:14]
    # |Q| = 2; the two products of the exponential's route (six terms each) and the
    # rounding of phi and of the angle are each a few units in the last place
    eps = 2.0 ** -53 if prec == W.FP64 else 2.0 ** -24
    assert np.abs(want - part[:, 6:14]).max() > 0.1
    assert np.abs(got - want).max() < 24 * eps * 2.0
