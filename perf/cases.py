"""Performance cases: the calls a user of the library makes, at the sizes it is used at.

A run of the framework is: the MV initial conditions of one event or of a batch of events (once per
event), then report intervals, each a few coupled steps (fields and particles) followed by the ensemble
observables, now and then with the FP64 field checks.  The cases are those calls, on the workloads of
workloads.py and of the benchmark, from one 32 x 32 event to one of 1024 x 1024 with 4e6 particles.

Every output is a view of the state in the device layout (the fields of the current time, the site fields
of the last push, the particles) or an array of the observables that the call returned.  The states of the
step cases are MV fields of one colour sheet per nucleus (the same field strengths as with 50, at a
fraction of the preparation), evolved to the time at which the particles form, where the particles are
still as they were sampled.
"""
import math

import numpy as np
import torch

from paper_2303_05599_gb300 import _binding as B
from paper_2303_05599_gb300 import workloads as W

# species of a workload: (mass, momentum mode, p0, p1), equal shares of the particles, and the formation
# time of all of them
SPECIES = {
    "charm_rest": ([(W.M_CHARM, W.MOM_FIXED_PT, 0.0, 0.0)], 0.06),
    "charm_spread": ([(W.M_CHARM, W.MOM_UNIFORM_PT, 0.0, 5.0)], 0.06),
    "charm_static": ([(W.M_CHARM, W.MOM_FIXED_PT, 0.5, 0.0), (math.inf, W.MOM_FIXED_PT, 0.0, 0.0)], 0.06),
    "beauty_jets": ([(W.M_BEAUTY, W.MOM_FIXED_PT, 2.0, 0.0), (0.0, W.MOM_FIXED_PT, 10.0, 0.0)], 0.02),
    "mixed": ([(W.M_CHARM, W.MOM_FIXED_PT, 0.5, 0.0), (W.M_BEAUTY, W.MOM_FIXED_PT, 2.0, 0.0),
               (0.0, W.MOM_FIXED_PT, 10.0, 0.0)], 0.02),
    "quark_jets": ([(1.0, W.MOM_ALONG_X, 10.0, 0.0), (0.0, W.MOM_EIKONAL_X, 0.0, 0.0)], 0.02),
    "none": ([], 0.02),
}

BASE = {"batch": False, "events": 1, "dtau": 0.125, "sheets": 1, "precision": "fp32", "tune": False, "steps": 0,
        "observe": "none", "probes": 0, "return_particles": False}


def _case(**kw):
    return dict(BASE, **kw)


def listed():
    return [
        # the initial conditions of the plain FP64 method's event: the call before every parity run
        _case(name="init_event_n32_fp64", kind="init", sizes="32", a_fm=3.0 / 32, sheets=50, precision="fp64",
              species="charm_rest", particles=1000),
        # one production event of heavy quarks: fields of 50 sheets and 2e5 particles
        _case(name="init_event_n256", kind="init", sizes="256", a_fm=10.0 / 256, sheets=50, species="charm_static",
              particles=200_000),
        # the start of a batch of events of uneven size (the 64-event workload's first nine)
        _case(name="init_batch9", kind="init", batch=True, sizes="64,128,256", events=9, a_fm=0.04, sheets=50,
              species="charm_spread", particles=10_000),
        # the smallest run: a report interval (0.05 fm/c) of the plain FP64 event, with the field checks
        _case(name="event_n32_fp64", kind="step", sizes="32", a_fm=3.0 / 32, precision="fp64", species="charm_rest",
              particles=1000, steps=4, observe="all", return_particles=True),
        # one small FP32 event on its own: ten steps and the sums
        _case(name="event_n64", kind="step", sizes="64", a_fm=0.04, species="charm_spread", particles=10_000, steps=10,
              observe="particles", return_particles=True),
        # the benchmark's batch of 64 uneven events: a report interval
        _case(name="batch64_report", kind="step", batch=True, sizes="64,128,256", events=64, a_fm=0.04, tune=True,
              species="charm_spread", particles=10_000, steps=10, observe="particles"),
        # 30 production events, observed after every step
        _case(name="batch30_n256_step", kind="step", batch=True, sizes="256", events=30, a_fm=10.0 / 256, tune=True,
              species="charm_static", particles=200_000, steps=1, observe="particles", return_particles=True),
        # the largest event with its 4e6 particles: a report interval's worth of steps
        _case(name="event_n1024_mixed", kind="step", batch=True, sizes="1024", a_fm=10.0 / 1024, tune=True,
              species="mixed", particles=4_000_000, steps=10, observe="particles"),
        # a lattice that is no multiple of a warp or a tile, through the single-event calls
        _case(name="event_n500_jets", kind="step", sizes="500", a_fm=10.0 / 500, species="beauty_jets",
              particles=1_000_000, steps=2, tune=True, return_particles=True),
        # the plain FP64 path on several events
        _case(name="batch9_fp64", kind="step", batch=True, sizes="64,128,256", events=9, a_fm=0.04, precision="fp64",
              species="charm_spread", particles=10_000, steps=2, observe="particles", return_particles=True),
        # the jet setup at dtau = a/16 with the correlator's probes
        _case(name="event_n1024_probes", kind="step", sizes="1024", a_fm=10.0 / 1024, dtau=1.0 / 16, tune=True,
              species="quark_jets", particles=200_000, probes=100_000, steps=4, observe="probes",
              return_particles=True),
        # the FP64 field checks of a batch, as every report with --field-checks and the last one of a run take
        _case(name="checks_batch18", kind="checks", batch=True, sizes="64,128,256", events=18, a_fm=0.04,
              species="charm_spread", particles=1000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Another case of the same calls, sizes spread over their range, odd ones among them."""
    kind = rng.choice(["init", "step", "step", "step", "checks"])
    precision = "fp64" if rng.random() < 0.3 else "fp32"
    sp = rng.choice(["charm_rest", "charm_spread", "charm_static", "beauty_jets", "mixed"])
    if kind == "init":
        if rng.random() < 0.5:
            sizes, events = str(rng.choice([32, 64, 128, 256, _log(rng, 20, 90)])), 1
        else:
            sizes, events = rng.choice(["64,128", "32,64,128", "64", "128", "48,64"]), rng.randint(2, 8)
        return _case(kind="init", batch=events > 1, sizes=sizes, events=events, a_fm=rng.uniform(0.03, 0.09),
                     sheets=rng.choice([10, 30, 50]), precision=precision, species=sp,
                     particles=_log(rng, 500, 100_000))
    if kind == "checks":
        return _case(kind="checks", batch=True, sizes=rng.choice(["64,128,256", "128", "256", "100,64", "33,250"]),
                     events=rng.randint(2, 24), a_fm=0.04, precision=precision, species="charm_spread",
                     particles=_log(rng, 300, 3000))
    if rng.random() < 0.5:  # one event
        n = rng.choice([32, 64, 128, 256, 512, 1024, _log(rng, 20, 500)])
        if precision == "fp64":
            n = min(n, 256)
        return _case(kind="step", sizes=str(n), a_fm=rng.uniform(0.02, 0.09), precision=precision,
                     dtau=rng.choice([0.125, 0.0625]), species=rng.choice([sp, sp, "none"]),
                     particles=_log(rng, 500, max(1000, 2 * n * n)), steps=rng.randint(1, 10), tune=n >= 256,
                     observe=rng.choice(["none", "particles", "all"]))
    big = precision == "fp32"
    sizes = rng.choice(["64,128,256", "256", "100,200", "64", "127,64"] + (["512"] if big else []))
    return _case(kind="step", batch=True, sizes=sizes, events=rng.randint(3, 40 if big and sizes != "512" else 8),
                 a_fm=0.04, precision=precision, species=sp, particles=_log(rng, 1000, 100_000),
                 steps=rng.randint(1, 10 if big else 2), tune=big, observe="particles")


# ---------------------------------------------------------------- states


def _up(n):
    return (n + 255) & ~255


def _sizes(case):
    s = [int(x) for x in case["sizes"].split(",")]
    return [s[e % len(s)] for e in range(case["events"])]


def _workloads(case, seed):
    kinds, t_form = SPECIES[case["species"]]
    out = []
    for e, n in enumerate(_sizes(case)):
        share = case["particles"] // max(1, len(kinds))
        sp = [W.Species(m, t_form, share, W.REP_F, mode, p0, p1) for m, mode, p0, p1 in kinds]
        out.append(W.Workload("case_e%d" % e, N=n, L_fm=case["a_fm"] * n, Ns=case["sheets"],
                              precision=W.FP64 if case["precision"] == "fp64" else W.FP32_2ROW,
                              dtau_over_a=case["dtau"], n_jets=case["probes"], seed=1000 * (seed % 1000003) + e,
                              species=sp))
    return out


class Layout:
    """Where an event's arrays lie in the caller's workspace: two slices of the fields, two of the site
    fields, the particles and the second particle buffer that the sort swaps with, each 256-byte aligned."""

    def __init__(self, w, fields, parts):
        self.real = torch.float64 if w.precision == W.FP64 else torch.float32
        self.b = 8 if w.precision == W.FP64 else 4
        self.sites, self.np = w.N * w.N, w.n_particles
        self.fields, self.site = fields, 48 * self.sites * self.b
        self.field_at = [0, _up(fields)]
        self.site_at = [2 * _up(fields), 2 * _up(fields) + _up(self.site)]
        first = 2 * _up(fields) + 2 * _up(self.site)
        self.parts_at = [first, first + _up(parts)]
        # state planes: FP64 xy, pxy, (eta, P_eta), q; FP32 (x, y, px, py), (eta, P_eta), q
        self.planes = [16, 16, 16, 64] if self.b == 8 else [16, 8, 32]
        self.starts = [sum(_up(k * self.np) for k in self.planes[:i]) for i in range(len(self.planes) + 1)]


class State:
    """A batch or an event, its workspace as a tensor of the state's precision, and its step."""

    def __init__(self, case, seed):
        self.case, self.ws = case, _workloads(case, seed)
        self.obj = B.Batch(self.ws) if case["batch"] else B.Event(self.ws[0])
        self.events = self.obj.events if case["batch"] else [self.obj]
        self.obj.workspace.zero_()
        torch.cuda.current_stream().synchronize()
        self.n, self.samplings, self.by_step = 0, 0, {}
        raw = self.obj.workspace
        base = -raw.data_ptr() % 256
        each = [_up(B.gl_workspace_bytes(w)) for w in self.ws]
        self.lay = [Layout(w, ev.native_bytes(B.GL_NATIVE_FIELDS), ev.native_bytes(B.GL_NATIVE_PARTICLES))
                    for w, ev in zip(self.ws, self.events)]
        end = base + raw.numel() - 256
        at = (end - sum(each)) if case["batch"] else base
        L = self.lay[0]
        self.flat = raw[base:base + (raw.numel() - base) // 16 * 16].view(L.real)
        self.start = [(at - base + sum(each[:e])) // L.b for e in range(len(each))]
        cyc = len(case["sizes"].split(","))
        self.groups = []  # events of one size are evenly spaced
        for g in range(min(cyc, len(each))):
            self.groups.append((g, len(range(g, len(each), cyc)), sum(each[:cyc]) // L.b))

    def view(self, offsets, k, count):
        """`count` bytes at offsets(layout)[k] of every event, one tensor for each size of event."""
        out = []
        for g, n, step in self.groups:
            L = self.lay[g]
            first = self.flat.storage_offset() + self.start[g] + offsets(L)[k] // L.b
            out.append(torch.as_strided(self.flat, (n, count(L) // L.b), (step, 1), first))
        return out

    def outputs(self, n, site, particles):
        out = {"fields": self.view(lambda L: L.field_at, n & 1, lambda L: L.fields)}
        if site:
            out["site"] = self.view(lambda L: L.site_at, (n - 1) & 1, lambda L: L.site)
        if particles:
            out["particles"] = self.view(lambda L: L.parts_at, self.buffer(n), lambda L: L.starts[-1])
        return out

    def buffer(self, n):
        """The particle buffer in use: swapped by the sort of each sampling and every sort_every steps."""
        return (self.samplings + n // self.ws[0].sort_every) % 2

    def stream(self):
        return torch.cuda.stream(self.obj.stream)


def _init(state):
    state.samplings += 1
    if state.case["batch"]:
        state.obj.init()
    else:
        state.obj.glasma_init()
        state.obj.wong_init()


def _formed(case):
    """The first step at which every particle is pushed."""
    return int(math.ceil(SPECIES[case["species"]][1] / case["a_fm"] / case["dtau"] - 1e-9))


def prepare(case, seed):
    s = State(case, seed)
    if case["kind"] == "init":
        return s
    with s.stream():
        _init(s)
        if case["kind"] == "checks":
            # a state with a Gauss residual to find: random momenta and scalar on the MV links
            rng = np.random.default_rng(seed)
            for which, d in ((B.GL_BUF_PHI, 1), (B.GL_BUF_E, 2), (B.GL_BUF_PI, 1)):
                s.obj.upload(which, [0.3 * rng.standard_normal(d * w.N * w.N * 8) for w in s.ws])
            return s
        if case["tune"]:
            s.obj.autotune()
        s.n = _formed(case)
        s.obj.step(s.n)
        s.obj.stream.synchronize()
    return s


# gl_obs as 64-bit words: counts from word 3, the per-species sums from 11, the field checks from 59
_WORDS = (11, 59, 66)


def _observed(records, real, checks):
    raw = np.stack([np.frombuffer(o, np.float64) for o in records])
    sums = raw[:, _WORDS[0]:_WORDS[2] if checks else _WORDS[1]]
    return {"counts": raw[:, 3:11].view(np.int64), "sums": sums.astype(np.float64 if real == torch.float64
                                                                       else np.float32)}


def run(s):
    case = s.case
    with s.stream():
        if case["kind"] == "init":
            _init(s)
            return s.outputs(0, False, True)
        if case["kind"] == "checks":
            obs = s.obj.observables(B.GL_OBS_FIELDS)
            return {"gauss": np.array([[o.gauss_max, o.gauss_rms] for o in obs]),
                    "unitarity": np.array([o.unitarity_max for o in obs])}
        s.obj.step(case["steps"])
        s.n += case["steps"]
        key = (s.n & 1, s.buffer(s.n))
        if key not in s.by_step:
            has = s.lay[0].np > 0
            s.by_step[key] = s.outputs(s.n, True, has and case["return_particles"])
        out = dict(s.by_step[key])
        if case["observe"] == "probes":
            out["probes"] = np.array(s.obj.jets_observables(), np.float32)
        elif case["observe"] != "none":
            obs = s.obj.observables(B.GL_OBS_PARTICLES if case["observe"] == "particles" else B.GL_OBS_ALL)
            out.update(_observed(obs if case["batch"] else [obs], s.lay[0].real, case["observe"] == "all"))
        return out


def work(case):
    """The bytes a pass has to move and its arithmetic.  A step reads and writes links, phi, e and pi and
    writes the six site fields; the push reads the site fields and the scalar and reads and writes 14 values
    a particle.  About 4,800 flops a site and 960 a particle and step.  The initial conditions: per nucleus
    and sheet eight normal variates, two real transforms of eight planes and one SU(3) exponential and
    product a site, then two 8 x 8 Newton solves of about four iterations a site."""
    b = 8 if case["precision"] == "fp64" else 4
    n, np_ = [float(x) for x in _sizes(case)], float(case["particles"] if case["species"] != "none" else 0)
    sites, ev = sum(x * x for x in n), case["events"]
    link = 18 if b == 8 else 12
    state = (2 * link + 32) * b
    if case["kind"] == "init":
        flops = sum(x * x * (2 * case["sheets"] * (8 * 40 + 8 * 2 * 2.5 * math.log2(x * x) + 700) + 2 * 4 * 4000)
                    for x in n)
        return {"bytes": sites * state + ev * np_ * (14 * b + 16), "flops": flops + ev * np_ * 1500}
    if case["kind"] == "checks":
        return {"bytes": sites * (state + 48 * b), "flops": sites * 900.0}
    step = sites * (2 * state + 48 * b) + sites * (56 * b if np_ else 0) + ev * np_ * (28 * b + 4)
    step += case["probes"] * 42 * 2 * b
    obs = ev * np_ * (14 * b + 12) if case["observe"] in ("particles", "all") else 0
    if case["observe"] == "all":
        obs += sites * (state + 48 * b)
    return {"bytes": case["steps"] * step + obs, "flops": case["steps"] * (4800 * sites + 960 * ev * np_)}


# ---------------------------------------------------------------- the same in 64 bits, in plain torch


def _generators(dev):
    t = torch.zeros(8, 3, 3, dtype=torch.complex128, device=dev)
    for a, i, j in ((0, 0, 1), (3, 0, 2), (5, 1, 2)):
        t[a, i, j] = t[a, j, i] = 0.5
        t[a + 1, i, j], t[a + 1, j, i] = -0.5j, 0.5j
    t[2, 0, 0], t[2, 1, 1] = 0.5, -0.5
    t[7] = torch.diag(torch.tensor([1.0, 1.0, -2.0], dtype=torch.complex128, device=dev)) / (2 * math.sqrt(3.0))
    return t


def _mm(a, b):
    return (a[..., :, :, None] * b[..., None, :, :]).sum(-2)


def _dag(a):
    return a.conj().transpose(-1, -2)


def _mat(x):
    return torch.einsum("...a,aij->...ij", x.to(torch.complex128), _generators(x.device))


def _comp(m):
    return 2 * torch.einsum("...ij,aji->...a", m, _generators(m.device)).real


def _iah(m):
    return _comp(0.5j * (m - _dag(m)))


def _up_t(u, x):
    return _comp(_mm(_mm(u, _mat(x)), _dag(u)))


def _dn_t(u, x):
    return _comp(_mm(_mm(_dag(u), _mat(x)), u))


def _icomm(x, y):
    a, b = _mat(x), _mat(y)
    return _comp(1j * (_mm(a, b) - _mm(b, a)))


def _expi(x):
    n = x.shape[:-1]
    return torch.linalg.matrix_exp(1j * _mat(x).reshape(-1, 3, 3)).reshape(*n, 3, 3)


def _fx(a):  # the value at x + 1, and below those at x - 1, y + 1, y - 1
    return torch.roll(a, -1, 1)


def _bx(a):
    return torch.roll(a, 1, 1)


def _fy(a):
    return torch.roll(a, -1, 0)


def _by(a):
    return torch.roll(a, 1, 0)


class Ref:
    """One event's fields and particles in 64 bits, read from a state's arrays and written as they are laid out."""

    def __init__(self, s, e):
        self.L, self.w, self.dt, self.n = s.lay[e], s.ws[e], s.case["dtau"], s.n
        at, L, N = s.start[e], s.lay[e], s.ws[e].N

        def planes(off, floats, width):
            p = s.flat[at + off // L.b: at + off // L.b + floats].double()
            return p.reshape(-1, N * N, width).permute(1, 0, 2).reshape(N * N, -1)

        width = 2 if L.b == 8 else 4
        f = planes(L.field_at[s.n & 1], L.fields // L.b, width)
        lw = 18 if L.b == 8 else 12
        self.U = [self._link(f[:, d * lw:(d + 1) * lw]).reshape(N, N, 3, 3) for d in range(2)]
        alg = [f[:, 2 * lw + 8 * k: 2 * lw + 8 * k + 8].reshape(N, N, 8) for k in range(4)]
        self.phi, self.e, self.pi = alg[0], [alg[1], alg[2]], alg[3]
        self.site = None
        if L.np == 0:
            return
        p0 = L.parts_at[s.buffer(s.n)]

        def plane(k, width):
            o = at + (p0 + L.starts[k]) // L.b
            return s.flat[o:o + L.np * width].double().reshape(L.np, width)

        if L.b == 8:
            xy, p, ep = plane(0, 2), plane(1, 2), plane(2, 2)
        else:
            xyp, ep = plane(0, 4), plane(1, 2)
            xy, p = xyp[:, :2], xyp[:, 2:]
        self.x, self.y, self.px, self.py = xy[:, 0], xy[:, 1], p[:, 0], p[:, 1]
        self.eta, self.Pe = ep[:, 0], ep[:, 1]
        o = at + (p0 + L.starts[-2]) // L.b
        self.q = s.flat[o:o + 8 * L.np].double().reshape(-1, L.np, width).permute(1, 0, 2).reshape(L.np, 8)
        o = at + (p0 + L.starts[-1]) // L.b
        self.sp = s.flat[o:o + (4 * L.np + L.b - 1) // L.b].view(torch.int32)[:L.np].long()
        self.pt0 = self.px ** 2 + self.py ** 2  # sampled momenta: nothing has been pushed yet

    @staticmethod
    def _link(f):
        m = torch.view_as_complex(f.reshape(f.shape[0], -1, 2).contiguous()).reshape(f.shape[0], -1, 3)
        if m.shape[1] == 2:
            m = torch.cat([m, torch.linalg.cross(m[:, 0], m[:, 1]).conj()[:, None]], 1)
        return m

    def field_step(self):
        n, dt = self.n, self.dt
        t, th = n * dt, n * dt + 0.5 * dt
        it = 1.0 / t if t > 0 else 0.0
        (ux, uy), phi = self.U, self.phi
        A = _iah(_mm(_mm(_mm(ux, _fx(uy)), _dag(_fy(ux))), _dag(uy)))
        Dn, Lf = _dn_t(_by(uy), _by(A)), _dn_t(_bx(ux), _bx(A))
        tx, ty = _up_t(ux, _fx(phi)), _up_t(uy, _fy(phi))
        bx, by = _dn_t(_bx(ux), _bx(phi)), _dn_t(_by(uy), _by(phi))
        ex = self.e[0] + dt * (t * (A - Dn) + it * _icomm(tx, phi))
        ey = self.e[1] + dt * (t * (Lf - A) + it * _icomm(ty, phi))
        pi = self.pi + dt * it * (tx + bx + ty + by - 4 * phi)
        sx, sy = self.e[0] + ex, self.e[1] + ey
        self.site = torch.stack([0.25 * it * (sx + _dn_t(_bx(ux), _bx(sx))),
                                 0.25 * it * (sy + _dn_t(_by(uy), _by(sy))), 0.5 * (self.pi + pi),
                                 -0.5 * it * (ty - by), 0.5 * it * (tx - bx),
                                 0.25 * (A + Lf + Dn + _dn_t(_by(uy), _by(Lf)))])
        self.U = [_mm(_expi(dt / th * ex), ux), _mm(_expi(dt / th * ey), uy)]
        self.phi, self.e, self.pi = phi + dt * th * pi, [ex, ey], pi

    def push(self):
        """The particles from t_n to t_n+1, with the site fields of t_n and the links and scalar of t_n+1."""
        dt, t, N = self.dt, self.n * self.dt, self.w.N
        mass = torch.tensor([x[0] for x in self.w.lattice_species()], dtype=torch.float64, device=self.x.device)
        mode = torch.tensor([2 if s.mom_mode == W.MOM_EIKONAL_X else 1 if math.isinf(s.mass_GeV) else 0
                             for s in self.w.species], device=self.x.device)[self.sp]
        ix, iy = torch.floor(self.x + 0.5), torch.floor(self.y + 0.5)
        at = (iy.long() % N) * N + ix.long() % N
        qE = [(self.q * f.reshape(-1, 8)[at]).sum(-1) for f in self.site]
        Ex, Ey, Ee, Bx, By, Be = qE
        m = torch.where(mode == 0, mass[self.sp], torch.zeros_like(Ex))
        w = self.Pe / t if t > 0 else torch.zeros_like(Ex)
        pt = torch.sqrt(self.px ** 2 + self.py ** 2 + w ** 2 + m ** 2)
        inv = torch.where(pt > 0, 1 / pt, torch.zeros_like(pt))
        vx, vy, vw = self.px * inv, self.py * inv, w * inv
        wong, eik = mode == 0, mode == 2
        deta = torch.where(wong, (dt / t if t > 0 else 0.0) * vw, torch.zeros_like(vw))
        self.px = self.px + dt * torch.where(wong, Ex + Be * vy - By * vw, Ex)
        self.py = self.py + dt * torch.where(wong, Ey - Be * vx + Bx * vw, torch.where(eik, Ey - Be, Ey))
        self.Pe = self.Pe + dt * torch.where(wong, t * (Ee - Bx * vy + By * vx), torch.where(eik, Ee + By, Ee))
        self.eta = self.eta + deta
        one, zero = torch.ones_like(vx), torch.zeros_like(vx)
        xn = self.x + dt * torch.where(wong, vx, torch.where(eik, one, zero))
        yn = self.y + dt * torch.where(wong, vy, zero)
        jx, jy = torch.floor(xn + 0.5), torch.floor(yn + 0.5)
        self.x, self.y = torch.remainder(xn, N), torch.remainder(yn, N)
        for axis, d, here, there in ((0, jx - ix, (iy, ix), (iy, jx)), (1, jy - iy, (iy, jx), (jy, jx))):
            for up, cell in ((1, here), (-1, there)):
                k = torch.nonzero(d == up)[:, 0]
                u = self.U[axis].reshape(-1, 3, 3)[(cell[0][k].long() % N) * N + cell[1][k].long() % N]
                self.q[k] = (_dn_t if up == 1 else _up_t)(u, self.q[k])
        k = torch.nonzero(deta != 0)[:, 0]
        cell = (jy[k].long() % N) * N + jx[k].long() % N
        self.q[k] = _up_t(_expi(-deta[k, None] * self.phi.reshape(-1, 8)[cell]), self.q[k])

    def sums(self):
        """[48]: sum p_x^2, p_y^2, p_L^2, p_T^2 - p_T^2 at formation, Casimir drifts, 8 species each."""
        t, out = self.n * self.dt, torch.zeros(6, B.GL_MAX_SPECIES, dtype=torch.float64)
        counts = [0] * B.GL_MAX_SPECIES
        for k, s in enumerate(self.w.species):
            i = torch.nonzero(self.sp == k)[:, 0]
            px, py, w = self.px[i], self.py[i], self.Pe[i] / t
            if s.mom_mode == W.MOM_EIKONAL_X or math.isinf(s.mass_GeV):
                pl = self.Pe[i]
            else:
                m = s.mass_GeV * self.w.a_GeVinv
                pl = torch.sqrt(px ** 2 + py ** 2 + w ** 2 + m ** 2) * torch.sinh(self.eta[i]) + w * torch.cosh(self.eta[i])
            for r, v in enumerate((px ** 2, py ** 2, pl ** 2, px ** 2 + py ** 2 - self.pt0[i])):
                out[r, k] = v.sum() / self.w.a_GeVinv ** 2
            counts[k] = len(i)
        return out.reshape(-1).cpu(), counts

    def _planes(self, values):
        width = 2 if self.L.b == 8 else 4
        return values.reshape(values.shape[0], -1, width).permute(1, 0, 2).reshape(-1)

    def packed_fields(self):
        rows = 3 if self.L.b == 8 else 2
        links = [torch.view_as_real(u[:, :, :rows].contiguous()).reshape(-1, 6 * rows) for u in self.U]
        alg = [x.reshape(-1, 8) for x in (self.phi, *self.e, self.pi)]
        return self._planes(torch.cat(links + alg, 1))

    def packed_site(self):
        return torch.cat([self._planes(x.reshape(-1, 8)) for x in self.site])

    def packed_particles(self):
        L = self.L
        out = torch.zeros(L.starts[-1] // L.b, dtype=torch.float64, device=self.x.device)
        st = lambda *v: torch.stack(v, 1).reshape(-1)  # noqa: E731
        head = [st(self.x, self.y), st(self.px, self.py)] if L.b == 8 else [st(self.x, self.y, self.px, self.py)]
        for o, v in zip(L.starts, head + [st(self.eta, self.Pe), self._planes(self.q)]):
            out[o // L.b:o // L.b + v.numel()] = v
        return out


# Philox4x32-10 on int64 tensors (Salmon, Moraes, Dror, Shaw, SC'11), and the draws made from it
_M32 = 0xFFFFFFFF


def _mulhilo(m, c):
    lo = (m * c) & _M32
    return (m * (c >> 16) + ((m * (c & 0xFFFF)) >> 16)) >> 16, lo


def _philox(c0, c1, c2, c3, seed):
    k0, k1 = seed & _M32, (seed >> 32) & _M32
    one = torch.zeros_like(c0)
    x, y, z, w = c0, one + c1, one + c2, one + c3
    for _ in range(10):
        h0, l0 = _mulhilo(0xD2511F53, x)
        h1, l1 = _mulhilo(0xCD9E8D57, z)
        x, y, z, w = h1 ^ y ^ k0, l1, h0 ^ w ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return [(v.double() + 0.5) / 4294967296.0 for v in (x, y, z, w)]


def _normals(u):
    out = []
    for a, b in ((u[0], u[1]), (u[2], u[3])):
        r = torch.sqrt(-2 * torch.log(a))
        out += [r * torch.cos(2 * math.pi * b), r * torch.sin(2 * math.pi * b)]
    return out


def _wilson(w, nucleus, dev):
    N = w.N
    site = torch.arange(N * N, device=dev)
    s2 = torch.sin(math.pi * torch.arange(N, device=dev, dtype=torch.float64) / N) ** 2
    k2 = 4 * (s2[:, None] + s2[None, :])
    g = 1 / (k2 + w.m_a ** 2)
    g[0, 0] = 0
    if w.Lambda_a > 0:
        g[k2 > w.Lambda_a ** 2] = 0
    v = torch.eye(3, dtype=torch.complex128, device=dev).expand(N, N, 3, 3)
    for sheet in range(w.Ns):
        c = 2 * (nucleus * w.Ns + sheet)
        z = torch.stack(sum((_normals(_philox(site, c + j, 1, 0, w.seed)) for j in range(2)), []), 0)
        rho = w.g2mu_a / math.sqrt(w.Ns) * z.reshape(8, N, N)
        alpha = torch.fft.ifft2(torch.fft.fft2(rho.to(torch.complex128)) * g).real
        v = _mm(v, _expi(-alpha.permute(1, 2, 0)))
    return v


def _match(ua, ub):
    """The Glasma link: Im tr T^a (U^A + U^B)(1 + U^+) = 0 by damped Newton steps from U^A U^B."""
    T = _generators(ua.device)
    one = torch.eye(3, dtype=torch.complex128, device=ua.device)
    w, u = ua + ub, _mm(ua, ub)

    def residual(u):
        f = torch.einsum("aij,...ji->...a", T, _mm(w, one + _dag(u))).imag
        return f, f.abs().amax(-1)

    f, r = residual(u)
    for _ in range(30):
        live = torch.nonzero(r > 1e-14)[:, 0]
        if not len(live):
            break
        k = torch.einsum("aij,njk,bki->nab", T, _mm(w[live], _dag(u[live])), T)
        dx = torch.linalg.solve(-k.real, -f[live, :, None])[..., 0]
        lam = torch.ones_like(r[live])
        todo = torch.arange(len(live), device=r.device)
        cur = u.clone()
        for half in range(30):
            un = _mm(_expi(lam[todo, None] * dx[todo]), cur[live[todo]])
            fn = torch.einsum("aij,...ji->...a", T, _mm(w[live[todo]], one + _dag(un))).imag
            rn = fn.abs().amax(-1)
            good = (rn < r[live[todo]]) | (half == 29)
            at = live[todo[good]]
            u[at], f[at], r[at] = un[good], fn[good], rn[good]
            lam[todo[~good]] *= 0.5
            todo = todo[~good]
            if not len(todo):
                break
    return u


def _q0():
    """Q^8 of the fundamental charge: the root of s^3 - 12 s - 20 / sqrt(3) near -1.06."""
    r = np.roots([1.0, 0.0, -12.0, -20 / math.sqrt(3.0)]).real
    s = float(r[np.argmin(np.abs(r + 1.06))])
    for _ in range(3):
        s -= (s ** 3 - 12 * s - 20 / math.sqrt(3.0)) / (3 * s * s - 12)
    return s


def _sampled(w, dev):
    """x, y, px, py, q and species of every particle in the order of its sampling."""
    parts = []
    s8 = _q0()
    q0 = torch.zeros(8, dtype=torch.float64, device=dev)
    q0[7], q0[4] = s8, -math.sqrt(4 - s8 * s8)
    for k, (sp, lat) in enumerate(zip(w.species, w.lattice_species())):
        i = torch.arange(sp.count, device=dev)
        u = _philox(i, k, 2, 0, w.seed)
        pt = lat[2] + (lat[3] - lat[2]) * u[3] if sp.mom_mode == W.MOM_UNIFORM_PT else lat[2] + 0 * u[3]
        px, py = pt * torch.cos(2 * math.pi * u[2]), pt * torch.sin(2 * math.pi * u[2])
        if sp.mom_mode == W.MOM_ALONG_X:
            px, py = lat[2] + 0 * px, 0 * py
        if sp.mom_mode == W.MOM_EIKONAL_X:
            px, py = 0 * px, 0 * py
        z = torch.stack(sum((_normals(_philox(i, k, 3, j, w.seed)) for j in range(5)), [])[:18], 1)
        h = torch.view_as_complex(z.reshape(-1, 3, 3, 2).contiguous()) / math.sqrt(2.0)
        cols = []
        for c in range(3):
            v = h[:, :, c]
            for _ in range(2):
                for o in cols:
                    v = v - (o.conj() * v).sum(-1, keepdim=True) * o
            cols.append(v / torch.sqrt((v.abs() ** 2).sum(-1, keepdim=True)))
        parts.append((w.N * u[0], w.N * u[1], px, py, _up_t(torch.stack(cols, -1), q0.expand(sp.count, 8)),
                      torch.full((sp.count,), k, device=dev)))
    return [torch.cat(v) for v in zip(*parts)]


def _exact_init(s):
    refs = []
    for e, w in enumerate(s.ws):
        dev = s.flat.device
        r = Ref.__new__(Ref)
        r.L, r.w, N = s.lay[e], w, w.N
        va, vb = _wilson(w, 0, dev), _wilson(w, 1, dev)
        r.U, links = [], []
        for f in (_fx, _fy):
            a, b = _mm(_dag(va), f(va)), _mm(_dag(vb), f(vb))
            links.append((a, b))
            r.U.append(_match(a.reshape(-1, 3, 3), b.reshape(-1, 3, 3)).reshape(N, N, 3, 3))
        pi = torch.zeros(N, N, 8, dtype=torch.float64, device=dev)
        for (a, b), back, u in zip(links, (_bx, _by), r.U):
            c = _icomm(-_iah(a), -_iah(b))
            pi -= 0.5 * (c + back(_dn_t(u, c)))
        r.pi, r.phi = pi, torch.zeros_like(pi)
        r.e = [torch.zeros_like(pi)] * 2
        x, y, px, py, q, sp = _sampled(w, dev)
        real = s.lay[e].real
        cx, cy = (torch.floor(v.to(real) + 0.5).long() % N for v in (x, y))
        motion = [2 if t.mom_mode == W.MOM_EIKONAL_X else 1 if math.isinf(t.mass_GeV) else 0 for t in w.species]
        seen = list(dict.fromkeys(motion))
        cls = torch.tensor([seen.index(m) for m in motion], device=dev)[sp]
        order = torch.argsort((cy * len(seen) + cls) * N + cx, stable=True)
        r.x, r.y, r.px, r.py, r.q = (v[order] for v in (x, y, px, py, q))
        r.eta = r.Pe = torch.zeros_like(r.x)
        refs.append(r)
    return refs


def _exact_checks(s):
    out = []
    for e in range(len(s.ws)):
        r = Ref(s, e)
        g = _icomm(r.phi, r.pi)
        for d, back in ((0, _bx), (1, _by)):
            g = g + r.e[d] - _dn_t(back(r.U[d]), back(r.e[d]))
        g2 = (g * g).sum(-1)
        out.append([math.sqrt(g2.max().item()), math.sqrt(g2.mean().item())])
    # the links' unitarity is that of the stored rounding, which 64 bits have no value for
    return {"gauss": np.array(out), "unitarity": None}


def _probes(s):
    """The correlator's probes as they are before the pass: x0, y0, W and the three integrals."""
    j = torch.from_numpy(s.obj.download(B.GL_BUF_JETS)).to(s.flat.device)
    W0 = torch.view_as_complex(j[:, 2:20].reshape(-1, 3, 3, 2).contiguous())
    return [j[:, 0], j[:, 1], W0, [j[:, 20 + 8 * i:28 + 8 * i] for i in range(3)]]


def _probe_step(p, r):
    t, N = r.n * r.dt, r.w.N
    x = p[0] + t
    ix = torch.floor(x + 0.5)
    at = (torch.floor(p[1] + 0.5).long() % N) * N + ix.long() % N
    Ex, Ey, Ee, _, By, Be = (f.reshape(-1, 8)[at] for f in r.site)
    for i, f in enumerate((Ex, Ey - Be, Ee + By)):
        p[3][i] = p[3][i] + r.dt * _up_t(p[2], f)
    k = torch.nonzero(torch.floor(x + r.dt + 0.5) != ix)[:, 0]
    p[2][k] = _mm(p[2][k], r.U[0].reshape(-1, 3, 3)[at[k]])


def exact(case, seed):
    """What run returns, in 64 bits, from the same arrays (step cases) or seeds (initial conditions)."""
    s = State(case, seed) if case["kind"] == "init" else prepare(case, seed)
    torch.cuda.synchronize()
    if case["kind"] == "checks":
        return _exact_checks(s)
    groups = lambda v: [torch.stack(v[g::len(s.groups)]) for g in range(len(s.groups))]  # noqa: E731
    if case["kind"] == "init":
        refs = _exact_init(s)
        return {"fields": groups([r.packed_fields() for r in refs]),
                "particles": groups([r.packed_particles() for r in refs])}
    has = s.lay[0].np > 0
    keep = {"fields": [], "site": [], "particles": []}
    sums, counts, probes = [], [], None
    for e in range(len(s.ws)):
        r = Ref(s, e)
        if case["observe"] == "probes":
            probes = _probes(s)
        for _ in range(case["steps"]):
            r.field_step()
            if has:
                r.push()
            if probes:
                _probe_step(probes, r)
            r.n += 1
        keep["fields"].append(r.packed_fields())
        keep["site"].append(r.packed_site())
        if has and case["return_particles"]:
            keep["particles"].append(r.packed_particles())
        if case["observe"] in ("particles", "all"):
            v, c = r.sums() if has else (torch.zeros(48, dtype=torch.float64), [0] * 8)
            if case["observe"] == "all":
                half = 0.5 * (r.site * r.site).sum(-1).mean((1, 2)).cpu()
                v = torch.cat([v, torch.tensor([0.0, 0.0, 0.0, half[0] + half[1], half[2], half[3] + half[4],
                                                half[5]], dtype=torch.float64)])
            sums.append(v)
            counts.append(c)
    out = {k: groups(v) for k, v in keep.items() if v}
    if sums:
        out["counts"], out["sums"] = np.array(counts, np.int64), torch.stack(sums).numpy()
    if probes:
        out["probes"] = np.array([(x * x).sum(-1).mean().item() / s.ws[0].a_GeVinv ** 2 for x in probes[3]])
    return out
