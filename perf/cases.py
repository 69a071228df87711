"""The work that users of this framework have it do, as cases that can be timed.

Every case goes through the public binding (paper_1506_07207_gb300.sic).  Sizes are
those of the repository's configurations, of its serving mix and of its tests, and odd
ones between them.  A case's kind says what one pass is:

* ``run``      a whole small simulation: create, step, read the history and the tracers
               back, destroy;
* ``chunk``    a resident simulation advanced by some steps, its history, field and
               device state then taken: the inner loop of every long run;
* ``batch``    several resident simulations advanced together;
* ``diag``     what an analysis reads of a state: mesh, density, field, moments, spectra;
* ``serve``    requests through the server, from submission to their histories.

A chunk or batch is called again and again on the same state, so its time step is small
enough that tens of thousands of steps leave the state what it was (a step's work does
not depend on the time step): quiet sheets stay quiet, folded ones stay as folded.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1506_07207_gb300 import inputs
from paper_1506_07207_gb300 import sic

BOX, LINEAR, NGP, CIC, FIRST = 0, 1, 2, 3, 4
POS_UNITS = 2.0 ** 30  # position units per box length


# ------------------------------------------------------------------ cases ----

def listed():
    return [
        # cold oscillation, whole: one sheet, the smallest thing that is ever run; latency
        dict(name="langmuir_run", kind="run", sheets=1, tracers=4096, nx=64, steps=500, dt=0.1),
        # linear Landau damping, the ordinary small plasma: 262 144 tracers, a few blocks per SM's worth of work
        dict(name="landau_linear", kind="chunk", state="landau", sheets=256, tracers=1024, nx=128, steps=64,
             dt=1e-3, deposit=BOX, refined=False),
        # two-stream at its full size while it is linear: quiet sheets, 16 tracers per cell of each
        dict(name="two_stream", kind="chunk", state="two_stream", sheets=512, tracers=16384, nx=1024, steps=16,
             dt=2e-4, deposit=BOX, refined=False),
        # nonlinear Landau late in its run: folded sheets, refined, so charges are per particle
        dict(name="landau_folded", kind="chunk", state="folded", sheets=1024, tracers=4096, nx=512, steps=16,
             dt=5e-5, deposit=BOX, refined=True),
        # a two-stream vortex at odd sizes, before any refinement: folded, one charge per sheet
        dict(name="two_stream_folded", kind="chunk", state="folded", sheets=255, tracers=9001, nx=1000, steps=16,
             dt=5e-5, deposit=BOX, refined=False),
        # the serving mix as admitted: sixteen requests resident together, the throughput case
        dict(name="batch_fresh", kind="batch", mix=11, members=16, steps=8, dt=2e-4, folded=0),
        # the same late in their lives: every second member folded and refined (two launches a step)
        dict(name="batch_late", kind="batch", mix=5, members=12, steps=8, dt=5e-5, folded=2),
        # piecewise-linear particles (Sec. 2.5) on folded sheets
        dict(name="linear_folded", kind="chunk", state="folded", sheets=256, tracers=2048, nx=256, steps=16,
             dt=5e-5, deposit=LINEAR, refined=False),
        # first-order weighting (Sec. 2.4), quiet sheets
        dict(name="first_order", kind="chunk", state="landau", sheets=256, tracers=2048, nx=256, steps=16,
             dt=2e-4, deposit=FIRST, refined=False),
        # irregular sheets: open and closed, ragged counts, a weight per tracer, an odd mesh
        dict(name="ragged", kind="chunk", state="ragged", sheets=301, tracers=3001, nx=777, steps=32,
             dt=5e-5, deposit=BOX, refined=False),
        # what the analysis of a nonlinear state reads (Sec. 2.3, 2.4 and 3.2)
        dict(name="diagnostics", kind="diag", state="folded", sheets=512, tracers=2048, nx=512, dt=5e-5,
             deposit=BOX, refined=False),
        # the server from submission to histories, long runs refining as they fold
        dict(name="serving", kind="serve", mix=3, members=10, steps=900, dt=0.05),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges; sizes log-uniform, as often odd as round."""
    def size(lo, hi):
        v = _log_int(rng, lo, hi)
        return 1 << max(1, round(math.log2(v))) if rng.random() < 0.4 else v

    kind = rng.choice(["run", "quiet", "quiet", "folded", "folded", "other", "ragged", "batch", "batch", "diag", "serve"])
    if kind == "run":
        return dict(kind="run", sheets=size(1, 64), tracers=size(500, 8000), nx=size(48, 1024),
                    steps=_log_int(rng, 100, 800), dt=0.1)
    if kind == "serve":
        return dict(kind="serve", mix=rng.randrange(1 << 20), members=rng.randint(3, 10),
                    steps=_log_int(rng, 200, 800), dt=0.05)
    if kind == "batch":
        folded = rng.choice([0, 0, 2, 3])
        c = dict(kind="batch", mix=rng.randrange(1 << 20), members=rng.randint(2, 14), steps=rng.choice([4, 8, 13]),
                 dt=5e-5 if folded else 2e-4, folded=folded)
        while work(c)["bytes"] > (2e9 if folded else 8e9):
            c["members"] -= 1
        return c
    if kind == "ragged":
        return dict(kind="chunk", state="ragged", sheets=size(5, 500), tracers=size(50, 4000), nx=size(32, 2048),
                    steps=rng.choice([8, 20, 32]), dt=5e-5, deposit=rng.choice([BOX, BOX, LINEAR, FIRST]), refined=False)
    state = rng.choice(["landau", "two_stream"]) if kind == "quiet" else rng.choice(["landau", "folded"]) if kind == "other" else "folded"
    c = dict(kind="diag" if kind == "diag" else "chunk", state=state, sheets=2 * size(16, 400), tracers=size(512, 8192),
             nx=size(64, 2048))
    if kind != "diag":
        c["steps"] = rng.choice([1, 5, 8, 16, 32])
    c["dt"] = 2e-4 if state != "folded" else 5e-5
    c["deposit"] = rng.choice([LINEAR, FIRST, NGP, CIC]) if kind == "other" else BOX
    c["refined"] = kind == "folded" and rng.random() < 0.5
    if c["deposit"] == LINEAR or kind == "diag":
        c["sheets"], c["tracers"] = min(c["sheets"], 256), min(c["tracers"], 2048)
    return c


# ----------------------------------------------------------------- inputs ----

def _rng(seed):
    return inputs.SplitMix64(0x51C0000 + seed)


def _device():
    return torch.device("cuda") if torch.cuda.is_available() else torch.device("cpu")


class Tracers:
    """Host arrays of one set-up: sheets of ordered tracers in a box."""

    def __init__(self, nx, L, dt, counts, closed, winding, x, v, w, compact=None, half_step=True):
        self.nx, self.L, self.dt = int(nx), float(L), float(dt)
        self.counts = np.asarray(counts, dtype=np.int64)
        self.closed, self.winding = np.asarray(closed, dtype=np.uint8), np.asarray(winding, dtype=np.int32)
        self.x, self.v, self.w = x, v, w   # float64 [sum(counts)], or None: the compact form
        self.compact = compact             # (x_template, v_sheet, w_sheet) of horizontal sheets
        self.half_step = half_step
        self.refine_at = 0.0               # particles longer than this are split once before the run starts

    def create(self, steps, deposit):
        kw = dict(half_step_init=self.half_step, history_len=max(1, steps), order=deposit)
        if self.compact is not None:
            return sic.Sim.sic_create_horizontal(self.nx, self.L, self.dt, *self.compact, **kw)
        s = sic.Sim.sic_create(self.nx, self.L, self.dt, self.counts, self.closed, self.winding, self.x, self.v,
                               self.w, **kw)
        if self.refine_at:
            s.sic_refine(self.refine_at)
        return s

    def full(self):
        """(x, v, w) per tracer."""
        if self.compact is None:
            return self.x, self.v, self.w
        xt, vs, ws = self.compact
        return np.tile(xt, vs.size), np.repeat(vs, xt.size), np.repeat(ws, xt.size)


def _quiet(state, r, sheets, tracers, nx, dt):
    """Horizontal sheets in the first part of a run; all share one position template."""
    if state == "landau":
        p = inputs.landau(0.005 + 0.01 * r.uniform(), 0.4 + 0.2 * r.uniform(), nx, sheets, tracers, dt=dt)
    else:
        p = inputs.two_stream(2.0 + r.uniform(), 0.05 + 0.1 * r.uniform(), 0.2, nx, sheets + sheets % 2, tracers,
                              eps=0.005 + 0.01 * r.uniform(), dt=dt)
    drift = 0.1 + 0.4 * r.uniform()
    x = p.x_template + r.uniform() * p.L
    return Tracers(nx, p.L, dt, p.counts, p.closed, p.winding, None, None, None, (x, p.v_sheet + drift, p.w_sheet))


def _folded(r, sheets, tracers, nx, dt, refined, device):
    """Sheets that counter-propagating waves have trapped and wound up until the longest
    particle is about half the box, where a run refines.  At 1024 x 4096 on 512 cells two
    thirds of the particles cross a cell edge, two fifths two or more, a fifth four or
    more, as in nonlinear Landau damping near t = 50.  The waves are given, so that the
    state takes no field solve."""
    k = 0.45 + 0.1 * r.uniform()
    L = 2.0 * math.pi / k
    vs = torch.linspace(-6.0, 6.0, sheets + 1, device=device, dtype=torch.float32)[:sheets] + 6.0 / sheets
    q = (torch.arange(tracers, device=device, dtype=torch.float32) + 0.5 * (1.0 + r.uniform())) * (L / tracers)
    x = q.repeat(sheets, 1).contiguous()
    v = vs[:, None].repeat(1, tracers).contiguous()
    amp, h = 0.57 + 0.06 * r.uniform(), 0.2
    waves = [(1.3, 0.7, 6.28 * r.uniform()), (0.5, 0.4, 6.28 * r.uniform()), (2.2, 0.5, 6.28 * r.uniform())]
    for i in range(400):
        t = i * h
        a = amp * (0.15 + 0.85 * math.exp(-0.2 * t))
        for omega, c, phase in waves:
            v -= h * a * c * (torch.sin(k * x + (phase - omega * t)) + torch.sin(k * x + (omega * t - phase)))
        x += h * v
        if i % 5 == 4:
            nxt = torch.roll(x, -1, 1)
            nxt[:, -1] += L
            longest = float((nxt - x).abs().max())
            if longest > 0.45 * L:
                break
    w = torch.exp(-0.5 * vs * vs)
    w = (w / w.sum() * (L / tracers)).double().cpu().numpy()
    drift = 0.1 + 0.4 * r.uniform()
    t = Tracers(nx, L, dt, np.full(sheets, tracers), np.ones(sheets), np.ones(sheets), x.double().cpu().numpy().ravel(),
                v.double().cpu().numpy().ravel() + drift, np.repeat(w, tracers))
    if refined:
        xd = x.double()
        nxt = torch.roll(xd, -1, 1)
        nxt[:, -1] += L
        t.refine_at = float(torch.topk((nxt - xd).abs().ravel(), 2).values.mean())  # the longest one alone
    return t


def _ragged(r, sheets, tracers, nx, dt):
    """Open and closed chains of any length in any order, a weight per tracer, points
    among the particles."""
    L = 4.0 * math.pi
    g = np.random.default_rng(r.next_u64())
    shape = np.random.default_rng(sheets * 8192 + tracers)  # sizes belong to the case, not to the seed
    counts = 2 + (shape.random(sheets) * (tracers - 1)).astype(np.int64)
    closed = (shape.random(sheets) < 0.7).astype(np.uint8)
    winding = np.where(closed == 1, np.where(shape.random(sheets) < 0.2, shape.integers(-1, 2, sheets), 1), 0)
    sheet = np.repeat(np.arange(sheets), counts)
    i = np.arange(counts.sum()) - np.repeat(np.cumsum(counts) - counts, counts)
    span = np.where(winding != 0, winding * L, (g.random(sheets) - 0.5) * L)
    x = (g.random(sheets) * L)[sheet] + span[sheet] * i / counts[sheet]
    x = x + (g.random(x.size) - 0.5) * L * np.minimum(0.3, 6.0 / counts[sheet])
    point = (i > 0) & (g.random(x.size) < 0.01)
    x[point] = x[np.flatnonzero(point) - 1]
    w = (0.5 + g.random(x.size)) * (L / x.size)
    v = (g.random(x.size) - 0.3) * 0.2
    return Tracers(nx, L, dt, counts, closed, winding, x, v, w, half_step=False)


def _tracers(case, seed):
    r = _rng(seed)
    if case["state"] == "folded":
        return _folded(r, case["sheets"], case["tracers"], case["nx"], case["dt"], case["refined"], _device())
    if case["state"] == "ragged":
        return _ragged(r, case["sheets"], case["tracers"], case["nx"], case["dt"])
    return _quiet(case["state"], r, case["sheets"], case["tracers"], case["nx"], case["dt"])


def _langmuir(case, seed):
    """A cold oscillation; several sheets share the charge."""
    r = _rng(seed)
    p = inputs.langmuir(case["tracers"], case["nx"], 0.5, 0.005 + 0.01 * r.uniform(), case["dt"], case["steps"])
    n = case["sheets"]
    v = 0.1 + 0.4 * r.uniform() + 0.01 * (np.arange(n) - 0.5 * (n - 1))
    return Tracers(case["nx"], p.L, case["dt"], np.full(n, case["tracers"]), np.ones(n), np.ones(n), None, None, None,
                   (p.x_template + r.uniform() * p.L, v, np.full(n, p.w_sheet[0] / n)))


def _members(case):
    """Sizes of a batch's members (the case's, not the seed's): powers of two over the
    serving mix's ranges and odd ones, about 20 million tracers at most each."""
    g = inputs.SplitMix64(0xBA7C4 + case["mix"])
    out = []
    for i in range(case["members"]):
        folded = bool(case["folded"]) and i % case["folded"] == 0
        m = 1 << (5 + int(g.uniform() * 6))
        n = 1 << (9 + int(g.uniform() * 8))
        nx = 1 << (6 + int(g.uniform() * 6))
        if g.uniform() < 0.3:
            m, n, nx = m - 2, n - 37, nx + 11
        cap = 1 << (21 if folded else 24)
        while m * n > cap:
            n //= 2
        two = not folded and g.uniform() < 0.5
        out.append(dict(state="folded" if folded else "two_stream" if two else "landau", sheets=m, tracers=n, nx=nx,
                        dt=case["dt"], refined=folded, deposit=BOX))
    return out


def _requests(case, seed):
    """Served requests: the serving mix's recipe at sizes up to 64 x 2048 and 256 cells."""
    g = inputs.SplitMix64(0x5EC5 + 977 * case["mix"])  # sizes and step counts
    r = _rng(seed)                                     # what fills them
    out = []
    for i in range(case["members"]):
        m, n, nx = 1 << (5 + int(2 * g.uniform())), 1 << (9 + int(3 * g.uniform())), 1 << (6 + int(3 * g.uniform()))
        steps = max(1, int(case["steps"] * (0.3 + 0.7 * g.uniform())))
        if g.uniform() < 0.4:
            kind, par = "landau", dict(alpha=math.exp(math.log(0.001) + r.uniform() * math.log(500.0)), k=0.3 + 0.3 * r.uniform())
        else:
            v0 = 1.0 + 2.0 * r.uniform()
            kind, par = "two_stream", dict(v0=v0, sigma=0.05 + 0.25 * r.uniform(), k=math.sqrt(3.0) / 2.0 * math.sqrt(0.5) / v0, eps=0.01)
        par.update(n_sheets=m, n_tracers=n, nx=nx, n_steps=steps, dt=case["dt"])
        out.append(inputs.Request(index=i, arrival=0.0, kind=kind, params=par))
    return out


# -------------------------------------------------------------------- run ----

def prepare(case, seed):
    kind = case["kind"]
    if kind == "run":
        return dict(case=case, tracers=_langmuir(case, seed))
    if kind == "serve":
        return dict(case=case, problems=[q.problem() for q in _requests(case, seed)])
    if kind == "batch":
        sims = [_tracers(m, seed + 1000 * i).create(case["steps"], m["deposit"]) for i, m in enumerate(_members(case))]
        return dict(case=case, sims=sims, batch=sic.Batch(sims))
    return dict(case=case, sim=_tracers(case, seed).create(case.get("steps", 1), case["deposit"]))


class _View:
    """Device memory of a simulation for torch.as_tensor (the simulation stays alive with it)."""

    def __init__(self, sim, address, n, typestr):
        self.sim = sim
        self.__cuda_array_interface__ = dict(shape=(n,), typestr=typestr, data=(address, False), version=3)


def _state(sim):
    """Positions (32-bit, as stored) and velocities where they lie, padding between sheets included."""
    pos, vel, off = sim.sic_device_state()
    n = int(off[-1]) + (int(sim.counts[-1]) + 31) // 32 * 32
    return dict(pos=torch.as_tensor(_View(sim, pos, n, "<i4"), device="cuda"),
                vel=torch.as_tensor(_View(sim, vel, n, "<f4"), device="cuda"))


def _history(h):
    return dict(field_energy=h[:, 0], kinetic_energy=h[:, 1], momentum=h[:, 2], charge=h[:, 3])


def run(state):
    case = state["case"]
    kind, steps = case["kind"], case.get("steps", 0)
    if kind == "run":
        sim = state["tracers"].create(steps, BOX)
        sim.sic_step(steps)
        h = sim.sic_history(steps)
        x, v = sim.sic_get_state()
        E = sim.sic_field()
        sim.sic_destroy()
        return dict(_history(h), x=x, v=v, E=E)
    if kind == "chunk":
        sim = state["sim"]
        sim.sic_step(steps)
        return dict(_history(sim.sic_history(steps)), E=sim.sic_field(), **_state(sim))
    if kind == "batch":
        state["batch"].sic_batch_step(steps)
        h = [s.sic_history(steps) for s in state["sims"]]
        return dict(_history(np.concatenate(h)), members=[_state(s) for s in state["sims"]])
    if kind == "diag":
        sim = state["sim"]
        mesh, rho = sim.sic_deposit()
        n0, j0 = sim.sic_moments(0)
        n1, j1 = sim.sic_moments(1)
        return dict(mesh=mesh, rho=rho, E=sim.sic_field(), n0=n0, j0=j0, n1=n1, j1=j1,
                    rho_k=sim.sic_spectrum(0), E_k=sim.sic_spectrum(1))
    server = sic.Server(hbm_budget=4 << 30, max_active=32, chunk_steps=32)
    for p in state["problems"]:
        server.sic_server_submit_horizontal(p, keep=True, history_len=p.n_steps)
    while server.sic_server_tick():
        pass
    results = sorted(server.sic_server_results(), key=lambda q: q["id"])
    hist = []
    for q, p in zip(results, state["problems"]):
        sim = sic.adopt_sim(q["sim"], p.nx, p.counts)
        hist.append(sim.sic_history(p.n_steps))
        sim.sic_destroy()
    server.sic_server_destroy()
    return dict(_history(np.concatenate(hist)), status=np.array([q["status"] for q in results]),
                steps=np.array([q["steps"] for q in results]), updates=np.array([q["segment_updates"] for q in results]))


def work(case):
    """A step reads and writes each tracer's position and velocity (4 bytes each), and reads
    a charge where charges are per tracer; about 40 operations for the push, the charge
    shares and the sums."""
    kind = case["kind"]
    if kind in ("run", "chunk"):
        n = case["sheets"] * case["tracers"] * (0.5 if case.get("state") == "ragged" else 1.0)
        per = 20 if case.get("refined") or case.get("state") == "ragged" else 16
        return dict(bytes=per * n * case["steps"], flops=40.0 * n * case["steps"])
    if kind == "diag":  # positions for the deposit, positions and velocities for each pair of moments
        n = case["sheets"] * case["tracers"]
        return dict(bytes=20.0 * n, flops=120.0 * n)
    if kind == "batch":
        n = [(m["sheets"] * m["tracers"], 20 if m["refined"] else 16) for m in _members(case)]
        return dict(bytes=float(case["steps"] * sum(a * b for a, b in n)), flops=40.0 * case["steps"] * sum(a for a, b in n))
    n = sum(q.work() for q in _requests(case, 0))
    return dict(bytes=16.0 * n, flops=40.0 * n)


# ------------------------------------------------------------------ exact ----
# The method's definitions in 64 bits with torch: none of the framework's code.

class _Plasma:
    """Sheets of tracers in cell units: x / dx, any number of windings."""

    def __init__(self, t: Tracers, deposit, device):
        x, v, w = (torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=device) for a in t.full())
        counts, closed, winding = t.counts, t.closed.astype(bool), t.winding.astype(np.int64)
        max_w = float(w.max())
        sigma = 2.0 ** math.floor(math.log2(2.0 ** 28 / max_w))
        while 2 * round(max_w * sigma * 0.5) > 2 ** 28:
            sigma *= 0.5
        self.t, self.deposit, self.device, self.nx, self.dx = t, deposit, device, t.nx, t.L / t.nx
        self.links(counts, closed, winding)
        half = torch.floor(w * sigma * 0.5 + 0.5)
        self.charge = float((half + torch.where(self.has, half[self.next], -half)).sum()) if deposit not in (NGP, CIC) else float(2 * half.sum())
        self.x, self.v, self.m = x / self.dx, v, w
        self.q = torch.where(self.has, 0.5 * (w + w[self.next]), 0.0)
        if t.refine_at:
            self.refine(t.refine_at / self.dx)
        self.solve()
        if t.half_step:
            self.v = self.v - 0.5 * t.dt * self.gather()

    def links(self, counts, closed, winding):
        """next[i]: the tracer that ends the particle starting at i; shift: its windings."""
        off = np.cumsum(counts) - counts
        nxt = np.arange(int(counts.sum())) + 1
        has = np.ones(nxt.size, dtype=bool)
        shift = np.zeros(nxt.size)
        last = off + counts - 1
        nxt[last] = off
        has[last] = closed
        shift[last] = np.where(closed, winding * self.nx, 0)
        self.counts, self.closed, self.winding, self.off = counts, closed, winding, off
        self.next = torch.as_tensor(nxt, device=self.device)
        self.has = torch.as_tensor(has, device=self.device)
        self.shift = torch.as_tensor(shift, device=self.device)

    def ends(self):
        return self.x, self.x[self.next] + self.shift

    def refine(self, length):
        a, b = self.ends()
        split = self.has & ((b - a).abs() > length)
        add = split.to(torch.int64)
        at = torch.arange(a.numel(), device=self.device) + torch.cumsum(add, 0) - add
        n = a.numel() + int(add.sum())
        new = at[split] + 1

        def grown(old, mid):
            out = torch.empty(n, dtype=torch.float64, device=self.device)
            out[at] = old
            out[new] = mid
            return out

        v1 = self.v[self.next]
        halved = torch.where(split, 0.5 * self.q, self.q)
        per_sheet = np.add.reduceat(add.cpu().numpy(), self.off)
        self.x, self.v = grown(self.x, 0.5 * (a + b)[split]), grown(self.v, 0.5 * (self.v + v1)[split])
        self.q = grown(halved, halved[split])
        self.m = self.q  # a tracer's mass is its particle's charge from now on
        self.links(self.counts + per_sheet, self.closed, self.winding)

    def kappa(self, a, b):
        """Slope of a piecewise-linear particle (Sec. 2.5), zero where it stays a box."""
        n = a.numel()
        prev = torch.zeros(n, dtype=torch.int64, device=self.device)
        at = torch.arange(n, device=self.device)
        prev[self.next] = at
        hp = torch.zeros(n, dtype=torch.bool, device=self.device)
        hp[self.next] = self.has
        hn = self.has[self.next]
        span = b - a
        lp, ls, ln = span[prev], span, span[self.next]
        qp, qs, qn = self.q[prev], self.q, self.q[self.next]
        cp, cn = -0.5 * (lp + ls), 0.5 * (ls + ln)  # centroids of the neighbours from this one's
        ok = self.has & hp & hn & (cp * cn < 0) & (lp != 0) & (ls != 0) & (ln != 0) & (span.abs() < self.nx) & (qs != 0)
        g = (qn / ln.abs() - qp / lp.abs()) / (cn - cp)
        k = g * ls.abs() / (2.0 * qs / ls.abs())
        return torch.where(ok, k, 0.0)

    def pieces(self, extra=()):
        """Every particle cut at the cell edges: yields (cell, lower and upper end in the cell,
        fractions of the particle's length there, indices of the particles)."""
        a, b = self.ends()
        lo, hi = torch.minimum(a, b), torch.maximum(a, b)
        i = torch.nonzero(self.has).ravel()
        lo, hi = lo[i], hi[i]
        first, last = torch.floor(lo), torch.floor(hi)
        k = 0
        while i.numel():
            c = first + k
            s0 = torch.clamp(lo - c, min=0.0)
            s1 = torch.clamp(hi - c, max=1.0)
            length = hi - lo
            point = length == 0
            t0 = torch.where(point, 0.0, (c + s0 - lo) / length)
            t1 = torch.where(point, 1.0, torch.where(last == c, 1.0, (c + s1 - lo) / length))
            t0 = torch.where(first == c, 0.0, t0)
            yield torch.remainder(c, self.nx).to(torch.int64), s0, s1, t0, t1, i
            k += 1
            go = last >= first + k
            i, lo, hi, first, last = i[go], lo[go], hi[go], first[go], last[go]

    def add(self, into, at, what):
        into += torch.bincount(at, weights=what, minlength=self.nx)[: self.nx]

    def mesh(self):
        rho = torch.zeros(self.nx, dtype=torch.float64, device=self.device)
        if self.deposit in (NGP, CIC):
            c = torch.remainder(self.x, self.nx)
            if self.deposit == NGP:
                self.add(rho, c.to(torch.int64) % self.nx, self.m)
            else:
                c = c - 0.5
                j = torch.floor(c)
                self.add(rho, torch.remainder(j, self.nx).to(torch.int64), self.m * (1 - (c - j)))
                self.add(rho, torch.remainder(j + 1, self.nx).to(torch.int64), self.m * (c - j))
            return rho
        a, b = self.ends()
        kappa = self.kappa(a, b) if self.deposit == LINEAR else None
        for c, s0, s1, t0, t1, i in self.pieces():
            q = self.q[i]
            if kappa is not None:
                kp = kappa[i]
                p = q * ((t1 + kp * t1 * (t1 - 1)) - (t0 + kp * t0 * (t0 - 1)))
            else:
                p = q * (t1 - t0)
            if self.deposit == FIRST:
                up = p * 0.5 * (s0 + s1)
                self.add(rho, c, p - up)
                self.add(rho, (c + 1) % self.nx, up)
            else:
                self.add(rho, c, p)
        return rho

    def solve(self):
        n = self.mesh() / self.dx
        self.rho = n - n.mean()
        step = 0.5 * (self.rho + torch.roll(self.rho, -1)) if self.deposit == FIRST else self.rho
        E = torch.cumsum(step, 0) * self.dx
        E = torch.roll(E, 1)
        E[0] = 0.0
        self.E = E - E.mean()

    def gather(self):
        c = torch.remainder(self.x, self.nx)
        j = torch.clamp(c.to(torch.int64), max=self.nx - 1)
        f = c - j
        return (1 - f) * self.E[j] + f * self.E[(j + 1) % self.nx]

    def step(self):
        """One step; its history row without the charge."""
        we = 0.5 * float((self.E * self.E).sum()) * self.dx
        v0 = self.v
        self.v = v0 + self.t.dt * self.gather()
        self.x = self.x + self.v * (self.t.dt / self.dx)
        self.solve()
        ke = 0.25 * float((self.m * (v0 * v0 + self.v * self.v)).sum())
        return we, ke, 0.5 * float((self.m * (v0 + self.v)).sum())

    def history(self, steps):
        h = np.array([self.step() for _ in range(steps)])
        return dict(field_energy=h[:, 0], kinetic_energy=h[:, 1], momentum=h[:, 2], charge=np.full(steps, self.charge))

    def velocities(self):
        """As stored: position units per step, sheets padded to 32 tracers with zeros."""
        pad = (self.counts + 31) // 32 * 32
        start = np.cumsum(pad) - pad
        at = np.arange(int(self.counts.sum())) + np.repeat(start - self.off, self.counts)
        out = np.zeros(int(pad.sum()))
        out[at] = self.v.cpu().numpy() * (self.t.dt / self.t.L * POS_UNITS)
        return out

    def unwrapped(self):
        """Positions along each sheet, the first one inside the box."""
        x = self.x.cpu().numpy()
        first = np.floor(x[self.off] / self.nx) * self.nx
        return (x - np.repeat(first, self.counts)) * self.dx

    def moments(self, weighting):
        """Number and current density (Sec. 2.3 on cells, Sec. 2.4 on nodes)."""
        n, j = (torch.zeros(self.nx, dtype=torch.float64, device=self.device) for _ in range(2))
        a, b = self.ends()
        va, vb = self.v, self.v[self.next]
        ma, mb = self.m, self.m[self.next]
        mean = (ma * va + mb * vb) / (ma + mb)
        back = b < a
        vl, vh = torch.where(back, vb, va), torch.where(back, va, vb)
        for c, s0, s1, t0, t1, i in self.pieces():
            q = self.q[i]
            p = q * (t1 - t0)
            if weighting == 0:
                self.add(n, c, p / self.dx)
                self.add(j, c, p * mean[i] / self.dx)
                continue
            # mean weight of the upper node, and of it with the velocity along the piece
            u0, u1 = vl[i] + (vh - vl)[i] * t0, vl[i] + (vh - vl)[i] * t1
            point = (a == b)[i]
            u0, u1 = torch.where(point, mean[i], u0), torch.where(point, mean[i], u1)
            up = 0.5 * (s0 + s1)
            upv = (2 * s0 * u0 + s0 * u1 + s1 * u0 + 2 * s1 * u1) / 6
            allv = 0.5 * (u0 + u1)
            self.add(n, c, p * (1 - up) / self.dx)
            self.add(n, (c + 1) % self.nx, p * up / self.dx)
            self.add(j, c, p * (allv - upv) / self.dx)
            self.add(j, (c + 1) % self.nx, p * upv / self.dx)
        return n.cpu().numpy(), j.cpu().numpy()


def exact(case, seed):
    kind, steps, device = case["kind"], case.get("steps", 0), _device()
    if kind == "serve":
        return None  # long nonlinear runs: neighbouring orbits part exponentially
    if kind == "run":
        p = _Plasma(_langmuir(case, seed), BOX, device)
        h = p.history(steps)
        return dict(h, x=p.unwrapped(), v=p.v.cpu().numpy(), E=p.E.cpu().numpy())
    if kind == "batch":
        rows, members = [], []
        for i, m in enumerate(_members(case)):
            p = _Plasma(_tracers(m, seed + 1000 * i), m["deposit"], device)
            rows.append(p.history(steps))
            members.append(dict(pos=None, vel=p.velocities()))
            del p
        return dict({k: np.concatenate([r[k] for r in rows]) for k in rows[0]}, members=members)
    p = _Plasma(_tracers(case, seed), case["deposit"], device)
    if kind == "chunk":
        return dict(p.history(steps), E=p.E.cpu().numpy(), pos=None, vel=p.velocities())
    (n0, j0), (n1, j1) = p.moments(0), p.moments(1)
    rho, E = p.rho.cpu().numpy(), p.E.cpu().numpy()
    return dict(mesh=None, rho=rho, E=E, n0=n0, j0=j0, n1=n1, j1=j1, rho_k=np.abs(np.fft.rfft(rho)),
                E_k=np.abs(np.fft.rfft(E)))
