"""The workloads this repository's speed is measured on, each through the public entry points.

listed() gives the named cases, draw() more of the same ranges, prepare() the handles and device
buffers that a program keeps, run() one pass, work() what a pass cannot do without, exact() the
same outputs from plain numpy in 64 bits.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2603_16623_gb300 import wake as wm
from paper_2603_16623_gb300 import workloads as W

# Keys of a case:
#   use        what one pass is:
#              "run"         reset + wake_run of one wake into host arrays (the README's first lines)
#              "solve"       preparation + march of all wakes in one batched submission, the four
#                            fields of every beam particle into device tensors
#              "stage"       one step of the beam-wake coupling: push, new binning, solve
#              "checkpoint"  load a ring state, march some slices, take the ring state
#              "query"       the fields of the current slice at arbitrary radii (device tensors)
#   march      "ab2", "rk4", "ions" (mobile hydrogen) or "grid" (adaptive beam grids)
#   precision  "mixed" or "fp64"
#   wakes      independent wakes in the batch, rings_lo..rings_hi rings (cells) each, evenly spread
#              over the logarithm
#   refined    1: the collider-like plasma and its two beams (20x finer cells near the axis);
#              2: geometric cells down to 1e-5 of the axis; 0: uniform cells, one driver
#   particles  beam particles per wake;  slices, dxi: the window;  queries: radii of "query"


def listed():
    return [
        # a single weak-driver wake: the smallest call there is, one CTA for 1000 dependent slices
        dict(name="linear_run", use="run", march="ab2", precision="mixed", wakes=1, rings_lo=200, rings_hi=200,
             refined=0, particles=20_000, slices=1000, dxi=0.02, n_b0=0.05, queries=0),
        # one collider-like blowout wake with driver and witness (the paper's setup), first half of the bubble
        dict(name="blowout_single", use="solve", march="ab2", precision="mixed", wakes=1, rings_lo=2000,
             rings_hi=2000, refined=1, particles=250_000, slices=800, dxi=0.005, n_b0=10.0, queries=0),
        # a parameter scan: independent wakes of 500 to 8000 rings in one submission (the bench's workload)
        dict(name="scan_batch", use="solve", march="ab2", precision="mixed", wakes=48, rings_lo=500, rings_hi=8000,
             refined=0, particles=120_000, slices=400, dxi=0.01, n_b0=5.0, queries=0),
        # the widest wake: 65,536 rings down to r = 1e-5, thousands of beam particles in a slice
        dict(name="large_single", use="solve", march="ab2", precision="mixed", wakes=1, rings_lo=65_536,
             rings_hi=65_536, refined=2, particles=500_000, slices=200, dxi=0.012, n_b0=10.0, queries=0),
        # a warm plasma restarted from a checkpoint: rings cross each other in every slice
        dict(name="warm_checkpoint", use="checkpoint", march="ab2", precision="mixed", wakes=1, rings_lo=6000,
             rings_hi=6000, refined=0, particles=20_000, slices=150, dxi=0.01, n_b0=1.0, queries=0),
        # one step of the coupled stage: the beams pushed, binned again, the wakes solved
        dict(name="stage_step", use="stage", march="ab2", precision="mixed", wakes=8, rings_lo=700, rings_hi=3000,
             refined=0, particles=240_000, slices=300, dxi=0.01, n_b0=2.0, queries=0),
        # the double-precision path: one wake, and a small scan
        dict(name="fp64_single", use="solve", march="ab2", precision="fp64", wakes=1, rings_lo=2000, rings_hi=2000,
             refined=0, particles=50_000, slices=250, dxi=0.01, n_b0=2.0, queries=0),
        dict(name="fp64_batch", use="solve", march="ab2", precision="fp64", wakes=24, rings_lo=500, rings_hi=8000,
             refined=0, particles=30_000, slices=80, dxi=0.02, n_b0=2.0, queries=0),
        # mobile ions, the Runge-Kutta integrator and adaptive beam grids, each on a scan
        dict(name="ions_batch", use="solve", march="ions", precision="mixed", wakes=24, rings_lo=500, rings_hi=4000,
             refined=0, particles=40_000, slices=250, dxi=0.01, n_b0=3.0, queries=0),
        dict(name="rk4_batch", use="solve", march="rk4", precision="mixed", wakes=24, rings_lo=500, rings_hi=8000,
             refined=0, particles=40_000, slices=96, dxi=0.02, n_b0=3.0, queries=0),
        dict(name="grid_batch", use="solve", march="grid", precision="mixed", wakes=24, rings_lo=500, rings_hi=8000,
             refined=0, particles=40_000, slices=250, dxi=0.01, n_b0=3.0, queries=0),
        # a field map of the current slice: many radii at once
        dict(name="field_query", use="query", march="ab2", precision="mixed", wakes=1, rings_lo=2000, rings_hi=2000,
             refined=0, particles=50_000, slices=200, dxi=0.01, n_b0=2.0, queries=20_000),
    ]


def draw(rng):
    def lg(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    use, march, precision = rng.choice([
        ("solve", "ab2", "mixed"), ("solve", "ab2", "mixed"), ("solve", "ab2", "mixed"), ("solve", "ab2", "fp64"),
        ("solve", "ions", "mixed"), ("solve", "rk4", "mixed"), ("solve", "grid", "mixed"), ("solve", "ions", "fp64"),
        ("solve", "rk4", "fp64"), ("run", "ab2", "mixed"), ("stage", "ab2", "mixed"), ("checkpoint", "ab2", "mixed"),
        ("query", "ab2", "mixed")])
    hi = 4000 if march == "ions" else 8000
    if use == "run":
        wakes, lo, hi, slices, parts, dxi, nb0 = 1, lg(150, 1500), 0, lg(200, 1000), lg(2000, 50_000), 0.02, 0.05
    elif use == "solve":
        wakes = lg(1, 32)
        lo = lg(200, hi)
        hi = lg(lo, hi) if wakes > 1 else lo
        dxi, nb0 = 0.01, rng.uniform(0.5, 5.0)
        parts = lg(2000, 100_000)
        slices = lg(40, 300) if march == "ab2" and precision == "mixed" else lg(20, 100)
    elif use == "stage":
        wakes, lo, slices, parts, dxi, nb0 = lg(1, 8), lg(300, 1500), lg(50, 300), lg(20_000, 240_000), 0.01, 2.0
        hi = 2 * lo
    elif use == "checkpoint":
        wakes, lo, slices, parts, dxi, nb0 = 1, lg(400, 16_000), lg(30, 150), lg(2000, 50_000), 0.01, 1.0
    else:
        wakes, lo, slices, parts, dxi, nb0 = 1, lg(200, 8000), 200, lg(2000, 50_000), 0.01, 2.0
    if wakes == 1:
        hi = lo
    parts = min(parts, 900 * slices)  # (a slice holds at most 8192)
    return dict(use=use, march=march, precision=precision, wakes=wakes, rings_lo=lo, rings_hi=hi, refined=0,
                particles=parts, slices=slices, dxi=dxi, n_b0=round(nb0, 3),
                queries=lg(100, 60_000) if use == "query" else 0)


# ----------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------
def _ring_counts(case):
    n, lo, hi = case["wakes"], case["rings_lo"], case["rings_hi"]
    return [int(round(lo * (hi / lo) ** ((i + 0.5) / n))) if hi > lo else lo for i in range(n)]


def _problems(case, seed):
    """The wakes of a case (workloads.Wake), beams drawn from the seed."""
    out = []
    window = case["slices"] * case["dxi"]
    for i, n in enumerate(_ring_counts(case)):
        s = (seed * 1009 + i * 7919) % (1 << 31)
        rng = np.random.Generator(np.random.PCG64(s))
        n_mp, nb0 = case["particles"], case["n_b0"]
        if case["refined"]:
            edges = W.edges_refined(n * 288 // 2000, 0.05, n - n * 288 // 2000, 6.0) if case["refined"] == 1 else \
                W.edges_geometric(n, 1e-5, 6.0)
            sz = 0.5 if case["refined"] == 1 else 0.3
            drv = W.gaussian_beam(n_mp * 4 // 5, nb0, 0.1, sz, 4 * sz, seed=s)
            wit = W.gaussian_beam(n_mp - n_mp * 4 // 5, 0.0, 1e-3 if case["refined"] == 1 else 1e-4, 0.5 * sz,
                                  min(10 * sz, 0.8 * window), seed=s + 1,
                                  total=0.42 * W.gaussian_charge(nb0, 0.1, sz))
            beams = [drv, wit]
        else:
            # a driver centred in the front half of the window
            if nb0 < 0.1:
                sr, sz, xc = 0.5, 1.0, 4.0
            else:
                nb0 *= rng.uniform(0.5, 1.5)
                sr = rng.uniform(0.1, 0.5)
                sz = rng.uniform(0.06, 0.12) * window
                xc = 4.0 * sz
            edges = W.edges_uniform(n, 5.0 if nb0 < 0.1 else max(6.0, 6.0 * math.sqrt(nb0) * sr))
            beams = [W.gaussian_beam(n_mp, nb0, sr, sz, xc, seed=s)]
        out.append(W.Wake(f"case{i}", edges, beams, case["dxi"], case["slices"],
                          ions=(1.0, 1836.0) if case["march"] == "ions" else None,
                          integrator="rk4" if case["march"] == "rk4" else "ab2",
                          grid_nr=32 if case["march"] == "grid" else 0))
    return out


def _warm_state(wk, seed):
    """Ring radii around the cell centres and thermal momenta."""
    rng = np.random.Generator(np.random.PCG64(seed + 17))
    c = 0.5 * (wk.edges[1:] + wk.edges[:-1])
    return np.abs(c + 0.3 * np.diff(wk.edges) * rng.standard_normal(wk.n_rings)), \
        0.1 * rng.standard_normal(wk.n_rings)


def _radii(case, wk, seed):
    return np.random.Generator(np.random.PCG64(seed + 29)).uniform(0.0, wk.edges[-1], case["queries"])


_STAGE_DT, _STAGE_GAMMA = 0.5, 2000.0


def prepare(case, seed):
    probs = _problems(case, seed)
    gs = [wm.Wake.from_workload(p, precision=case["precision"]) for p in probs]
    st = {"case": case, "gs": gs}
    dt = torch.float64 if case["precision"] == "fp64" else torch.float32
    n_out = case["queries"] if case["use"] == "query" else sum(g.n_beam for g in gs)
    # one tensor per field, every wake's particles in their place
    st["out"] = {k: torch.zeros(n_out, dtype=dt, device="cuda") for k in ("ez", "wr", "bt", "psi")}
    off, st["views"] = 0, []
    for g in gs:
        st["views"].append({k: v[off:off + g.n_beam] for k, v in st["out"].items()})
        off += g.n_beam
    if case["use"] == "checkpoint":
        st["rho"], st["ur"] = _warm_state(probs[0], seed)
    if case["use"] == "query":
        st["r"] = torch.from_numpy(_radii(case, probs[0], seed)).to("cuda")
        gs[0].step_slices(case["slices"] // 2)
    if case["use"] == "stage":
        for g, p in zip(gs, probs):
            r = np.concatenate([b.r for b in p.beams])
            z = np.zeros(r.shape[0])
            g.set_beam_phase_space(r, z, z, z, np.full(r.shape[0], _STAGE_GAMMA))
        wm.wake_batch_reset_run(gs)
    return st


def run(st):
    case, gs = st["case"], st["gs"]
    use = case["use"]
    if use == "run":
        gs[0].reset()
        status, ez, wr, _ = gs[0].run()
        return {"status": status, "ez": ez, "wr": wr}
    if use == "checkpoint":
        g = gs[0]
        g.set_ring_state(0, st["rho"], st["ur"])
        g.step_slices(case["slices"])
        rho, ur = g.ring_state()
        return {"rho": rho.astype(g.dtype), "ur": ur.astype(g.dtype)}
    if use == "query":
        gs[0].fields_at_device(st["r"], st["out"])
        return st["out"]
    if use == "stage":
        wm.wake_batch_push_beam(gs, _STAGE_DT)
    wm.wake_batch_reset_run(gs)
    for g, v in zip(gs, st["views"]):
        g.beam_fields_device(v)
    return st["out"]


# arithmetic of one ring in one slice: the operations of the method's formulas (one slice evaluation and the
# push; four evaluations with RK4; both species with ions)
_FLOPS = {"ab2": 117.0, "rk4": 468.0, "ions": 2 * 97.5, "grid": 117.0}


def work(case):
    rings = float(sum(_ring_counts(case)))
    parts = float(case["particles"] * case["wakes"])
    real = 8 if case["precision"] == "fp64" else 4
    if case["use"] == "query":
        return {"bytes": case["queries"] * (8 + 4 * real) + rings * 5 * real, "flops": rings * 104.0 + case["queries"] * 20.0}
    ring_slices = rings * case["slices"]
    flops = ring_slices * _FLOPS[case["march"]] + parts * 20.0
    if case["use"] == "checkpoint":
        return {"bytes": rings * (2 * 8 + 2 * 8) + parts * 16, "flops": flops}
    n_out = 2 if case["use"] == "run" else 4
    by = parts * (24 + n_out * real) + rings * 8 * (2 if case["march"] == "ions" else 1)
    if case["use"] == "stage":
        by += parts * 96
    return {"bytes": by, "flops": flops}


# ----------------------------------------------------------------------------
# the same in plain numpy, 64 bits
# ----------------------------------------------------------------------------
def _excl(a):
    out = np.zeros(a.shape[0] + 1)
    np.cumsum(a, out=out[1:])
    return out


def _prefix_maps(m00, m01, m10, m11):
    """Inclusive products M_p ... M_0 of 2x2 matrices (log-step scan)."""
    n, d = m00.shape[0], 1
    a, b, c, e = m00.copy(), m01.copy(), m10.copy(), m11.copy()
    while d < n:
        x0, x1, x2, x3 = a[d:], b[d:], c[d:], e[d:]
        y0, y1, y2, y3 = a[:-d], b[:-d], c[:-d], e[:-d]
        z = x0 * y0 + x1 * y2, x0 * y1 + x1 * y3, x2 * y0 + x3 * y2, x2 * y1 + x3 * y3
        a[d:], b[d:], c[d:], e[d:] = z
        d *= 2
    return a, b, c, e


def _solve_bp(r, A, B, C):
    """a_k, b_k (k = 0..n) of B = a r + b / r between the rings, b_0 = 0, a_n = 0."""
    n = r.shape[0]
    h = 0.5 * A
    f = _prefix_maps(1 + h * r, h / r, -h * r ** 3, 1 - h * r)
    R0, R1 = np.concatenate([[1.0], f[0]]), np.concatenate([[0.0], f[2]])
    i = [x[::-1] for x in (1 - h * r, -h / r, h * r ** 3, 1 + h * r)]
    g = _prefix_maps(*i)
    D0, D1 = np.concatenate([g[1][::-1], [0.0]]), np.concatenate([g[3][::-1], [1.0]])
    s0 = 0.25 * (2 * B + A * C)
    s1 = 0.25 * r * (4 * C - 2 * B * r - A * C * r)
    q0, q1, d0, d1 = R0[1:], R1[1:], D0[1:], D1[1:]
    wr = q0 * d1 - q1 * d0
    ga, de = (s0 * d1 - s1 * d0) / wr, (q0 * s1 - q1 * s0) / wr
    G = np.concatenate([np.cumsum(ga[::-1])[::-1], [0.0]])
    H = _excl(de)
    a, b = -G * R0 + H * D0, -G * R1 + H * D1
    a[n], b[n] = 0.0, H[n]
    return a, b


class _Beam:
    """The binned beam: per slice the radius-sorted particles and the charge inside."""

    def __init__(self, wk, xi=None, r=None):
        xi = np.concatenate([b.xi for b in wk.beams]) if xi is None else xi
        self.r = np.concatenate([b.r for b in wk.beams]) if r is None else r
        self.qw = np.concatenate([b.q * b.w for b in wk.beams])
        self.species = np.concatenate([np.full(b.n, k) for k, b in enumerate(wk.beams)])
        sl = np.floor(xi / wk.dxi + 0.5)
        self.inside = (sl >= 0) & (sl < wk.n_steps)
        order = np.lexsort((self.r, np.where(self.inside, sl, wk.n_steps)))
        self.order = order[:int(self.inside.sum())]
        self.off = np.searchsorted(sl[self.order], np.arange(wk.n_steps + 1), side="left")
        self.norm = 1.0 / (2.0 * math.pi * wk.dxi)

    def at(self, s):
        if s >= self.off.shape[0] - 1:
            return np.zeros(0, dtype=np.int64), np.zeros(0), np.zeros(1)
        k = self.order[self.off[s]:self.off[s + 1]]
        return k, self.r[k], _excl(self.qw[k])

    def field(self, s, x, weight=1.0):
        """B_theta of slice s's particles at radii x > 0."""
        _, r, q = self.at(s)
        return weight * self.norm * q[np.searchsorted(r, x, side="left")] / x


class _Column:
    """One species' rings, cell weights and (electrons only) the analytic ion column."""

    def __init__(self, wk):
        e = wk.edges
        c, d = 0.5 * (e[1:] + e[:-1]), np.diff(e)
        self.w, self.wh = wk.density * c * d, wk.density * (0.5 * c * d - 0.125 * d * d)
        self.c, self.rm, self.n0 = c, e[-1], wk.density

    def ion(self, x):
        rm, n0 = self.rm, self.n0
        inside = 0.5 * n0 * np.minimum(x, rm) ** 2
        c0 = 0.25 * n0 * rm * rm - 0.5 * n0 * rm * rm * math.log(rm)
        with np.errstate(divide="ignore"):
            psi = np.where(x <= rm, c0 - 0.25 * n0 * x * x, -0.5 * n0 * rm * rm * np.log(np.maximum(x, 1e-300)))
        return inside, psi


def _sources(w, r, u, pb, g, dpr, dpz, bb):
    wr = w / r
    A = wr / pb
    B = -wr * g * dpr / pb ** 2 + wr * bb / pb + w / (r * r) * u * u / pb ** 2 + wr * u * u * dpr / pb ** 3 - \
        wr * u * dpz / pb ** 2
    return A, B, -wr * (g / pb - 1 - u * u / pb ** 2)


def _bp_rings(a, b, r):
    return 0.5 * ((a[:-1] + a[1:]) * r + (b[:-1] + b[1:]) / r)


def _slice(col, r, u, w, wh, bb):
    """The fields of one slice at sorted rings; returns what the pushes and the off-ring fields need."""
    ln = np.log(r)
    S, L = _excl(w), _excl(w * ln)
    I, ion = col.ion(r)
    psi = (L[-1] - L[:-1]) + S[:-1] * ln + ion
    dpr = (S[:-1] + wh - I) / r
    pb = 1 + psi
    g = (1 + u * u + pb * pb) / (2 * pb)
    t = w * u / (r * pb)
    T = _excl(t)
    dpz = -((T[-1] - T[1:]) + (1 - wh / w) * t)
    a, b = _solve_bp(r, *_sources(w, r, u, pb, g, dpr, dpz, bb))
    return dict(pb=pb, g=g, dpr=dpr, bp=_bp_rings(a, b, r), S=S, L=L, T=T, a=a, b=b)


def _off_rings(col, F, r, x):
    """psi, d_rho psi, d_zeta psi, B^(p) at radii x >= 0 off the rings."""
    k = np.searchsorted(r, x, side="left")
    I, ion = col.ion(x)
    ax = x > 0
    xs = np.where(ax, x, 1.0)
    psi = F["L"][-1] - F["L"][k] + F["S"][k] * np.log(xs) + ion
    return psi, np.where(ax, (F["S"][k] - I) / xs, 0.0), -(F["T"][-1] - F["T"][k]), \
        np.where(ax, F["a"][k] * xs + F["b"][k] / xs, 0.0)


def _enclosed(beam, s, x):
    """The beam's own field at its particles: charge strictly inside."""
    _, r, q = beam.at(s)
    xs = np.where(x > 0, x, 1.0)
    return np.where(x > 0, beam.norm * q[np.searchsorted(r, x, side="left")] / xs, 0.0)


def _reflect(r, u):
    s = np.where(r < 0, -1.0, 1.0)
    return r * s, u * s, s


class _Grids:
    """Adaptive beam grids: nr cells per species out to (1 + 1/nr) of its largest radius."""

    def __init__(self, wk, beam):
        self.nr, self.beam = wk.grid_nr, beam
        self.R = [(1 + 1 / self.nr) * max(b.r.max(), 1e-12) for b in wk.beams]

    def deposit(self, s):
        k, r, _ = self.beam.at(s)
        self.B = []
        for b, R in enumerate(self.R):
            x = np.arange(self.nr + 1) * (R / self.nr)
            m = self.beam.species[k] == b
            q = np.zeros(self.nr + 1)
            np.add.at(q, np.minimum(np.searchsorted(x, r[m], side="right"), self.nr), self.beam.qw[k[m]])
            B = np.zeros(self.nr + 1)
            B[1:] = self.beam.norm * np.cumsum(q)[1:] / x[1:]
            self.B.append((x, B))

    def field(self, x):
        v = np.zeros_like(x)
        for xs, B in self.B:
            v += np.where(x >= xs[-1], B[-1] * xs[-1] / np.maximum(x, 1e-300), np.interp(x, xs, B))
        return v


def _march(case, wk, beam, state=None, stop=None, query=None):
    """Marches one wake; returns the beam fields, the final (rho, u) by ring id, and query fields."""
    col = _Column(wk)
    n, h = wk.n_rings, wk.dxi
    r, u = (col.c.copy(), np.zeros(n)) if state is None else (state[0].copy(), state[1].copy())
    ids = np.arange(n)
    fr0 = fu0 = None
    out = {k: np.zeros(beam.r.shape[0]) for k in ("ez", "wr", "bt", "psi")}
    grids = _Grids(wk, beam) if wk.grid_nr else None

    def put(s, F, rs):
        k, x, _ = beam.at(s)
        if grids:
            for b, (xs, _) in enumerate(grids.B):
                psi, dpr, dpz, bp = _off_rings(col, F, rs, xs)
                m = beam.species[k] == b
                bt = np.where(xs > 0, bp + grids.field(xs), 0.0)
                for key, v in (("ez", -dpz), ("wr", -dpr), ("bt", bt), ("psi", psi)):
                    out[key][k[m]] = np.interp(x[m], xs, v)
            return
        psi, dpr, dpz, bp = _off_rings(col, F, rs, x)
        out["ez"][k], out["wr"][k], out["bt"][k], out["psi"][k] = -dpz, -dpr, bp + _enclosed(beam, s, x), psi

    def derivs(rr, uu, idr, src):
        rr, uu, sg = _reflect(rr, uu)
        o = np.argsort(rr, kind="stable")
        F = _slice(col, rr[o], uu[o], col.w[idr[o]], col.wh[idr[o]], src(rr[o]))
        fr, fu = np.empty_like(rr), np.empty_like(rr)
        fr[o] = sg[o] * uu[o] / F["pb"]
        fu[o] = sg[o] * (F["g"] * F["dpr"] / F["pb"] - (F["bp"] + src(rr[o])))
        return fr, fu

    for s in range(wk.n_steps if stop is None else stop + 1):
        o = np.argsort(r, kind="stable")
        r, u, ids = r[o], u[o], ids[o]
        if fr0 is not None:
            fr0, fu0 = fr0[o], fu0[o]
        if grids:
            grids.deposit(s)
        bb = grids.field(r) if grids else beam.field(s, r)
        F = _slice(col, r, u, col.w[ids], col.wh[ids], bb)
        if stop is not None and s == stop:
            psi, dpr, dpz, bp = _off_rings(col, F, r, query)
            return {"ez": -dpz, "wr": -dpr, "bt": bp + _enclosed(beam, s, query), "psi": psi}
        put(s, F, r)
        if not (np.all(F["pb"] > 0) and np.all(np.isfinite(F["bp"]))):
            break
        fr, fu = u / F["pb"], F["g"] * F["dpr"] / F["pb"] - (F["bp"] + bb)
        if wk.integrator == "rk4":
            mid = lambda x, s=s: beam.field(s, x, 0.5) + beam.field(s + 1, x, 0.5)  # noqa: E731
            end = lambda x, s=s: beam.field(s + 1, x)  # noqa: E731
            r2, u2 = derivs(r + h / 2 * fr, u + h / 2 * fu, ids, mid)
            r3, u3 = derivs(r + h / 2 * r2, u + h / 2 * u2, ids, mid)
            r4, u4 = derivs(r + h * r3, u + h * u3, ids, end)
            r, u, _ = _reflect(r + h / 6 * (fr + 2 * r2 + 2 * r3 + r4), u + h / 6 * (fu + 2 * u2 + 2 * u3 + u4))
            continue
        gr, gu = (fr, fu) if fr0 is None else (1.5 * fr - 0.5 * fr0, 1.5 * fu - 0.5 * fu0)
        r, u, sg = _reflect(r + h * gr, u + h * gu)
        fr0, fu0 = fr * sg, fu * sg
    rho, ur = np.empty(n), np.empty(n)
    rho[ids], ur[ids] = r, u
    return out, rho, ur


def _gather(x, r, F, F0, edge, Fe, outside):
    """The other species' ring values at radii x: linear between its rings, from the axis value F0, to the
    outside value at the plasma edge, exact outside values beyond."""
    if edge > r[-1]:
        xs, fs = np.concatenate([[0.0], r, [edge]]), np.concatenate([[F0], F, [Fe]])
    else:
        xs, fs = np.concatenate([[0.0], r]), np.concatenate([[F0], F])
    return np.where((x <= r[-1]) | (x < edge), np.interp(x, xs, fs), outside)


def _march_ions(case, wk, beam):
    """Electrons and ions as two ring species."""
    col = _Column(wk)
    n, h, edge = wk.n_rings, wk.dxi, wk.edges[-1]
    z, mass = wk.ions
    qm = (-1.0, z / mass)
    sp = [dict(r=col.c.copy(), u=np.zeros(n), w=sgn * col.w, wh=sgn * col.wh, f=None) for sgn in (1.0, -1.0)]
    out = {k: np.zeros(beam.r.shape[0]) for k in ("ez", "wr", "bt", "psi")}
    for s in range(wk.n_steps):
        for p in sp:
            o = np.argsort(p["r"], kind="stable")
            p.update(r=p["r"][o], u=p["u"][o], w=p["w"][o], wh=p["wh"][o],
                     f=None if p["f"] is None else [x[o] for x in p["f"]])
            ln = np.log(p["r"])
            p["S"], p["L"] = _excl(p["w"]), _excl(p["w"] * ln)
            p["psi"] = (p["L"][-1] - p["L"][:-1]) + p["S"][:-1] * ln
            p["dpr"] = (p["S"][:-1] + p["wh"]) / p["r"]
            p["bb"] = beam.field(s, p["r"])
        for p, q, k in ((sp[0], sp[1], qm[0]), (sp[1], sp[0], qm[1])):
            r, St = p["r"], q["S"][-1]
            psi = p["psi"] + _gather(r, q["r"], q["psi"], q["L"][-1], edge, St * math.log(edge), St * np.log(r))
            p["dprt"] = p["dpr"] + _gather(r, q["r"], q["dpr"], 0.0, edge, St / edge, St / r)
            p["pb"] = 1 - k * psi
            p["g"] = (1 + p["u"] ** 2 + p["pb"] ** 2) / (2 * p["pb"])
            t = p["w"] * p["u"] / (r * p["pb"])
            p["T"] = _excl(t)
            p["dpz"] = -((p["T"][-1] - p["T"][1:]) + (1 - p["wh"] / p["w"]) * t)
        el, io = sp
        dpz = el["dpz"] + _gather(el["r"], io["r"], io["dpz"], -io["T"][-1], edge, 0.0, 0.0)
        a, b = _solve_bp(el["r"], *_sources(el["w"], el["r"], el["u"], el["pb"], el["g"], el["dprt"], dpz, el["bb"]))
        el["bp"] = _bp_rings(a, b, el["r"])
        io["bp"] = _gather(io["r"], el["r"], el["bp"], 0.0, edge, b[-1] / edge, b[-1] / io["r"])
        k, x, _ = beam.at(s)
        xs = np.maximum(x, 1e-300)
        i = [np.searchsorted(p["r"], x, side="left") for p in sp]
        St = sum(p["S"][j] for p, j in zip(sp, i))
        out["psi"][k] = sum(p["L"][-1] - p["L"][j] for p, j in zip(sp, i)) + St * np.log(xs)
        out["wr"][k] = -St / xs
        out["ez"][k] = sum(p["T"][-1] - p["T"][j] for p, j in zip(sp, i))
        out["bt"][k] = a[i[0]] * x + b[i[0]] / xs + _enclosed(beam, s, x)
        if not all(np.all(p["pb"] > 0) for p in sp):
            break
        for p, c in zip(sp, qm):
            fr, fu = p["u"] / p["pb"], -c * (p["g"] * p["dprt"] / p["pb"] - (p["bp"] + p["bb"]))
            gr, gu = (fr, fu) if p["f"] is None else (1.5 * fr - 0.5 * p["f"][0], 1.5 * fu - 0.5 * p["f"][1])
            p["r"], p["u"], sg = _reflect(p["r"] + h * gr, p["u"] + h * gu)
            p["f"] = [fr * sg, fu * sg]
    return out, None, None


def _push(wk, out, dt):
    """One Boris step from the start of the stage (y = 0, u = (0, 0, gamma)): new xi and r."""
    q = np.concatenate([np.full(b.n, b.q) for b in wk.beams])
    x, xi = np.concatenate([b.r for b in wk.beams]), np.concatenate([b.xi for b in wk.beams])
    h = 0.5 * q * dt
    er, by = out["wr"] + out["bt"], out["bt"]
    on = x > 0
    ex, by = np.where(on, er, 0.0), np.where(on, by, 0.0)
    ux, uz = h * ex, _STAGE_GAMMA + h * out["ez"]
    t = h * by / np.sqrt(1 + ux * ux + uz * uz)
    sn = 2 * t / (1 + t * t)
    px, pz = ux - uz * t, uz + ux * t
    ux, uz = ux - pz * sn, uz + px * sn
    ux, uz = ux + h * ex, uz + h * out["ez"]
    gam = np.sqrt(1 + ux * ux + uz * uz)
    return xi + dt * (1 + ux * ux) / (gam * (gam + uz)), np.abs(x + dt * ux / gam)


_EXACT_S = 25.0  # (about twice the seconds it takes) leave out what would take longer


def exact(case, seed):
    evals = sum((6e-4 + n * 6.5e-7) * case["slices"] for n in _ring_counts(case))
    evals *= {"ab2": 1, "grid": 1.3, "ions": 2.0, "rk4": 4.4}[case["march"]] * (2 if case["use"] == "stage" else 1)
    if evals > _EXACT_S:
        return None
    with np.errstate(all="ignore"):
        got = []
        for wk in _problems(case, seed):
            beam = _Beam(wk)
            if case["use"] == "checkpoint":
                _, rho, ur = _march(case, wk, beam, _warm_state(wk, seed))
                return {"rho": rho, "ur": ur}
            if case["use"] == "query":
                return _march(case, wk, beam, stop=case["slices"] // 2, query=_radii(case, wk, seed))
            m = _march_ions if case["march"] == "ions" else _march
            out = m(case, wk, beam)[0]
            if case["use"] == "stage":
                out = _march(case, wk, _Beam(wk, *_push(wk, out, _STAGE_DT)))[0]
            got.append(out)
    if case["use"] == "run":
        return {"status": None, "ez": got[0]["ez"], "wr": got[0]["wr"]}
    return {k: np.concatenate([o[k] for o in got]) for k in ("ez", "wr", "bt", "psi")}
