"""The work that the performance of this framework is judged by.

Each case is one thing that a program built on the framework does: a context
advanced through some steps and its fields read, a run resumed from a
checkpoint, a whole request from host arrays to host arrays, a batch of
specimens, the neighbour service and the material-point service.  The sizes
are those of the repository's workloads (`specimen.py`) and of the ranges its
batched and served forms draw from.

listed()            the cases, with what each stands for
draw(rng)           one more case of the same ranges
prepare(case, seed) inputs and the objects that a program keeps
run(state)          one pass
work(case)          bytes and operations that a pass cannot do without
exact(case, seed)   the same outputs from plain torch in FP64

Outputs of FP64 contexts are handed back in FP64, those of mixed-precision
contexts in FP32, the precision of that path's pair sums and stresses.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1901_07374_gb300 import specimen as S
from paper_1901_07374_gb300 import tlsph

FIELDS = ("U", "V", "F", "SIGMA", "FORCE", "EPSP", "DAMAGE")
DIAGS = ("kinetic_energy", "internal_energy", "max_epsp", "max_damage")


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # The smallest specimen (the Cockcroft-Latham bar of 2048 particles) in the binding's default
        # precision, watched through its diagnostics: launches and latency.
        dict(name="fp64_bar_2k", kind="bar", precision="fp64", damage="cl", nx=8, ny=8, nz=32, watch=5, steps=20),
        # The default Taylor impact on the rigid wall, from contact on: yield, Johnson-Cook hardening with
        # rate, ragged lattice rows.
        dict(name="fp64_taylor_12k", kind="taylor", precision="fp64", n=12000, steps=40),
        # A bar of odd dimensions in which every particle flows, resumed from a checkpoint: the FP64
        # radial return with Cockcroft-Latham damage (an eigenvalue per particle and step).
        dict(name="fp64_flow_43k", kind="flow", precision="fp64", damage="cl", nx=19, ny=21, nz=107, steps=10),
        # A quarter of the Johnson-Cook bar in FP64: throughput of the accurate path.
        dict(name="fp64_bar_256k", kind="bar", precision="fp64", damage="jc", nx=40, ny=40, nz=160, watch=0,
             steps=5),
        # The smallest specimen in mixed precision, watched through its diagnostics.
        dict(name="mixed_bar_2k", kind="bar", precision="mixed", damage="cl", nx=8, ny=8, nz=32, watch=5, steps=20),
        # A bar of odd dimensions in the middle of the batched form's range, plastic flow, resumed from a
        # checkpoint: the mixed path's FP64 return on every particle.
        dict(name="mixed_flow_43k", kind="flow", precision="mixed", damage="cl", nx=19, ny=21, nz=107, steps=20),
        # The GTN notched bar at its full size in plastic flow, resumed from a checkpoint: Newton returns
        # on every particle, neighbour slices that are partly explicit.
        dict(name="mixed_gtn_456k", kind="notched", precision="mixed", radius=5e-3, height=20e-3, notch=1e-3,
             spacing=0.15e-3, steps=10),
        # The headline workload, the 1.02M-particle Johnson-Cook bar, with the plan the autotuner settles on.
        dict(name="mixed_bar_1m", kind="bar", precision="mixed", damage="jc", nx=40, ny=40, nz=640, watch=0, steps=20,
             tuned=True),
        # A served request as a whole: a Taylor cylinder from host arrays through creation and its first
        # steps to fields in host memory, context released.
        dict(name="request_taylor_60k", kind="request", precision="mixed", n=60000, steps=50),
        # Sixteen bars of the batched workload (2000 to 200000 particles) advanced together from a graph.
        dict(name="batch_16_bars", kind="batch", count=16, n_min=2000, n_max=200000, steps=20),
        # The allocation-free neighbour service on a body close to its particle limit.
        dict(name="neighbors_209k", kind="neighbors", nx=37, ny=53, nz=107),
        # Material points of a GTN parameter study.
        dict(name="points_gtn_200k", kind="points", damage="gtn", n=200003),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _box(rng, lo, hi):
    n = _log(rng, lo, hi)
    nx = max(5, round((n / rng.uniform(2.0, 8.0)) ** (1.0 / 3.0)))
    ny = max(5, nx + rng.randint(-2, 3))
    return dict(nx=nx, ny=ny, nz=max(6, round(n / (nx * ny))))


def draw(rng):
    kind = rng.choice(("bar", "bar", "bar", "flow", "flow", "taylor", "taylor", "notched", "request", "batch",
                       "neighbors", "points"))
    precision = rng.choice(("fp64", "mixed"))
    big = 100000 if precision == "fp64" else 600000
    if kind == "bar":
        watch = rng.choice((0, 0, 3))
        return dict(kind=kind, precision=precision, damage=rng.choice(("cl", "jc")), **_box(rng, 500, big),
                    watch=watch, steps=rng.randint(3, 8))
    if kind == "flow":
        return dict(kind=kind, precision=precision, damage="cl", **_box(rng, 500, big), steps=rng.randint(5, 12))
    if kind == "taylor":
        return dict(kind=kind, precision=precision, n=int(_log(rng, 2000, big / 2)), steps=rng.randint(5, 25))
    if kind == "notched":
        return dict(kind=kind, precision="mixed", radius=5e-3, height=20e-3, notch=1e-3,
                    spacing=_log(rng, 0.16e-3, 0.6e-3), steps=rng.randint(4, 10))
    if kind == "request":
        return dict(kind=kind, precision="mixed", n=int(_log(rng, 2000, 200000)), steps=rng.randint(20, 60))
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(2, 24), n_min=2000, n_max=int(_log(rng, 5000, 100000)),
                    steps=rng.randint(10, 20))
    if kind == "neighbors":
        return dict(kind=kind, **_box(rng, 1000, 240000))
    return dict(kind=kind, damage=rng.choice(("cl", "jc", "gtn")), n=int(_log(rng, 1000, 400000)))


# ---------------------------------------------------------------- inputs
def _vibration(sp, seed, amplitude):
    """A smooth velocity field: three standing waves with phases from the seed."""
    u = S.uniform(seed, 12, stream=21).reshape(3, 4)
    X = sp.X - sp.X.min(axis=0)
    ext = np.maximum(X.max(axis=0), sp.spacing)
    V = np.zeros_like(X)
    for k in range(3):
        arg = 2.0 * math.pi * (u[k, 3] + X[:, 2] / ext[2] * (1 + k))
        for c in range(3):
            V[:, c] += amplitude * (u[k, c] + math.copysign(0.5, u[k, c] - 0.5)) * np.sin(arg + c * X[:, c] / ext[c])
    return V


def _workload(case, seed):
    """The specimen, materials and step parameters of a case, from the seed alone."""
    kind = case["kind"]
    if kind in ("bar", "flow"):
        make = S.tensile_bar_cl if case["damage"] == "cl" else S.tensile_bar_jc
        w = make(case["nx"], case["ny"], case["nz"], seed=seed, v_grip=0.05 if kind == "bar" else 5.0)
        if kind == "bar":       # slow grips on a bar that vibrates: elastic however long the run goes on
            sp = w.specimen
            free = sp.bc_mask == 0
            sp.bc_vel[free] = _vibration(sp, seed, 0.6)[free]
    elif kind == "notched":
        w = S.notched_bar_gtn(case["radius"], case["height"], case["spacing"], case["notch"], seed=seed, v_grip=5.0)
    else:
        w = S.taylor_impact(case["n"], v_impact=150.0 + 150.0 * float(S.uniform(seed, 1, stream=22)[0]))
        w.specimen.X[:, 2] -= 0.499 * w.specimen.spacing    # the foot at the wall: contact from the first step on
    return w


def _flow_state(w, seed):
    """Plastic flow (S.plastic_flow_state) with a strain drawn from the seed and a Cauchy stress and a plastic
    strain that go with it; the yield stress of that plastic strain."""
    strain = 0.008 + 0.006 * float(S.uniform(seed, 1, stream=23)[0])
    st = S.plastic_flow_state(w, strain)
    m = w.materials[0]
    ep = 0.5 * strain * (1.0 + 0.2 * S.uniform(seed, w.specimen.N, stream=24))
    flow = (m["A"] + m["B"] * ep ** m["n"]) / m["A"]
    st["STRESS_DEV"] = st["STRESS_DEV"] * flow[:, None]
    st["SIGMA"] = st["STRESS_DEV"].copy()
    st["EPSP"] = ep
    return st


def _points(case, seed):
    n = case["n"]
    m = {"cl": S.aluminium_cl(), "jc": S.aluminium_jc(), "gtn": S.aluminium_gtn()}[case["damage"]]
    g = torch.Generator().manual_seed(seed)
    d = torch.randn(n, 3, 3, dtype=torch.float64, generator=g)
    deps = 2e-3 * torch.rand(n, 1, 1, dtype=torch.float64, generator=g) * 0.5 * (d + d.transpose(1, 2))
    J = 1.0 + 1.5e-3 * torch.randn(n, dtype=torch.float64, generator=g)
    s = torch.randn(n, 3, 3, dtype=torch.float64, generator=g)
    s = 0.5 * (s + s.transpose(1, 2))
    s = s - torch.diag_embed(s.diagonal(dim1=1, dim2=2).mean(1, keepdim=True).expand(n, 3))
    seq = (1.5 * (s * s).sum((1, 2))).sqrt()
    state = torch.zeros(n, 16, dtype=torch.float64)
    state[:, :9] = (s * (0.95 * m["A"] / seq)[:, None, None]).reshape(n, 9)
    state[:, 10] = 0.05 * torch.rand(n, dtype=torch.float64, generator=g)
    state[:, 12] = 0.3 * torch.rand(n, dtype=torch.float64, generator=g)
    if case["damage"] == "gtn":
        state[:, 14] = 0.001 + 0.02 * torch.rand(n, dtype=torch.float64, generator=g)
        state[:, 13] = m["q1"] * state[:, 14]
    return m, deps.reshape(n, 9).cuda(), J.cuda(), state.cuda()


def _batch(case, seed):
    """Bars as in the batched workload: particle counts spread over the logarithm of the range, damage constants
    within 20 % of the Johnson-Cook bar's; slow grips on bars that vibrate."""
    out = []
    u = S.uniform(seed, 4 * case["count"], stream=25).reshape(-1, 4)
    for k in range(case["count"]):
        n = case["n_min"] * (case["n_max"] / case["n_min"]) ** ((k + 0.5) / case["count"])
        nx = max(3, round((n / 4.0) ** (1.0 / 3.0)))
        w = S.tensile_bar_jc(nx, nx, 4 * nx, seed=seed * 1009 + k, v_grip=0.05)
        for key, f in zip(("D1", "D2", "D3", "C"), u[k]):
            w.materials[0][key] *= 0.8 + 0.4 * float(f)
        free = w.specimen.bc_mask == 0
        w.specimen.bc_vel[free] = _vibration(w.specimen, seed + k, 0.6)[free]
        out.append(w)
    return out


def prepare(case, seed):
    kind = case["kind"]
    if kind == "neighbors":
        sp = S.tensile_bar(case["nx"], case["ny"], case["nz"], 0.5e-3, 0.01, seed)
        X = torch.from_numpy(sp.X).cuda()
        return dict(case, X=X, rc=1.5e-3, row_ptr=torch.empty(sp.N + 1, dtype=torch.int64, device="cuda"),
                    col=torch.full((124 * sp.N,), -1, dtype=torch.int32, device="cuda"))
    if kind == "points":
        m, deps, J, state = _points(case, seed)
        return dict(case, mat=m, deps=deps, J=J, state=state)
    if kind == "batch":
        ws = _batch(case, seed)
        sims = [tlsph.Simulation.from_workload(w, precision="mixed", line_order=True) for w in ws]
        b = tlsph.Batch(len(sims))
        b.set(sims)
        return dict(case, sims=sims, batch=b)
    if kind == "request":
        return dict(case, w=_workload(case, seed))
    w = _workload(case, seed)
    sim = tlsph.Simulation.from_workload(w, precision=case["precision"])
    if case.get("tuned"):
        sim.set_plan((5, 128, 8, 128))
    state = dict(case, sim=sim)
    if kind in ("flow", "notched"):
        for k, v in _flow_state(w, seed).items():
            sim.set(k, v)
    if kind != "bar":
        state["start"] = sim.checkpoint()
    return state


# ---------------------------------------------------------------- one pass
def _read(sim, names):
    if sim.precision == "mixed":
        return {k: sim.get_device(k).float() for k in names}
    return {k: sim.get_device(k) for k in names}


def run(state):
    kind = state["kind"]
    if kind == "bar":
        sim, seen = state["sim"], []
        for _ in range(state["watch"]):
            sim.step(state["steps"])
            d = sim.diagnostics()
            seen.append([d[k] for k in DIAGS])
        if not seen:
            sim.step(state["steps"])
        out = _read(sim, FIELDS)
        if seen:
            t = torch.tensor(seen, dtype=torch.float64)
            out["diagnostics"] = t.float() if sim.precision == "mixed" else t
        return out
    if kind in ("flow", "notched", "taylor"):
        sim = state["sim"]
        sim.restore(state["start"])
        sim.step(state["steps"])
        out = _read(sim, FIELDS)
        if kind == "notched":
            out.update(_read(sim, ("POROSITY",)))
        return out
    if kind == "request":
        w = state["w"]
        with tlsph.Simulation.from_workload(w, precision=state["precision"]) as sim:
            sim.step(state["steps"])
            sim.sync()
            return {k: sim.get(k).astype(np.float32) for k in ("U", "V", "SIGMA", "EPSP", "DAMAGE")}
    if kind == "batch":
        state["batch"].step(state["steps"], graph=True)
        return [_read(s, ("U", "V", "SIGMA")) for s in state["sims"]]
    if kind == "neighbors":
        nnz = tlsph.neighbors_noalloc(state["X"], state["rc"], state["row_ptr"], state["col"])
        return [nnz, state["row_ptr"], state["col"]]
    st = state["state"].clone()
    tlsph.material_point_batch(state["mat"], 1e-7, state["deps"], state["J"], st)
    return st


# ---------------------------------------------------------------- what a pass cannot do without
def _box_pairs(nx, ny, nz):
    """Directed neighbour pairs of a jittered box lattice at a cutoff of three spacings (a pair at exactly
    three spacings is in about every second time)."""
    total = 0.0
    for a in range(-3, 4):
        for b in range(-3, 4):
            for c in range(-3, 4):
                r2 = a * a + b * b + c * c
                if 0 < r2 <= 9:
                    full = max(0, nx - abs(a)) * max(0, ny - abs(b)) * max(0, nz - abs(c))
                    total += full if r2 < 9 else 0.5 * full
    return total


def _particles(case):
    """(particles, directed pairs) of a case, from its dimensions."""
    kind = case["kind"]
    if kind in ("bar", "flow", "neighbors"):
        nx, ny, nz = case["nx"], case["ny"], case["nz"]
        return nx * ny * nz, _box_pairs(nx, ny, nz)
    if kind == "notched":
        n = math.pi * case["radius"] ** 2 * case["height"] / case["spacing"] ** 3
        return n, 100.0 * n
    if kind == "batch":     # the mean of a log-uniform particle count
        lo, hi = case["n_min"], case["n_max"]
        n = case["count"] * (hi - lo) / math.log(hi / lo)
        return n, 95.0 * n
    return case["n"], 95.0 * case["n"]


def work(case):
    kind = case["kind"]
    n, pairs = _particles(case)
    if kind == "neighbors":
        return dict(bytes=24.0 * n + 8.0 * (n + 1) + 4.0 * pairs, flops=8.0 * pairs)
    if kind == "points":
        return dict(bytes=n * 8.0 * (9 + 1 + 16 + 16), flops=n * (1500.0 if case["damage"] == "gtn" else 250.0))
    # the state of a particle read and written once per step: u, v, F, stress deviator, stress, plastic strain,
    # its rate, initiation, damage, porosity, energy (FP64; FP32 pairs and singles in the mixed path) and
    # what is read only: L^-1, mass, material; a pair: 15 + 46 multiply-adds, its index from the lattice order
    word = 8.0 if case.get("precision") == "fp64" else 5.0
    steps = case["steps"] * max(1, case.get("watch", 0))
    return dict(bytes=steps * n * word * (2 * (6 + 9 + 6 + 6 + 6) + 12), flops=steps * pairs * 2.0 * 61.0)


# ---------------------------------------------------------------- the same in plain torch, FP64
def _dev():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _moduli(m):
    return m["E"] / (3.0 * (1.0 - 2.0 * m["nu"])), m["E"] / (2.0 * (1.0 + m["nu"]))


def _hard(m, ep):
    return m["A"] + m["B"] * torch.where(ep > 0, ep.clamp(min=1e-300) ** m["n"], torch.zeros_like(ep))


def _rate(m, epdot):
    if m["C"] == 0.0:
        return torch.ones_like(epdot)
    return 1.0 + m["C"] * torch.log((epdot / m["epsdot0"]).clamp(min=1.0))


def _vm(s):
    return (1.5 * (s * s).sum((1, 2))).sqrt()


def _fstar(m, f):
    mid = m["fc"] + (1.0 / m["q1"] - m["fc"]) / (m["fF"] - m["fc"]) * (f - m["fc"])
    return torch.where(f <= m["fc"], f, torch.where(f >= m["fF"], torch.full_like(f, 1.0 / m["q1"]), mid))


def _material(m, dt, de, J, p):
    """Constitutive and damage update of the points of `p` (sd, sm, ep, epdot, dinit, D, f), in place; all of
    them intact, linear equation of state.  Returns the mask of the points that fail."""
    K, G = _moduli(m)
    eye = torch.eye(3, dtype=de.dtype, device=de.device)
    ed = de - eye * (de.diagonal(dim1=1, dim2=2).sum(1) / 3.0)[:, None, None]
    omd = 1.0 - p["D"]
    tr = p["sd"] + 2.0 * G * omd[:, None, None] * ed
    seq = _vm(tr)
    sm = K * (J - 1.0)
    sm = torch.where(sm > 0, sm * omd, sm)
    if m["damage"] != S.DAMAGE_GTN:
        sf = _hard(m, p["ep"]) * _rate(m, p["epdot"]) * omd
        plastic = seq > sf
        dep = torch.where(plastic, (seq - sf) / (3.0 * G * omd), torch.zeros_like(seq))
        p["sd"] = torch.where(plastic[:, None, None], (sf / seq.clamp(min=1e-300))[:, None, None] * tr, tr)
        p["ep"] = p["ep"] + dep
        p["epdot"] = dep / dt
        p["sm"] = sm
        if m["damage"] == S.DAMAGE_CL:
            s1 = torch.linalg.eigvalsh(p["sd"] + p["sm"][:, None, None] * eye)[:, 2]
            p["dinit"] = p["dinit"] + s1.clamp(min=0) * dep / m["Wcr"]
        else:
            sq = _vm(p["sd"])
            tri = torch.where(sq < 1e-12 * K, torch.zeros_like(sq), p["sm"] / sq.clamp(min=1e-300))
            ef = (m["D1"] + m["D2"] * torch.exp(m["D3"] * tri)) * (1.0 + dep / dt / m["epsdot0"]) ** m["D4"]
            p["dinit"] = p["dinit"] + dep / ef.clamp(min=1e-12)
        p["D"] = torch.where(p["dinit"] >= 1.0, (10.0 * (p["dinit"] - 1.0)).clamp(max=1.0), torch.zeros_like(seq))
        return p["D"] >= 1.0
    f, ep0, q1, q2 = p["f"], p["ep"], m["q1"], m["q2"]
    fs, rate = _fstar(m, f), _rate(m, p["epdot"])
    tri = sm / seq.clamp(min=1e-300)
    sM = _hard(m, ep0) * rate
    a1, c0 = 1.5 * q2 * tri, 1.0 + m["q3"] * fs * fs
    xt = seq / sM
    plastic = (xt * xt + 2.0 * q1 * fs * torch.cosh(a1 * xt) - c0 > 0) & (seq >= 1e-12 * K)
    x = xt.clamp(max=1.0)
    for _ in range(60):
        phi = x * x + 2.0 * q1 * fs * torch.cosh(a1 * x) - c0
        x = torch.where(plastic, x - phi / (2.0 * x + 2.0 * q1 * fs * a1 * torch.sinh(a1 * x)), x)
    sh = torch.sinh(a1 * x)
    kf = (x + 1.5 * q1 * q2 * f * tri * sh) / (3.0 * G * omd * (1.0 - f))
    hi = ((seq - x * sM) * kf).clamp(min=0)
    lo, d = torch.zeros_like(hi), hi.clone()
    for _ in range(100):        # Newton inside a bracket
        e = (ep0 + d).clamp(min=1e-300)
        g = d - (seq - x * _hard(m, ep0 + d) * rate) * kf
        hi, lo = torch.where(g > 0, d, hi), torch.where(g > 0, lo, d)
        dn = d - g / (1.0 + x * m["B"] * m["n"] * e ** (m["n"] - 1.0) * rate * kf)
        d = torch.where((dn >= lo) & (dn <= hi), dn, 0.5 * (lo + hi))
    ep = ep0 + d
    sMn = _hard(m, ep) * rate
    sy = x * sMn
    depeq = (seq - sy) / (3.0 * G * omd)
    alpha = 1.5 * (sMn / sy) * q1 * q2 * f * sh
    om = (1.0 - (27.0 * torch.linalg.det(tr) / (2.0 * seq ** 3)) ** 2).clamp(0, 1)
    z = (ep - m["eN"]) / m["sN"]
    nucl = m["fN"] / (m["sN"] * math.sqrt(2.0 * math.pi)) * torch.exp(-0.5 * z * z) * d
    grow = (1.0 - f) / (alpha * tri + 1.0) * (sMn / sy) * (alpha * (1.0 - f) + f * m["komega"] * om) * d
    p["sd"] = torch.where(plastic[:, None, None], (sy / seq)[:, None, None] * tr, tr)
    p["sm"] = torch.where(plastic, sm - 3.0 * G * omd * tri * depeq, sm)
    p["ep"] = torch.where(plastic, ep, ep0)
    p["epdot"] = torch.where(plastic, d / dt, torch.zeros_like(d))
    p["f"] = torch.where(plastic, (f + nucl + grow).clamp(0, m["fF"]), f)
    p["D"] = torch.where(p["f"] >= m["fF"], torch.ones_like(f), q1 * _fstar(m, p["f"]))
    return p["D"] >= 1.0


class _Exact:
    """The time step on a (jittered) cubic lattice: neighbours j of row i as a dense table over the lattice
    offsets within reach, rows in chunks."""

    CHUNK = 131072

    def __init__(self, w):
        dev, sp = _dev(), w.specimen
        self.w, self.m, self.h, self.dt = w, w.materials[0], w.h, w.dt
        t = lambda a: torch.as_tensor(a, device=dev)  # noqa: E731
        self.X, self.vol = t(sp.X), t(sp.vol)
        self.bc, self.bcv = t(sp.bc_mask).bool(), t(sp.bc_vel)
        N = sp.N
        idx = torch.round((self.X - self.X.min(0).values) / sp.spacing).long() + 4
        n = idx.max(0).values + 5
        grid = torch.full((int(n[0]) * int(n[1]) * int(n[2]),), -1, dtype=torch.int32, device=dev)
        flat = (idx[:, 0] * n[1] + idx[:, 1]) * n[2] + idx[:, 2]
        grid[flat] = torch.arange(N, dtype=torch.int32, device=dev)
        off = [(a, b, c) for a in range(-3, 4) for b in range(-3, 4) for c in range(-3, 4)
               if 0 < a * a + b * b + c * c <= 9]
        shift = torch.tensor([(a * int(n[1]) + b) * int(n[2]) + c for a, b, c in off], device=dev)
        self.rows = []
        for r0 in range(0, N, self.CHUNK):
            i = slice(r0, min(N, r0 + self.CHUNK))
            j = grid[flat[i, None] + shift]
            d = self.X[j.clamp(min=0).long()] - self.X[i, None]
            r2 = (d * d).sum(2)
            near = (j >= 0) & (r2 < w.rc * w.rc)
            d = torch.where(near[..., None], d, torch.full_like(d, w.rc))    # no neighbour: weight 0, finite terms
            r2 = torch.where(near, r2, (d * d).sum(2))
            r = r2.sqrt()
            q = r / self.h
            a, b = (2.0 - q).clamp(min=0), (1.0 - q).clamp(min=0)
            norm = 1.0 / (math.pi * self.h ** 3)
            V = self.vol[j.clamp(min=0).long()]
            g = torch.where(near, V * (3.0 * b * b - 0.75 * a * a) * (norm / self.h) / r, torch.zeros_like(r))
            k = torch.where(near, V * (0.25 * a ** 3 - b ** 3) * norm * self.m["E"] / r2, torch.zeros_like(r))
            L = torch.einsum("nk,nka,nkb->nab", g, d, d)
            self.rows.append((i, j.clamp(min=0).long(), d, g, k, torch.linalg.inv(L)))
        z = lambda *s: torch.zeros(N, *s, dtype=torch.float64, device=dev)  # noqa: E731
        self.U, self.V, self.force = z(3), self.bcv.clone(), z(3)
        self.F = torch.eye(3, dtype=torch.float64, device=dev).repeat(N, 1, 1)
        self.p = dict(sd=z(3, 3), sm=z(), ep=z(), epdot=z(), dinit=z(), D=z(), f=t(sp.f0).clone())
        if self.m["damage"] == S.DAMAGE_GTN:
            self.p["D"] = self.m["q1"] * _fstar(self.m, self.p["f"])
        self.sig, self.e = z(3, 3), z()
        self.failed = torch.zeros(N, dtype=torch.bool, device=dev)
        self.mass = self.m["rho0"] * self.vol

    def load(self, st):
        t = lambda a: torch.as_tensor(a, device=self.X.device)  # noqa: E731
        self.U, self.V, self.F = t(st["U"]), t(st["V"]), t(st["F"]).reshape(-1, 3, 3)
        self.p["sd"], self.sig = t(st["STRESS_DEV"]).reshape(-1, 3, 3), t(st["SIGMA"]).reshape(-1, 3, 3)
        self.p["ep"] = t(st["EPSP"])

    def _bc(self, v):
        v = torch.where(self.bc[:, None], self.bcv, v)
        return torch.where(self.failed[:, None], torch.zeros_like(v), v)

    def _wall(self, u, v):
        if self.w.wall:
            below = self.X[:, 2] + u[:, 2] < 0
            u[:, 2] = torch.where(below, -self.X[:, 2], u[:, 2])
            v[:, 2] = torch.where(below, v[:, 2].clamp(min=0), v[:, 2])

    def run(self, steps):
        dt, p = self.dt, self.p
        vh = self._bc(self.V + 0.5 * dt * self.force / self.mass[:, None])
        u1 = self.U + dt * vh
        self._wall(u1, vh)
        A = torch.zeros_like(self.F)
        for _ in range(steps):
            omd = 1.0 - p["D"]
            Fd = torch.empty_like(self.F)
            for i, j, d, g, k, Li in self.rows:
                M = torch.einsum("nka,nkb->nab", (g * omd[j])[..., None] * (vh[j] - vh[i, None]), d)
                Fd[i] = M @ Li
            go = ~self.failed
            self.F = torch.where(go[:, None, None], self.F + dt * Fd, self.F)
            J = torch.linalg.det(self.F)
            Fi = torch.linalg.inv(self.F)
            Lv = Fd @ Fi
            d_ = 0.5 * (Lv + Lv.transpose(1, 2))
            R = self.F.clone()
            for _ in range(12):         # polar rotation: Newton's iteration
                R = 0.5 * (R + torch.linalg.inv(R).transpose(1, 2))
            Rt = R.transpose(1, 2)
            new = dict(p)
            fails = _material(self.m, dt, dt * (Rt @ d_ @ R), J, new) & go
            for key, v in new.items():
                keep = go.reshape(-1, *([1] * (v.dim() - 1)))
                p[key] = torch.where(keep, v, p[key])
            dead = fails | self.failed
            eye = torch.eye(3, dtype=torch.float64, device=R.device)
            sg = R @ (p["sd"] + p["sm"][:, None, None] * eye) @ Rt
            sg = torch.where(dead[:, None, None], torch.zeros_like(sg), sg)
            p["sd"] = torch.where(dead[:, None, None], torch.zeros_like(sg), p["sd"])
            power = ((self.sig + sg) * d_).sum((1, 2))
            self.e = self.e + torch.where(go, 0.5 * dt * J / self.m["rho0"] * power, torch.zeros_like(J))
            self.sig, self.failed = sg, dead
            P = J[:, None, None] * sg @ Fi.transpose(1, 2)
            for i, j, d, g, k, Li in self.rows:
                A[i] = P[i] @ Li.transpose(1, 2)
            omd = 1.0 - p["D"]
            G = self.F - eye
            for i, j, d, g, k, Li in self.rows:
                s1 = ((g * omd[j])[..., None] * d).sum(1)
                s2 = torch.einsum("nkab,nkb->na", A[j], g[..., None] * d)
                f = (A[i] @ s1[..., None])[..., 0] + omd[i, None] * s2
                u = u1[j] - u1[i, None]
                x = d + u
                err = torch.einsum("nkab,nkb->nka", G[j] + G[i, None], d) - 2.0 * u
                c = k * omd[j] * (err * x).sum(2) / (x * x).sum(2)
                f = f - 0.5 * self.w.hg_alpha * omd[i, None] * (c[..., None] * x).sum(1)
                self.force[i] = self.vol[i, None] * f
            a = self.force / self.mass[:, None]
            self.U = u1
            self.V = self._bc(vh + 0.5 * dt * a)
            vh = self._bc(self.V + 0.5 * dt * a)
            u1 = u1 + dt * vh
            self._wall(u1, vh)

    def fields(self, names):
        n = self.X.shape[0]
        all_ = dict(U=self.U, V=self.V, F=self.F.reshape(n, 9), SIGMA=self.sig.reshape(n, 9), FORCE=self.force,
                    EPSP=self.p["ep"], DAMAGE=self.p["D"], POROSITY=self.p["f"])
        return {k: all_[k].clone() for k in names}

    def diagnostics(self):
        ke = (0.5 * self.mass * (self.V * self.V).sum(1)).sum()
        return [float(ke), float((self.mass * self.e).sum()), float(self.p["ep"].max()), float(self.p["D"].max())]


def exact(case, seed):
    kind = case["kind"]
    if kind == "neighbors":
        return None
    if kind == "points":
        m, deps, J, st = _points(case, seed)
        n = case["n"]
        de = deps.reshape(n, 3, 3)
        p = dict(sd=st[:, :9].reshape(n, 3, 3), sm=st[:, 9], ep=st[:, 10], epdot=st[:, 11], dinit=st[:, 12],
                 D=st[:, 13], f=st[:, 14])
        dead = _material(m, 1e-7, 0.5 * (de + de.transpose(1, 2)), J, p)
        p["sd"] = torch.where(dead[:, None, None], torch.zeros_like(de), p["sd"])
        p["sm"] = torch.where(dead, torch.zeros_like(J), p["sm"])
        one = [p[k][:, None] for k in ("sm", "ep", "epdot", "dinit", "D", "f")]
        return torch.cat([p["sd"].reshape(n, 9), *one, dead.double()[:, None]], 1)
    if kind == "batch":
        out = []
        for w in _batch(case, seed):
            x = _Exact(w)
            x.run(case["steps"])
            out.append(x.fields(("U", "V", "SIGMA")))
        return out
    w = _workload(case, seed)
    x = _Exact(w)
    if kind == "request":
        x.run(case["steps"])
        return x.fields(("U", "V", "SIGMA", "EPSP", "DAMAGE"))
    if kind in ("flow", "notched"):
        x.load(_flow_state(w, seed))
    seen = []
    for _ in range(case.get("watch", 0)):
        x.run(case["steps"])
        seen.append(x.diagnostics())
    if not seen:
        x.run(case["steps"])
    out = x.fields(FIELDS)
    if kind == "notched":
        out.update(x.fields(("POROSITY",)))
    if seen:
        out["diagnostics"] = torch.tensor(seen, dtype=torch.float64)
    return out
