"""Timed cases of the library's main paths, each one pass through its public entry points.

A case is a dict of plain values.  `form` says which calls it makes:

  lattice   one lattice: init from pulses, a run of time steps with probes recorded (harmonic
            sources where asked for), the series, the spectrum of their sum and a snapshot of P
  ensemble  uneven trumpets advanced together: init, steps, series and every member's lowest modes
  sweep     the resonance sweep: one lattice per source frequency, steady-state response
  spectrum  mode frequencies of host series
  fit       Adam training of the surrogate network
  grad      loss and gradient of the surrogate network on one batch
  predict   surrogate inference

Snapshots and series are kept at the storage width of the lattice they come from, as a program
that writes them out keeps them, and mode frequencies in the single precision the surrogate's
targets have.  `exact` computes the same outputs in 64 bits with plain torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import lbw_workloads as W
from paper_1705_01801_gb300 import lbw, sweep

PREC = {"f64": W.PREC_F64, "f32": W.PREC_F32, "f16": W.PREC_F16S, "bf16": W.PREC_BF16S}
KEEP = {"f64": torch.float64, "f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
ELEM = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2}
RANGES = {"wide": ((32, 96), (32, 96), (128, 512)),    # the benchmark's ensemble
          "small": ((12, 24), (32, 48), (40, 80))}     # the surrogate's training ensembles
IN_DIM = 7                                             # geometry features of a trumpet


def listed():
    return [
        # The 2-D reference run: small, FP64, Dirichlet rim; thousands of steps of a lattice that
        # fits in cache, so what counts is the time between two steps.
        _lattice("disk_f64", "disk", 128, 128, 1, "f64", 1000, 1, 4),
        # The 3-D cylinder with closed ends, eight random-phase pulses and sixteen probes.
        _lattice("cylinder_f32", "cylinder", 128, 128, 256, "f32", 1000, 8, 16),
        # The flared horn in 16-bit storage: the reduced-precision production run.
        _lattice("trumpet_f16", "trumpet", 256, 256, 512, "f16", 500, 1, 32),
        # The largest lattice, 50 million nodes, in both storage widths it is run in.
        _lattice("torus_f32", "torus", 192, 1024, 256, "f32", 300, 1, 64),
        _lattice("torus_bf16", "torus", 192, 1024, 256, "bf16", 300, 1, 64),
        # A cylinder whose angular extent is no multiple of the tile width, as a user picks it.
        _lattice("cylinder_odd_f32", "cylinder", 100, 100, 250, "f32", 300, 1, 16),
        # The paper's torus (20 x 200 x 30 cells) driven by its ring source, in FP64.
        _lattice("torus_paper_f64", "paper_torus", 20, 200, 30, "f64", 1000, 0, 4, source=True),
        # The paper's open-closed pipe swept over 41 source frequencies.
        dict(name="pipe_sweep_f32", form="sweep", n1=20, n2=5, n3=100, prec="f32", freqs=41, steps=1000),
        # Uneven trumpets advanced together with every member's lowest modes: the surrogate's data.
        dict(name="ensemble_f32", form="ensemble", range="wide", members=48, prec="f32", steps=512, modes=8,
             sizes=5),
        # The sixteen probe series of the cylinder's full run.
        dict(name="spectrum_16x20000", form="spectrum", series=16, T=20000, modes=8),
        # Surrogate training on the ensemble's 408 training members, and a batch of queries.
        dict(name="fit_b64", form="fit", samples=408, batch=64, hidden=256, depth=4, out=8, steps=400),
        dict(name="predict_bf16_400", form="predict", samples=400, hidden=256, depth=4, out=8, bf16=True),
    ]


def _lattice(name, kind, n1, n2, n3, prec, steps, pulses, probes, source=False):
    return dict(name=name, form="lattice", kind=kind, n1=n1, n2=n2, n3=n3, prec=prec, steps=steps,
                pulses=pulses, probes=probes, source=source)


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    form = rng.choice(["lattice"] * 6 + ["ensemble"] * 2 + ["sweep", "spectrum", "fit", "grad", "predict"])
    if form == "lattice":
        kind = rng.choice(["disk", "cylinder", "trumpet", "torus"])
        nodes = _log(rng, 5e3, 2e5 if kind == "disk" else 2e7)
        n2 = 64 * _log(rng, 1, 8) if rng.random() < 0.5 else rng.randint(24, 300)
        if kind == "disk":
            n3 = 1
            n1 = max(12, min(1024, nodes // n2))
        else:
            n1 = max(10, min(256, int((nodes / n2) ** 0.5 * rng.uniform(0.5, 1.0))))
            if kind == "torus":  # arcs along the major circle stay longer than c
                n2 = min(n2, 30 * n1)
            # a flare over fewer cells than the radius is wide would be too steep for c
            n3 = max(n1 + n2 // 12 if kind == "trumpet" else 8, min(1024, nodes // (n1 * n2)))
        case = _lattice("", kind, n1, n2, n3, rng.choice(["f64", "f32", "f32", "f16", "bf16"]), 0,
                        rng.choice([1, 1, 8]), rng.choice([4, 16, 64]), source=rng.random() < 0.2)
        case["steps"] = min(_log(rng, 50, 2000), max(50, int(4e9 // (n1 * n2 * n3))))
    elif form == "ensemble":
        span = rng.choice(["wide", "small"])
        case = dict(form=form, range=span, members=_log(rng, 4, 40 if span == "wide" else 384),
                    prec=rng.choice(["f32", "f32", "f64", "f16", "bf16"]), steps=_log(rng, 64, 512), modes=8,
                    sizes=rng.randint(1, 10 ** 6))
        if case["prec"] == "f64":  # FP64 arithmetic is an order slower
            case["members"] = max(2, case["members"] // 8)
    elif form == "sweep":
        case = dict(form=form, n1=rng.randint(8, 32), n2=rng.randint(3, 48), n3=rng.randint(40, 160),
                    prec=rng.choice(["f64", "f32"]), freqs=rng.randint(9, 64), steps=_log(rng, 200, 1500))
    elif form == "spectrum":
        T = _log(rng, 256, 65536)
        case = dict(form=form, series=max(1, min(_log(rng, 1, 64), 1500000 // T)), T=T, modes=rng.choice([1, 8, 16]))
    else:
        case = dict(form=form, samples=rng.randint(200, 4000), hidden=rng.choice([64, 96, 128, 200, 256]), depth=4,
                    out=rng.choice([1, 2, 8]))
        if form == "fit":
            case.update(batch=rng.choice([16, 32, 50, 64, 128]), steps=_log(rng, 50, 600))
        if form == "predict":
            case.update(samples=_log(rng, 1, 20000), bf16=rng.random() < 0.6)
    case.pop("name", None)
    return case


# ------------------------------------------------------------------------- inputs ---------

def _spec(case):
    n, prec = (case["n1"], case["n2"], case["n3"]), PREC[case["prec"]]
    kind = case.get("kind", "pipe")
    if kind == "disk":
        return W.disk(n[0], n[1], prec=prec)
    if kind == "paper_torus":  # R = 640, r up to 409.6, D = 0.65 at the outer wall, rigid inner wall at 12
        return W.GridSpec(kind=W.KIND_TOROIDAL, n=n,
                          h=((409.6 - 12.0) / n[0], 2 * math.pi / n[1], 2 * math.pi / n[2]), x0=(12.0, 0, 0),
                          c=2.0, damping=0.65, geom=(640.0, 0, 0, 0), prec=prec,
                          bc=(W.BC_BOUNCE, W.BC_BOUNCE) + (W.BC_PERIODIC,) * 4)
    if kind == "pipe":  # closed at z = 0, free at the far end, r from 1 to 25 on 20 cells
        return W.GridSpec(kind=W.KIND_CYLINDRICAL, n=n, h=(1.2, 2 * math.pi / n[1], 1.0),
                          x0=(max(1.0, W.r_inner(0.1, n[1])), 0, 0), c=0.1, damping=0.98, prec=prec,
                          bc=(W.BC_BOUNCE, W.BC_BOUNCE, W.BC_PERIODIC, W.BC_PERIODIC, W.BC_BOUNCE, W.BC_FREE))
    return {"cylinder": W.cylinder, "trumpet": W.trumpet, "torus": W.torus}[kind](*n, prec=prec)


def _lattice_inputs(case, seed):
    spec = _spec(case)
    rng = np.random.default_rng(seed)
    pulses = W.pulses(spec, seed, case["pulses"], random_phase=case["pulses"] > 1)
    source = None
    if case["source"]:
        n1, n2, n3 = spec.n
        q1, q3 = int(rng.integers(0, n1)), int(rng.integers(0, n3))
        ring = np.array([[q1, j, q3] for j in range(n2)], np.int32)
        source = (ring, 0, 1.0, float(rng.uniform(0.02, 0.2)))
    return spec, pulses, W.probes(spec, seed, case["probes"]), source


def _ensemble_inputs(case, seed):
    r, th, z = RANGES[case["range"]]
    specs, _ = W.ensemble(case["members"], seed=case["sizes"], r_range=r, theta_range=th, z_range=z,
                          prec=PREC[case["prec"]])
    rng = np.random.default_rng(seed)
    pulses, probes = [], []
    for s in specs:
        p, q = W.ensemble_excitation(s, sigma=float(rng.uniform(2.0, 4.0)))
        pulses.append(p)
        probes.append(q)
    return specs, pulses, np.stack(probes)


def _sweep_inputs(case, seed):
    spec = _spec(case)
    n1, n2, n3 = spec.n
    ring = np.array([[0, j, 0] for j in range(n2)], np.int32)
    lo = np.random.default_rng(seed).uniform(0.0008, 0.002)
    return spec, ring, [n1 // 10, 0, n3 // 10], np.linspace(lo, 12 * lo, case["freqs"])


def _series(case, seed):
    """Decaying modes over a little noise, as probes of a pulse-excited resonator record them."""
    rng = np.random.default_rng(seed)
    T, n, modes = case["T"], case["series"], 24
    t = np.arange(T)
    om = np.sort(rng.uniform(0.02, 1.2, modes))
    a = rng.uniform(0.05, 1.0, (n, modes)) * np.exp(-om)
    ph = rng.uniform(0, 2 * np.pi, (n, modes))
    x = np.zeros((n, T))
    for m in range(modes):
        x += a[:, m:m + 1] * np.cos(om[m] * t + ph[:, m:m + 1]) * np.exp(-0.2 * t / T)
    return x + 1e-6 * rng.normal(size=(n, T))


def _net_inputs(case, seed):
    rng = np.random.default_rng(seed)
    x = rng.normal(size=(case["samples"], IN_DIM)).astype(np.float32)
    t = np.tanh(x @ rng.normal(size=(IN_DIM, case["out"])) * 0.5) + 0.05 * rng.normal(size=(len(x), case["out"]))
    order = None
    if case["form"] == "fit":
        b = min(case["batch"], len(x))
        order = np.concatenate([rng.permutation(len(x))[:b] for _ in range(case["steps"])]).astype(np.int32)
    return x, t.astype(np.float32), order


def _dims(case):
    return [IN_DIM] + [case["hidden"]] * (case["depth"] - 1) + [case["out"]]


def _params(case, seed):
    """Glorot-uniform weights and small biases, one vector: per layer W (out x in), then b."""
    rng = np.random.default_rng(seed + 17)
    p = []
    for a, b in zip(_dims(case)[:-1], _dims(case)[1:]):
        s = math.sqrt(6.0 / (a + b))
        p += [rng.uniform(-s, s, a * b), rng.uniform(-0.05, 0.05, b)]
    return np.concatenate(p).astype(np.float32)


def prepare(case, seed):
    form = case["form"]
    if form == "lattice":
        spec, pulses, probes, source = _lattice_inputs(case, seed)
        g = lbw.Grid(spec)
        g.set_probes(probes, case["steps"])
        if source is not None:
            g.set_sources(source[0], kind=source[1], amp=source[2], omega=source[3])
        return dict(case=case, grid=g, pulses=pulses)
    if form == "ensemble":
        specs, pulses, probes = _ensemble_inputs(case, seed)
        b = lbw.Batch(specs)
        b.set_probes(probes, case["steps"])
        return dict(case=case, batch=b, pulses=pulses)
    if form == "sweep":
        return dict(case=case, args=_sweep_inputs(case, seed))
    if form == "spectrum":
        return dict(case=case, x=_series(case, seed))
    x, t, order = _net_inputs(case, seed)
    net = lbw.MLP(IN_DIM, hidden=case["hidden"], depth=case["depth"], out_dim=case["out"], seed=seed)
    p = _params(case, seed)
    net.set_params(p)
    return dict(case=case, net=net, p=p, x=x, t=t, order=order)


# ------------------------------------------------------------------------- one pass -------

def _kept(a, prec):
    return torch.from_numpy(a).to(KEEP[prec])


def _table(peaks, k):
    """Peaks of several series as rows of k, zeros where fewer were found."""
    out = np.zeros((2, len(peaks), k), np.float32)
    for row, (f, a) in enumerate(peaks):
        out[0, row, :len(f)], out[1, row, :len(a)] = f, a
    return {"freq": out[0], "amp": out[1]}


def run(state):
    case = state["case"]
    form = case["form"]
    if form == "lattice":
        g, prec = state["grid"], case["prec"]
        g.init(state["pulses"])
        g.step(case["steps"])
        out = {"series": _kept(g.read_probes(), prec)}
        if prec in ("f64", "f32"):
            out.update(_table([g.spectrum(-1, 4)], 4))
        out["P"] = _kept(g.get_P(), prec)
        return out
    if form == "ensemble":
        b = state["batch"]
        b.init(state["pulses"])
        b.step(case["steps"])
        out = {"series": _kept(b.read_probes(), case["prec"])}
        freq, amp, count = b.spectrum(case["modes"], lowest=True)
        if case["prec"] in ("f64", "f32"):
            out.update(freq=freq.astype(np.float32), amp=amp.astype(np.float32), count=count)
        return out
    if form == "sweep":
        spec, ring, probe, omegas = state["args"]
        r = sweep.resonance_curve(spec, ring, probe, omegas, steps=case["steps"], tail=case["steps"] // 4)
        return _kept(r, case["prec"])
    if form == "spectrum":
        return _table(lbw.lbw_spectrum_series(state["x"], case["modes"]), case["modes"])
    net = state["net"]
    if form == "fit":
        net.set_params(state["p"])
        b = min(case["batch"], case["samples"])
        return {"loss": net.train(state["x"], state["t"], state["order"], b, 1e-3), "params": net.get_params()}
    if form == "grad":
        loss, g = net.grad(state["x"], state["t"])
        return {"loss": np.float32(loss), "grad": g}
    return net.predict_bf16(state["x"]) if case["bf16"] else net.forward(state["x"])


# ------------------------------------------------------------------------- work -----------

def work(case):
    form = case["form"]
    if form in ("lattice", "ensemble", "sweep"):
        if form == "ensemble":
            r, th, z = RANGES[case["range"]]
            specs, _ = W.ensemble(case["members"], seed=case["sizes"], r_range=r, theta_range=th, z_range=z)
            nodes, series = sum(s.nodes for s in specs), 8 * case["members"]
        else:
            nodes = case["n1"] * case["n2"] * case["n3"] * case.get("freqs", 1)
            series = case.get("probes", case.get("freqs"))
        # seven populations read and written per node and step, the initial populations written,
        # the series, and (lattice) the last populations read for the snapshot
        b = nodes * case["steps"] * 14 * ELEM[case["prec"]] + nodes * 7 * ELEM[case["prec"]]
        b += series * case["steps"] * 8
        if form == "lattice":
            b += nodes * (7 * ELEM[case["prec"]] + 8)
        return {"bytes": b, "flops": nodes * case["steps"] * 60}
    if form == "spectrum":
        M = 1 << math.ceil(math.log2(4 * case["T"]))
        # the series in; a real transform and 81 sums over the series for each refined peak
        return {"bytes": 8 * case["series"] * (case["T"] + 2 * case["modes"]),
                "flops": case["series"] * (2.5 * M * math.log2(M) + case["modes"] * 81 * case["T"] * 4)}
    d = _dims(case)
    weights = sum(a * b for a, b in zip(d[:-1], d[1:]))
    params = weights + sum(d[1:])
    if form == "fit":
        rows = min(case["batch"], case["samples"])
        # per step the weights, their gradient and both moments are read and written once
        return {"bytes": case["steps"] * (4 * rows * (IN_DIM + case["out"]) + 4 * 7 * params),
                "flops": case["steps"] * (6 * weights * rows + 12 * params)}
    io = 4 * case["samples"] * (IN_DIM + case["out"])
    if form == "grad":
        return {"bytes": io + 8 * params, "flops": 6 * weights * case["samples"]}
    return {"bytes": io + (2 if case["bf16"] else 4) * params, "flops": 2 * weights * case["samples"]}


# ------------------------------------------------------------------------- 64-bit values --

DEV = "cuda" if torch.cuda.is_available() else "cpu"


def _metric(spec, q1, q3):
    """sqrt g, g^11, g^22, g^33, g^13, G^1, G^3 in lattice coordinates at rows q1 x planes q3
    (arrays broadcast as [q3, q1]; ghost positions allowed)."""
    r = spec.x0[0] + (q1[None, :] + 0.5) * spec.h[0]
    w = spec.x0[2] + (q3[:, None] + 0.5) * spec.h[2]
    one = np.ones(np.broadcast(r, w).shape)
    r, w = r * one, w * one
    sg, g11, g22, g33, g13, G1, G3 = one, one, one, one, 0 * one, 0 * one, 0 * one
    if spec.kind in (W.KIND_POLAR, W.KIND_CYLINDRICAL):
        sg, g22, G1 = r, r ** -2, -1 / r
    elif spec.kind == W.KIND_TRUMPET:
        a0, b, al = spec.geom[:3]
        e = np.exp(al * w)
        s, ds = (a0 + b * e) / (a0 + b), b * al * e / (a0 + b)
        dds = al * ds
        sg, g11, g13, g22 = r * s * s, (1 + (r * ds) ** 2) / s ** 2, -r * ds / s, (r * s) ** -2
        G1 = (r * r * s * dds - 2 * (r * ds) ** 2 - 1) / (r * s * s)
    else:
        R = spec.geom[0]
        Rr = R + r * np.cos(w)
        sg, g22, g33 = r * Rr, Rr ** -2, r ** -2
        G1, G3 = -(R + 2 * r * np.cos(w)) / (r * Rr), np.sin(w) / (r * Rr)
    h = spec.h
    return [sg * h[0] * h[1] * h[2], g11 / h[0] ** 2, g22 / h[1] ** 2, g33 / h[2] ** 2, g13 / (h[0] * h[2]),
            G1 / h[0], G3 / h[2]]


class _Exact:
    """One lattice (or `copies` of it, one source frequency each) in 64 bits: the scheme written
    with whole-array torch operations on [population][copy, q3, q1, q2]; q2 is periodic."""

    def __init__(self, spec, copies=1):
        self.spec, (n1, n2, n3) = spec, spec.n
        self.shape = (copies, n3, n1, n2)
        at = lambda v: torch.from_numpy(np.ascontiguousarray(v)).to(DEV)[None, :, :, None]  # noqa: E731
        q1, q3 = np.arange(n1), np.arange(n3)
        m = _metric(spec, q1, q3)
        c2, cs2 = spec.c ** 2, spec.cs2
        self.sg, self.mG1, self.mG3 = at(m[0]), at(-c2 * m[5]), at(-c2 * m[6])
        self.h22 = at(0.5 * (c2 * m[2] - cs2))
        self.k = {}  # (dim of [copy, q3, q1, q2], side) -> half K^{1b}, half K^{3b} at that neighbour
        self.s1, self.s3 = torch.zeros_like(self.sg), torch.zeros_like(self.sg)
        for b, dim, n in ((0, 2, n1), (2, 1, n3)):
            for side in (-1, 1):
                face = spec.bc[2 * b + (side > 0)]
                p = (q1 if b == 0 else q3) + side
                if face == W.BC_PERIODIC:
                    p = p % n
                mn = _metric(spec, p, q3) if b == 0 else _metric(spec, q1, p)
                K11, K13, K33 = c2 * mn[1] - cs2, c2 * mn[4], c2 * mn[3] - cs2
                k1, k3 = (K11, K13) if b == 0 else (K13, K33)
                k1, k3 = 0.5 * side * k1, 0.5 * side * k3
                if face != W.BC_PERIODIC:  # the ghost's density is a multiple of the node's own
                    edge = [slice(None), slice(None)]
                    edge[1 if b == 0 else 0] = slice(-1, None) if side > 0 else slice(0, 1)
                    edge = tuple(edge)
                    own = 1.0 if face == W.BC_FREE else (1.0 if face == W.BC_BOUNCE else -1.0) * mn[0] / m[0]
                    e1, e3 = np.zeros_like(k1), np.zeros_like(k3)
                    e1[edge], e3[edge] = (k1 * own)[edge], (k3 * own)[edge]
                    self.s1, self.s3 = self.s1 + at(e1), self.s3 + at(e3)
                    k1[edge] = k3[edge] = 0.0
                self.k[dim, side] = at(k1), at(k3)
        self.w0, self.w1 = 1 - 3 * cs2, cs2 / 2
        self.src = None

    def _shifted_momentum_terms(self, rho):
        """Half the forcing term of each axis."""
        D1, D3 = self.s1 * rho, self.s3 * rho
        for (dim, side), (k1, k3) in self.k.items():
            r = torch.roll(rho, -side, dim)
            D1, D3 = torch.addcmul(D1, k1, r), torch.addcmul(D3, k3, r)
        D2 = self.h22 * (torch.roll(rho, -1, 3) - torch.roll(rho, 1, 3))
        return 0.5 * (self.mG1 * rho - D1), -0.5 * D2, 0.5 * (self.mG3 * rho - D3)

    def init(self, pulses):
        s = self.spec
        q = [torch.arange(n, dtype=torch.float64, device=DEV) + 0.5 for n in s.n]
        u1 = (s.x0[0] + q[0] * s.h[0])[None, None, :, None]
        u2 = (s.x0[1] + q[1] * s.h[1])[None, None, None, :]
        u3 = (s.x0[2] + q[2] * s.h[2])[None, :, None, None]
        if s.kind == W.KIND_TOROIDAL:
            R = s.geom[0] + u1 * torch.cos(u3)
            X = (R * torch.cos(u2), R * torch.sin(u2), u1 * torch.sin(u3))
        else:
            f = 1.0
            if s.kind == W.KIND_TRUMPET:
                f = (s.geom[0] + s.geom[1] * torch.exp(s.geom[2] * u3)) / (s.geom[0] + s.geom[1])
            X = (u1 * f * torch.cos(u2), u1 * f * torch.sin(u2), u3)
        P = torch.zeros(self.shape, dtype=torch.float64, device=DEV)
        for x, y, z, sigma, amp in pulses:
            P += amp * torch.exp(-((X[0] - x) ** 2 + (X[1] - y) ** 2 + (X[2] - z) ** 2) / (2 * sigma * sigma))
        rho = self.sg * P
        j = self._shifted_momentum_terms(rho)
        e = 0.5 * self.spec.cs2 * rho
        self.f = [self.w0 * rho] + [e + 0.5 * sgn * j[a] for a in range(3) for sgn in (1, -1)]
        self.t = 0

    def step(self):
        s, f = self.spec, self.f
        g = [f[0]]
        for a, dim in ((0, 2), (1, 3), (2, 1)):
            for sgn in (1, -1):
                i, o = 1 + 2 * a + (sgn < 0), 1 + 2 * a + (sgn > 0)
                v = torch.roll(f[i], sgn, dim)
                face = s.bc[2 * a + (sgn < 0)]
                if face != W.BC_PERIODIC:
                    at = 0 if sgn > 0 else s.n[a] - 1
                    own, opp = f[i].select(dim, at), f[o].select(dim, at)
                    v.select(dim, at).copy_(own if face == W.BC_FREE else
                                            (s.damping if face == W.BC_BOUNCE else -1.0) * opp)
                g.append(v)
        rho = g[0] + g[1] + g[2] + g[3] + g[4] + g[5] + g[6]
        self.rho = rho
        F = self._shifted_momentum_terms(rho)
        e = s.cs2 * rho
        out = [2 * self.w0 * rho - g[0]]
        for a in range(3):
            p, m = g[1 + 2 * a], g[2 + 2 * a]
            j = p - m + F[a]
            out += [e + j - p, e - j - m]
        self.f = out
        self.t += 1
        if self.src is not None:  # P = amp sin(omega t): the equilibrium that carries it
            (q1, q2, q3), amp, om = self.src
            v = self.sg[0, q3, q1, 0] * (amp * torch.sin(om * self.t))[:, None]
            for i in range(7):
                self.f[i][:, q3, q1, q2] = (self.w0 if i == 0 else self.w1) * v

    def sources(self, q, amp, omegas):
        q = torch.from_numpy(np.asarray(q, np.int64)).to(DEV)
        self.src = ((q[:, 0], q[:, 1], q[:, 2]), amp, torch.as_tensor(omegas, dtype=torch.float64, device=DEV))

    def record(self, probes, steps):
        """The probes' series [copy, probe, step] of `steps` time steps."""
        q = torch.from_numpy(np.asarray(probes, np.int64).reshape(-1, 3)).to(DEV)
        inv = 1.0 / self.sg[0, q[:, 2], q[:, 0], 0]
        out = torch.empty(self.shape[0], len(q), steps, dtype=torch.float64, device=DEV)
        for t in range(steps):
            self.step()
            out[:, :, t] = self.rho[:, q[:, 2], q[:, 0], q[:, 1]] * inv
        return out

    def P(self):
        return (self.f[0] + self.f[1] + self.f[2] + self.f[3] + self.f[4] + self.f[5] + self.f[6]) / self.sg


def _peaks(x, k, lowest=False, rel=1e-3):
    """The estimator the header describes: Hann window, zero padding, local maxima, a parabola
    through log-power and 40 golden-section steps on the windowed transform."""
    x = torch.as_tensor(x, dtype=torch.float64, device=DEV)
    T = x.numel()
    t = torch.arange(T, dtype=torch.float64, device=DEV)
    w = 0.5 - 0.5 * torch.cos(2 * math.pi * t / (T - 1))
    xw = w * (x - x.mean())
    M = 1
    while M < 4 * T:
        M *= 2
    pw = (torch.fft.rfft(xw, M).abs() ** 2).cpu().numpy()
    mid = pw[1:M // 2]
    ok = (mid > pw[:M // 2 - 1]) & (mid >= pw[2:M // 2 + 1]) & (mid >= rel * pw[1:].max())
    j = np.nonzero(ok)[0] + 1
    j = np.sort((j if lowest else j[np.argsort(-pw[j], kind="stable")])[:k])
    if len(j) == 0:
        return np.zeros(0), np.zeros(0)
    la, lb, lc = np.log(pw[j - 1]), np.log(pw[j]), np.log(pw[j + 1])
    om = 2 * math.pi * (j + 0.5 * (la - lc) / (la - 2 * lb + lc)) / M

    def power(o):
        ph = torch.as_tensor(o, device=DEV)[:, None] * t[None, :]
        return ((torch.cos(ph) @ xw) ** 2 + (torch.sin(ph) @ xw) ** 2).cpu().numpy()

    a, b = om - 2 * math.pi / M, om + 2 * math.pi / M
    gold = (math.sqrt(5) - 1) / 2
    for _ in range(40):
        c, d = b - gold * (b - a), a + gold * (b - a)
        up = power(c) > power(d)
        a, b = np.where(up, a, c), np.where(up, d, b)
    om = 0.5 * (a + b)
    return om, 2 * np.sqrt(power(om)) / float(w.sum())


def _peak_table(series, k, lowest=False):
    out = np.zeros((2, len(series), k))
    for row, x in enumerate(series):
        f, a = _peaks(x, k, lowest)
        out[0, row, :len(f)], out[1, row, :len(a)] = f, a
    return {"freq": out[0], "amp": out[1]}


def _layers(case, p):
    out, off = [], 0
    for a, b in zip(_dims(case)[:-1], _dims(case)[1:]):
        out.append((p[off:off + a * b].reshape(b, a), p[off + a * b:off + a * b + b]))
        off += a * b + b
    return out


def _forward(layers, x):
    for n, (A, b) in enumerate(layers):
        x = x @ A.T + b
        if n + 1 < len(layers):
            x = torch.tanh(x)
    return x


def _loss_grad(case, p, x, t):
    p = p.detach().requires_grad_(True)
    loss = ((_forward(_layers(case, p), x) - t) ** 2).mean()
    loss.backward()
    return loss.detach(), p.grad


def exact(case, seed):
    form = case["form"]
    if form == "lattice":
        if case["n1"] * case["n2"] * case["n3"] * case["steps"] > 2e10:
            return None  # over 20 seconds in 64 bits
        spec, pulses, probes, source = _lattice_inputs(case, seed)
        e = _Exact(spec)
        e.init(pulses)
        if source is not None:
            e.sources(source[0], source[2], [source[3]])
        series = e.record(probes, case["steps"])[0]
        out = {"series": series, "P": e.P()[0]}
        if case["prec"] in ("f64", "f32"):
            out.update(_peak_table([series.sum(0)], 4))
        return out
    if form == "ensemble":
        specs, pulses, probes = _ensemble_inputs(case, seed)
        if case["members"] * case["steps"] > 26000:
            return None
        series = []
        for s, p, q in zip(specs, pulses, probes):
            e = _Exact(s)
            e.init(p)
            series.append(e.record(q, case["steps"])[0])
        out = {"series": torch.stack(series)}
        if case["prec"] in ("f64", "f32"):
            out.update(_peak_table([v.sum(0) for v in series], case["modes"], lowest=True), count=None)
        return out
    if form == "sweep":
        spec, ring, probe, omegas = _sweep_inputs(case, seed)
        e = _Exact(spec, len(omegas))
        e.init(np.zeros((0, 5)))
        e.sources(ring, 1.0, omegas)
        return e.record([probe], case["steps"])[:, 0, -(case["steps"] // 4):].abs().amax(1)
    if form == "spectrum":
        return _peak_table(_series(case, seed), case["modes"])
    x, t, order = _net_inputs(case, seed)
    p = torch.from_numpy(_params(case, seed)).to(DEV)
    x, t = (torch.from_numpy(v).to(DEV).double() for v in (x, t))
    if form == "predict":
        layers = [(A.to(torch.bfloat16) if case["bf16"] else A, b) for A, b in _layers(case, p)]
        return _forward([(A.double(), b.double()) for A, b in layers], x)
    p = p.double()
    if form == "grad":
        loss, g = _loss_grad(case, p, x, t)
        return {"loss": loss, "grad": g}
    b, curve = min(case["batch"], case["samples"]), []
    m, v = torch.zeros_like(p), torch.zeros_like(p)
    for s in range(case["steps"]):
        rows = torch.from_numpy(order[s * b:(s + 1) * b].astype(np.int64)).to(DEV)
        loss, g = _loss_grad(case, p, x[rows], t[rows])
        curve.append(loss)
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        p = p - 1e-3 * (m / (1 - 0.9 ** (s + 1))) / ((v / (1 - 0.999 ** (s + 1))).sqrt() + 1e-8)
    return {"loss": torch.stack(curve), "params": p}
