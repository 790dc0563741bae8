"""Performance cases of the framework: the work its users have it do.

Three families, each through the public Python face:

  grid      one simulation domain (fdtd.Grid): a number of time steps, then
            the probe records of those steps and the six fields
  batch     many grounding domains advanced together (fdtd.Batch): a number
            of steps, then every domain's gap voltage
  predict   surrogate.Surrogate.predict: waveforms and predicted errors for
            rows of electrode parameters (host arrays in, host arrays out)
  train     one minibatch step of the surrogate network (gather, forward,
            loss, backward, Adam), as surrogate.fit runs it

``exact`` restates the method in 64 bits with plain torch: Yee updates with
averaged media, thin wires, CPML, Debye poles by the auxiliary differential
equation, current sources and probes; and the network with autograd.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2207_06908_gb300 import fdtd, mlp, surrogate
from paper_2207_06908_gb300 import workloads as W

EPS0, MU0 = 8.8541878128e-12, 1.25663706212e-6
CAPACITY = 1 << 17          # probe samples a grid can record
SHOWN = 10                  # domains of a batch whose fields come back with the traces


def listed():
    return [
        # a small closed box with a soil half-space and point probes: the first
        # thing a new user runs, and the size of parameter sweeps on one grid
        _grid("box_48", "box", (48, 48, 48), steps=100, cpml=0),
        # a small open domain of odd sides: nothing divides the tiles
        _grid("open_61x75x53", "ground", (61, 75, 53), steps=50, cpml=7, layers=2),
        # the apparent-resistivity electrode array over three dispersive layers
        _grid("array_100x100x80", "array", (100, 100, 80), steps=50, cpml=10, layers=3, poles=4),
        # a strike to a lattice tower of oblique wires
        _grid("tower_160x160x200", "tower", (160, 160, 200), steps=32, cpml=10),
        # the standard open grid: soil, 10-cell layer, base-fed vertical wire
        _grid("wire_256", "ground", (256, 256, 256), steps=20, cpml=10),
        # the same grid over a four-pole dispersive soil
        _grid("dispersive_256", "ground", (256, 256, 256), steps=12, cpml=10, poles=4),
        # the large grounding-mesh grid
        _grid("mesh_512x512x384", "mesh", (512, 512, 384), steps=8, cpml=12, layers=2),
        # a handful of surrogate-size domains: the re-runs of rejected inputs
        _batch("batch_8x64", 8, 64, 64, steps=100),
        # a sweep of uneven grounding domains
        _batch("batch_96_uneven", 96, 48, 128, steps=48),
        # one electrode asked for interactively; a design sweep
        dict(name="predict_1", kind="predict", rows=1),
        dict(name="predict_4096", kind="predict", rows=4096),
        # the training step at the default minibatch
        dict(name="train_256", kind="train", rows=256),
    ]


def draw(rng: random.Random):
    kind = rng.choice(["grid", "grid", "grid", "batch", "predict", "train"])
    if kind == "predict":
        return dict(kind=kind, rows=_log_int(rng, 2, 8192))
    if kind == "train":
        return dict(kind=kind, rows=_log_int(rng, 32, 4096))
    if kind == "batch":
        lo = rng.randint(48, 96)
        hi = rng.randint(lo, 128)
        k = _log_int(rng, 2, 96)
        c = _batch("", k, lo, hi, steps=max(8, min(rng.randint(16, 64), int(3e9 / (k * hi ** 3)))))
    else:
        layout = rng.choice(["box", "ground", "ground", "ground"])
        n = tuple(_log_int(rng, 40, 288) for _ in range(3))
        d = 0 if layout == "box" else rng.randint(4, 12)
        cells = n[0] * n[1] * n[2]
        c = _grid("", layout, n, steps=max(8, min(100, int(4e8 / cells)) + rng.randint(0, 3)), cpml=d,
                  layers=rng.randint(1, 3), poles=rng.choice([0, 0, 0, 1, 2, 4]) if layout == "ground" else 0)
    del c["name"]
    return c


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid(name, layout, n, steps, cpml, layers=1, poles=0):
    return dict(name=name, kind="grid", layout=layout, nx=n[0], ny=n[1], nz=n[2], steps=steps, cpml=cpml,
                layers=layers, poles=poles)


def _batch(name, domains, lo, hi, steps):
    """domains grounding domains with sides spread evenly over lo..hi"""
    return dict(name=name, kind="batch", domains=domains, lo=lo, hi=hi, steps=steps)


# ---- inputs ------------------------------------------------------------------
def _scenario(case, seed):
    """The domain of a grid case; soil, source and pole values from the seed."""
    rng = np.random.default_rng([7, seed])
    n, d = (case["nx"], case["ny"], case["nz"]), case["cpml"]
    soil = lambda: (float(rng.uniform(4.0, 40.0)), float(10 ** rng.uniform(-4.0, -1.0)), 1.0)
    amp = float(rng.uniform(0.5, 2.0))
    if case["layout"] == "mesh":
        sc = W.config3(4000)
        sc.materials = [(1.0, 0.0, 1.0), soil(), soil()]
    elif case["layout"] == "array":
        sc = W.three_layer_array(4000)
        # the array's pulse starts at step 1941: take it from there
        sc.sources = [(nd, ax, amp * np.asarray(cur)[1900:]) for nd, ax, cur in sc.sources]
        sc.debye = {m: (list(np.asarray(de) * rng.uniform(0.8, 1.2)), list(ta)) for m, (de, ta) in sc.debye.items()}
    elif case["layout"] == "tower":
        sc = W.lightning_tower("oblique", 4000, i0=1e4 * amp, n=n)
        sc.materials = [(1.0, 0.0, 1.0), soil()]
    else:
        dx = 0.5
        dt = W.time_step(dx, 0.99)
        cx, cy, ks = n[0] // 2, n[1] // 2, n[2] // 2
        depth = max(1, (ks - d) // (2 * case["layers"]))
        blocks = [((0, 0, 0), (n[0], n[1], ks - depth * q), q + 1) for q in range(case["layers"])]
        mats = [(1.0, 0.0, 1.0)] + [soil() for _ in range(case["layers"])]
        t = W.sample_times(4000, dx, 0.99)
        if case["layout"] == "box":
            sc = W.Scenario("box", n, dx, 0.99, 0, W.paint_blocks(n, blocks), mats,
                            sources=[((cx, cy, ks + 4), 2, amp * W.gaussian_derivative(t, 20 * dt, 120 * dt))],
                            probes=[(W.PROBE_E, (cx + 6, cy, ks + 4), 2, 1), (W.PROBE_E, (cx, cy + 6, ks - 4), 2, 1),
                                    (W.PROBE_E, (cx // 2, cy + cy // 2, ks + 6), 0, 1)])
        else:
            top = min(ks + 61, n[2] - d - 2)
            heights = [h for h in (ks + 1, ks + 16, ks + 31, ks + 46, ks + 60) if h < top]
            sc = W.Scenario("ground", n, dx, 0.99, d, W.paint_blocks(n, blocks), mats,
                            wires=[((cx, cy, ks + 1), (cx, cy, top), 0.005)],
                            sources=[((cx, cy, ks), 2, amp * W.ramp(t, 1e3, 0.25e-6))],
                            probes=[(W.PROBE_V, (cx, cy, ks), 2, 1)] +
                                   [(W.PROBE_I, (cx, cy, h), 2, 1) for h in heights])
            if case["poles"]:
                p, s = case["poles"], W.PAPER_SOIL
                sc.debye = {m: ([v * float(rng.uniform(0.5, 1.5)) for v in s["deps"][:p]], s["tau"][:p])
                            for m in range(1, case["layers"] + 1)}
    # the size of the fields follows the source: amperes in the box and the
    # array, kiloamperes elsewhere
    sc.fields = _fields(n, rng, 100.0 if case["layout"] in ("box", "array") else 1e4)
    return sc


def _fields(n, rng, size):
    """A smooth state as a run in progress has it: products of a few
    standing waves per axis that vanish on the low walls, E about `size` V/m
    and H that over 377 ohm.  Six (x, y, z) triples of vectors."""
    f = []
    for c in range(6):
        vs = []
        for m in n:
            x = np.arange(m) / m
            vs.append(sum(rng.uniform(-1, 1) * np.sin(math.pi * rng.integers(1, max(2, m // 8)) * x) for _ in range(3)))
        vs[2] = vs[2] * (size if c < 3 else size / 377.0)
        f.append([np.asarray(v, np.float32) for v in vs])
    return f


def _outer(v, dtype=torch.float32):
    x, y, z = (torch.as_tensor(a, device="cuda") for a in v)
    return (z[:, None, None] * y[None, :, None] * x[None, None, :]).to(dtype)


def _domains(case, seed):
    """The domains of a batch case: sides from the case, soils, rods and
    rises from the seed."""
    rng = np.random.default_rng([11, seed])
    out = []
    for n in _sides(case):
        lmax = min(10.0, W.GROUND_DX * (n - 28))
        sc = W.grounding_domain(n, float(rng.uniform(4.0, 40.0)), float(10 ** rng.uniform(-4.0, -1.0)),
                                float(rng.uniform(1.0, lmax)), 0.008, 0.0, 0.25e-6, n_steps=4000)
        sc.fields = _fields(sc.n, rng, 1e4)
        out.append(sc)
    return out


def _sides(case):
    k = case["domains"]
    # evenly spread, in a fixed mixed order as a parameter sweep meets them
    s = [case["lo"] + ((q * 37) % k) * (case["hi"] - case["lo"]) // max(1, k - 1) for q in range(k)]
    return [min(v, case["hi"]) for v in s]


def _params(case, seed):
    rng = np.random.default_rng([13, seed])
    r = case["rows"]
    depth = rng.uniform(0.0, 1.0, r)
    length = rng.uniform(1.0, 9.0 - depth)
    return np.stack([rng.uniform(4.0, 40.0, r), rng.uniform(-4.0, -1.0, r), length, rng.uniform(0.004, 0.016, r), depth,
                     rng.uniform(0.1e-6, 0.5e-6, r)], axis=1)


def _training(case, seed):
    """weights, encoded features, target waveforms, row weights and the
    minibatch of one training step"""
    rng = np.random.default_rng([17, seed])
    sizes = surrogate.MAIN_SIZES
    ws = []
    for k, n in zip(sizes[:-1], sizes[1:]):
        ws += [(rng.standard_normal((n, k)) * math.sqrt(2.0 / k)).astype(np.float32),
               (0.1 * rng.standard_normal(n)).astype(np.float32)]
    rows = case["rows"]
    total = 2 * rows
    F = rng.uniform(-1, 1, (total, sizes[0])).astype(np.float32)
    t = np.linspace(0.0, 1.0, sizes[-1])
    T = (np.exp(F[:, 1:2]) * (1 + 0.3 * F[:, 2:3] * np.exp(-t / (0.05 + 0.02 * F[:, 0:1] ** 2)))).astype(np.float32)
    w = (1.0 / np.sum(T.astype(np.float64) ** 2, axis=1)).astype(np.float32).reshape(-1, 1)
    idx = rng.permutation(total)[:rows].astype(np.int32)
    return ws, F, T, w, idx


LR = 1e-3


# ---- prepare and run ---------------------------------------------------------
def _build(sc):
    g = fdtd.from_scenario(sc, probe_capacity=CAPACITY)
    for c, v in enumerate(sc.fields):
        g.set_field(c, _outer(v).cpu().numpy())
    return g


def prepare(case, seed):
    kind = case["kind"]
    if kind == "grid":
        sc = _scenario(case, seed)
        return dict(kind=kind, grid=_build(sc), steps=case["steps"], views={},
                    probes=len(sc.probes) + len(sc.owire_probes))
    if kind == "batch":
        grids = [_build(sc) for sc in _domains(case, seed)]
        return dict(kind=kind, grids=grids, batch=fdtd.Batch(grids), steps=case["steps"], views={})
    if kind == "predict":
        return dict(kind=kind, net=surrogate.Surrogate.load(surrogate.WEIGHTS), params=_params(case, seed))
    ws, F, T, w, idx = _training(case, seed)
    rows = case["rows"]
    net = surrogate.Network(surrogate.MAIN_SIZES, [mlp.ACT_GELU] * 3 + [mlp.ACT_NONE], weights=ws)
    dev = lambda a: torch.as_tensor(a, device="cuda")
    new = lambda k: torch.empty((rows, k), dtype=torch.float32, device="cuda")
    return dict(kind=kind, net=net, F=dev(F), T=dev(T), w=dev(w), idx=dev(idx), xb=new(F.shape[1]), tb=new(T.shape[1]),
                wb=new(1), dy=new(T.shape[1]), loss=torch.zeros(1, device="cuda"))


class _Device:
    """a field array of a grid, for torch.as_tensor (which keeps this object,
    and with it the grid that owns the memory)"""

    def __init__(self, grid, ptr, pitch, plane):
        self.grid = grid
        self.__cuda_array_interface__ = dict(shape=grid.shape, typestr="<f4", data=(ptr, False), version=2,
                                             strides=(4 * plane, 4 * pitch, 4))


def _fields_of(g, views):
    """the grid's six current fields as device tensors (views of its own buffers)"""
    out = []
    for c in range(6):
        ptr, pitch, plane = g.field_device(c)
        if ptr not in views:
            views[ptr] = torch.as_tensor(_Device(g, ptr, pitch, plane), device="cuda")
        out.append(views[ptr])
    return out


def run(state):
    kind = state["kind"]
    if kind == "grid":
        g, steps = state["grid"], state["steps"]
        first = min(g.step_count, CAPACITY - steps)
        g.step(steps)
        probes = [g.read_probe(p, first, steps) for p in range(state["probes"])]
        return dict(probes=probes, fields=_fields_of(g, state["views"]))
    if kind == "batch":
        b, grids, steps = state["batch"], state["grids"], state["steps"]
        first = min(grids[0].step_count, CAPACITY - steps)
        b.step(steps)
        b.synchronize()
        gap = np.stack([g.read_probe(0, first, steps) for g in grids])
        return dict(gap=gap, fields=[_fields_of(g, state["views"]) for g in grids[:SHOWN]])
    if kind == "predict":
        wave, err = state["net"].predict(state["params"])
        return dict(wave=wave, err=err)
    net, idx = state["net"], state["idx"]
    mlp.gather_rows(state["F"], idx, state["xb"])
    mlp.gather_rows(state["T"], idx, state["tb"])
    mlp.gather_rows(state["w"], idx, state["wb"])
    out = net.forward(state["xb"])
    state["loss"].zero_()
    mlp.mse(out, state["tb"], 1.0 / idx.numel(), state["dy"], state["loss"], state["wb"])
    net.backward(state["dy"])
    net.adam(LR)
    return dict(loss=state["loss"], out=out, grads=net.g, params=net.params, bf16=net.Wb)


# ---- what a pass cannot do without ---------------------------------------------
def work(case):
    kind = case["kind"]
    if kind == "grid":
        b, f = _step_work((case["nx"], case["ny"], case["nz"]), case["cpml"])
        if case["poles"]:
            # below the surface: per cell three components' pole currents read and written
            soil = case["nx"] * case["ny"] * (60 if case["layout"] == "array" else case["nz"] // 2)
            b += soil * 3 * 8 * case["poles"]
            f += soil * 3 * 6 * case["poles"]
        return dict(bytes=b * case["steps"], flops=f * case["steps"])
    if kind == "batch":
        per = [_step_work((n, n, n), W.GROUND_CPML) for n in _sides(case)]
        return dict(bytes=sum(p[0] for p in per) * case["steps"], flops=sum(p[1] for p in per) * case["steps"])
    rows, sizes = case["rows"], surrogate.MAIN_SIZES
    weights = sum(a * b for a, b in zip(sizes[:-1], sizes[1:]))
    biases = sum(sizes[1:])
    if kind == "predict":
        hs = surrogate.HEAD_SIZES
        head = sum(a * b for a, b in zip(hs[:-1], hs[1:]))
        return dict(bytes=2 * (weights + head) + 4 * (biases + sum(hs[1:])) + 4 * rows * (6 + 512 + 1),
                    flops=2 * rows * (weights + head))
    # features, targets and row weights in; the output, gradients, updated
    # parameters, moments and BF16 weights out; the moments and parameters in
    return dict(bytes=4 * rows * (6 + 512 + 1 + 512) + weights * (2 + 4 + 12 + 12 + 2) + biases * (4 + 24),
                flops=2 * rows * (3 * weights - sizes[0] * sizes[1]))


def _step_work(n, d):
    """one time step: the six fields read and written and a class byte per
    cell; in the layer four auxiliaries per cell and axis read and written"""
    nx, ny, nz = n
    cells = nx * ny * nz
    slab = 2 * d * (ny * nz + nx * nz + nx * ny)
    return 49 * cells + 32 * slab, 36 * cells + 24 * slab


# ---- 64-bit restatement ----------------------------------------------------------
def _up(a, axis):
    """the neighbour at +1 along axis (0 = x), zero past the end"""
    dim = 2 - axis
    out = torch.zeros_like(a)
    m = a.shape[dim]
    out.narrow(dim, 0, m - 1).copy_(a.narrow(dim, 1, m - 1))
    return out


def _down(a, axis):
    """the neighbour at -1 along axis, zero past the end"""
    dim = 2 - axis
    out = torch.zeros_like(a)
    m = a.shape[dim]
    out.narrow(dim, 1, m - 1).copy_(a.narrow(dim, 0, m - 1))
    return out


def _mean4(v, c):
    """mean over the four cells around an edge along axis c"""
    for u in ((c + 1) % 3, (c + 2) % 3):
        v = 0.5 * (v + _down(v, u))
    return v


def _wire_factors(sc):
    """Thin wires: the on-wire E edges are conductors; around each node the
    radial E take eps and sigma times m = ln(1 / 0.23) / ln(dx / radius), and
    each H those E read takes mu / m; where wires meet the smaller m rules."""
    n, fe, fh, pec = sc.n, {}, {}, set()
    low = lambda f, key, m: f.__setitem__(key, min(m, f.get(key, m)))
    for p0, p1, radius in sc.wires:
        a = [u for u in range(3) if p1[u] != p0[u]][0]
        m = math.log(1 / 0.23) / math.log(sc.dx / radius)
        for s in range(p1[a] - p0[a] + 1):
            p = list(p0)
            p[a] += s
            for c in ((a + 1) % 3, (a + 2) % 3):
                for back in (0, 1):
                    q = list(p)
                    q[c] -= back
                    if any(q[u] < (0 if u == c else 1) or q[u] > n[u] - 1 for u in range(3)):
                        continue
                    low(fe, (c, *q), m)
                    for h, v in (((c + 2) % 3, (c + 1) % 3), ((c + 1) % 3, (c + 2) % 3)):
                        low(fh, (h, *q), m)
                        r = list(q)
                        r[v] -= 1
                        low(fh, (h, *r), m)
            if s < p1[a] - p0[a]:
                pec.add((a, *p))
    return fe, fh, pec


def _put(a, entries):
    """a[k, j, i] = value for each (i, j, k, value)"""
    if entries:
        i, j, k, v = zip(*entries)
        a[list(k), list(j), list(i)] = torch.tensor(v, dtype=a.dtype, device=a.device)


class _Exact:
    """One domain of a scenario advanced in 64 bits."""

    def __init__(self, sc):
        self.sc, self.n, self.dx = sc, sc.n, sc.dx
        self.dt = dt = W.time_step(sc.dx, sc.courant)
        f64 = dict(dtype=torch.float64, device="cuda")
        self.E = [_outer(v).double() for v in sc.fields[:3]]
        self.H = [_outer(v).double() for v in sc.fields[3:]]
        cm = torch.as_tensor(sc.cell_material, device="cuda").int()
        tab = torch.tensor(sc.materials, **f64)
        fe, fh, pec = _wire_factors(sc)
        at = lambda f, c: [(*k[1:], v) for k, v in f.items() if k[0] == c]
        npole = max([len(d) for d, _ in sc.debye.values()], default=0)
        self.ca, self.cb, self.db, self.pole = [], [], [], []
        for c in range(3):
            m = torch.ones(cm.shape, **f64)
            _put(m, at(fe, c))
            eps = EPS0 * m * _mean4(tab[:, 0][cm], c)
            sig = m * _mean4(tab[:, 1][cm], c)
            sb = torch.zeros_like(eps)
            pole = []
            for p in range(npole):
                de = torch.zeros(len(sc.materials), **f64)
                ta = torch.zeros(len(sc.materials), **f64)
                for mat, (dl, tl) in sc.debye.items():
                    if p < len(dl):
                        de[mat], ta[mat] = dl[p], tl[p]
                d4 = _mean4(de[cm], c)
                t4 = torch.where(d4 > 0, _mean4((de * ta)[cm], c) / d4.clamp_min(1e-300), torch.ones_like(d4))
                beta = 2 * EPS0 * d4 * m * dt / (2 * t4 + dt)
                k = torch.where(d4 > 0, (2 * t4 - dt) / (2 * t4 + dt), torch.zeros_like(d4))
                sb += beta
                pole.append([k, beta])
            D = 2 * eps + sb + sig * dt
            ca, cb = (2 * eps + sb - sig * dt) / D, 2 * dt / (D * self.dx)
            on = torch.ones(cm.shape, **f64)              # 0 on the walls and on the wires
            for u in ((c + 1) % 3, (c + 2) % 3):
                on.narrow(2 - u, 0, 1).zero_()
            _put(on, [(*k[1:], 0.0) for k in pec if k[0] == c])
            self.ca.append(ca * on)
            self.cb.append(cb * on)
            # per pole: the E update's factor, the current's decay and its gain
            self.pole.append([(-dt * (1 + k) / D * on * (b > 0), k, b / dt * on) for k, b in pole])
            m = torch.ones(cm.shape, **f64)
            _put(m, at(fh, c))
            mu = tab[:, 2][cm]
            db = dt * m / (MU0 * 0.5 * (mu + _down(mu, c)) * self.dx)
            db.narrow(2 - c, 0, 1).zero_()
            self.db.append(db)
        self.J = [[torch.zeros(cm.shape, **f64) for _ in range(npole)] for _ in range(3)]
        self.psi = {}
        self.step_no = 0

    def _layer(self, dif, c, u, at_half):
        """CPML of the difference along axis u: psi <- b psi + c dif,
        dif <- dif / kappa + psi in the two layers (kappa = 1, alpha = 0)"""
        d, n = self.sc.cpml, self.n[u]
        if not d:
            return dif
        sigma_max = 0.8 * 4.0 / (math.sqrt(MU0 / EPS0) * self.dx)
        for side in (0, 1):
            lo = 0 if side == 0 else n - d
            i = torch.arange(lo, lo + d, dtype=torch.float64, device="cuda") + (0.5 if at_half else 0.0)
            rho = (d - i) if side == 0 else (i - (n - d))
            b = torch.exp(-sigma_max * (rho / d) ** 3 * self.dt / EPS0)
            shape = [1, 1, 1]
            shape[2 - u] = d
            b = b.reshape(shape)
            part = dif.narrow(2 - u, lo, d)
            key = (c, u, at_half, side)
            psi = self.psi.get(key)
            psi = (b - 1) * part if psi is None else b * psi + (b - 1) * part
            self.psi[key] = psi
            part += psi
        return dif

    def step(self):
        E, H, sc = self.E, self.H, self.sc
        for c in range(3):
            a, b = (c + 1) % 3, (c + 2) % 3
            # dH_c/dt ~ dE_a/d_b - dE_b/d_a
            x = self._layer(_up(E[a], b) - E[a], c, b, True)
            x = x - self._layer(_up(E[b], a) - E[b], c, a, True)
            H[c] = H[c] + self.db[c] * x
        new = []
        for c in range(3):
            a, b = (c + 1) % 3, (c + 2) % 3
            x = self._layer(H[b] - _down(H[b], a), c, a, False)
            x = x - self._layer(H[a] - _down(H[a], b), c, b, False)
            e = self.ca[c] * E[c] + self.cb[c] * x
            for (cj, _, _), J in zip(self.pole[c], self.J[c]):
                e = e + cj * J
            new.append(e)
        for node, axis, cur in sc.sources:
            i, j, k = node
            if self.step_no < len(cur):
                new[axis][k, j, i] -= self.cb[axis][k, j, i] / self.dx * float(cur[self.step_no])
        for c in range(3):
            for p, (_, k, be) in enumerate(self.pole[c]):
                self.J[c][p] = k * self.J[c][p] + be * (new[c] - E[c])
        self.E = new
        self.step_no += 1

    def probe(self, kind, node, axis, edges):
        i, j, k = node
        if kind == W.PROBE_E:
            return self.E[axis][k, j, i]
        if kind == W.PROBE_V:
            run = [slice(q, q + 1) for q in node]
            run[axis] = slice(node[axis], node[axis] + edges)
            return -self.dx * self.E[axis][run[2], run[1], run[0]].sum()
        a, b = (axis + 1) % 3, (axis + 2) % 3
        before = lambda u: tuple(q - (1 if v == u else 0) for v, q in enumerate(node))
        at = lambda f, q: f[q[2], q[1], q[0]]
        return self.dx * ((at(self.H[b], node) - at(self.H[b], before(a))) -
                          (at(self.H[a], node) - at(self.H[a], before(b))))

    def run(self, steps, probes):
        rec = []
        for _ in range(steps):
            self.step()
            rec.append(torch.stack([self.probe(*p) for p in probes]))
        return torch.stack(rec, dim=1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "grid":
        sc = _scenario(case, seed)
        if sc.owires:
            return None                     # oblique wires: no plain restatement here
        x = _Exact(sc)
        rec = x.run(case["steps"], sc.probes)
        return dict(probes=list(rec), fields=x.E + x.H)
    if kind == "batch":
        gap, fields = [], []
        for q, sc in enumerate(_domains(case, seed)):
            x = _Exact(sc)
            gap.append(x.run(case["steps"], sc.probes[:1])[0])
            if q < SHOWN:
                fields.append(x.E + x.H)
        return dict(gap=torch.stack(gap), fields=fields)
    act = torch.nn.functional.gelu
    if kind == "predict":
        z = np.load(surrogate.WEIGHTS)
        p = _params(case, seed)
        cells = lambda v: np.rint(v / W.GROUND_DX) * W.GROUND_DX
        f = np.stack([(p[:, 0] - 22.0) / 18.0, (p[:, 1] + 2.5) / 1.5, (np.maximum(cells(p[:, 2]), W.GROUND_DX) - 5.0) / 4.0,
                      (np.log(p[:, 3]) - np.log(0.008)) / 0.7, (cells(p[:, 4]) - 0.5) / 0.5,
                      (p[:, 5] - 0.3e-6) / 0.2e-6], axis=1)
        out = {}
        for name, sizes in (("main", surrogate.MAIN_SIZES), ("head", surrogate.HEAD_SIZES)):
            h = torch.as_tensor(f, device="cuda")
            for l in range(len(sizes) - 1):
                bits = z[f"{name}_w{l}_bf16"].astype(np.uint32) << 16
                h = h @ torch.as_tensor(bits.view(np.float32), device="cuda").double().T + \
                    torch.as_tensor(z[f"{name}_b{l}"], device="cuda").double()
                h = act(h) if l < len(sizes) - 2 else h
            out[name] = h
        return dict(wave=100.0 * out["main"], err=torch.exp(out["head"][:, 0]))
    ws, F, T, w, idx = _training(case, seed)
    dev = lambda a: torch.as_tensor(a, device="cuda").double()
    F, T, w, idx = dev(F), dev(T), dev(w), torch.as_tensor(idx, device="cuda").long()
    master = [dev(a) for a in ws]
    # the forward and backward passes read the weights as they are stored for them, in BF16
    used = [torch.as_tensor(a, device="cuda").to(torch.bfloat16).double() if q % 2 == 0 else dev(a)
            for q, a in enumerate(ws)]
    used = [u.requires_grad_() for u in used]
    h = F[idx]
    for l in range(4):
        h = h @ used[2 * l].T + used[2 * l + 1]
        h = act(h) if l < 3 else h
    loss = (w[idx] * (h - T[idx]) ** 2).sum() / len(idx)
    grads = torch.autograd.grad(loss, used)
    params = [p - LR * g / (g.abs() + 1e-8) for p, g in zip(master, grads)]   # Adam's first step
    return dict(loss=loss.detach().reshape(1), out=h.detach(), grads=list(grads), params=params,
                bf16=[p.to(torch.float32).to(torch.bfloat16) for p in params[::2]])
