"""Performance cases of the lattice-Boltzmann Maxwell library, run through its Python entry points.

The work is what a user of the library has it do: the runs of the paper's Section IV (arXiv
2309.08068) on one-dimensional and cubic lattices, runs from a checkpoint, refinement sweeps as one
batch, and gradients of a plane loss. Sizes come from the library's own workloads
(``paper_2309_08068_gb300/workloads.py``), experiments, tests and benchmark. A pass starts from
fields or populations that the caller holds on the device, so it can be repeated on the same state.

Kinds of a case:
* ``run``      start from E and B, step, read E and B: one simulation.
* ``samples``  start from E and B, step to the last ``window`` steps, then one step and one field
               read at a time: how an amplitude is sampled for a fit (the skin-effect and dipole
               experiments).
* ``restart``  load populations with their time, step, read the populations back: one leg of a run
               between checkpoints.
* ``sweep``    the skin-effect test on cubes of growing size, stepped together as a ``Batch``.
* ``adjoint``  loss and gradients of a plane loss with respect to the medium.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2309_08068_gb300 import workloads as wl
from paper_2309_08068_gb300.lbm import Batch, Lattice

POPULATIONS = {"mm": 48, "hv": 36}  # moving values per cell
VALUE_BYTES = {"f32": 4, "f24": 3, "f16": 2, "bf16": 2}
# Additions and multiplications of one cell update as the method states it: moments, E and J,
# equilibria and collision of every value.
FLOPS = {"mm": 330, "hv": 250}
SCALE = {"f32": 0.0, "bf16": 0.0, "f16": 2.0 ** 20, "f24": 2.0 ** 20}  # fields of the order of 1e-4


def _case(kind, setup, model, shape, steps, storage="f32", **more):
    nx, ny, nz = shape
    return {"kind": kind, "setup": setup, "model": model, "nx": nx, "ny": ny, "nz": nz, "steps": steps,
            "storage": storage, **more}


def listed():
    return [
        # The smallest calls: the amplitude fit of the skin-effect experiment at its coarsest grid
        # samples the field after every single step of its last periods.
        dict(_case("samples", "skin", "mm", (1, 1, 500), 100, window=50), name="samples_1d_mm"),
        # The paper's one-dimensional runs (Sections IV-A, IV-B and IV-D): some thousand cells and
        # about as many steps. The test suite's dielectric pulse, and a skin-effect grid.
        dict(_case("run", "pulse", "mm", (1, 1, 1024), 1500), name="pulse_1d_mm"),
        dict(_case("run", "skin", "hv", (1, 1, 4000), 3000), name="skin_1d_hv"),
        # The dipole experiment (Section IV-C) on its coarse grids, for its own number of steps.
        dict(_case("run", "dipole", "mm", (32, 32, 32), 22), name="dipole_32_mm"),
        dict(_case("run", "dipole", "hv", (64, 64, 64), 95), name="dipole_64_hv"),
        # A ragged lattice of a few materials between two checkpoints, an odd number of steps.
        dict(_case("restart", "materials", "hv", (97, 53, 71), 25), name="restart_ragged_hv"),
        # The wide slab lattice of the accuracy tests: a material table, a long x axis.
        dict(_case("run", "slabs", "mm", (512, 64, 64), 60), name="slabs_mm"),
        # The benchmark's lattices, both models.
        dict(_case("run", "dipole", "mm", (256, 256, 256), 30), name="dipole_256_mm"),
        dict(_case("run", "dipole", "hv", (256, 256, 256), 30), name="dipole_256_hv"),
        # 16-bit storage, the throughput option, on a lattice well beyond the caches.
        dict(_case("run", "dipole", "mm", (208, 208, 208), 30, "bf16"), name="dipole_208_mm_bf16"),
        # The refinement sweep (cubes of 32, 48, ... cells) up to 112.
        dict(_case("sweep", "skin", "mm", (112, 112, 112), 56), name="sweep_mm"),
        # Inverse design: gradient with respect to a per-cell permittivity.
        dict(_case("adjoint", "medium", "mm", (128, 128, 128), 48, sigma=False), name="adjoint_128_mm"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


MOST = 16_000_000 * 30  # cell updates of a drawn case


def draw(rng):
    kind = rng.choice(["samples", "line", "line", "cube", "cube", "cube", "restart", "slabs", "sweep", "adjoint"])
    model = rng.choice(["mm", "hv"])
    if kind == "samples":
        window = rng.randint(20, 80)
        return _case("samples", "skin", model, (1, 1, _log(rng, 400, 8000)), window + rng.randint(20, 200), window=window)
    if kind == "line":  # the one-dimensional experiments: 256 to 8192 cells
        nz = _log(rng, 256, 8192)
        return _case("run", rng.choice(["pulse", "skin"]), model, (1, 1, nz), int(nz * rng.uniform(0.5, 1.5)))
    if kind == "cube":  # dipoles, not always exact cubes
        n = _log(rng, 24, 250)
        shape = tuple(max(20, int(n * rng.uniform(0.85, 1.15))) for _ in range(3))
        steps = max(2, min(rng.randint(16, 100), MOST // math.prod(shape)))
        storage = rng.choice(["f32", "f32", "f32", "bf16", "f16", "f24"])
        return _case("run", "dipole", model, shape, steps, storage)
    if kind == "restart":
        shape = tuple(_log(rng, 17, 160) for _ in range(3))
        return _case("restart", "materials", model, shape, rng.randint(1, 40))
    if kind == "slabs":
        shape = (_log(rng, 128, 600), _log(rng, 16, 96), _log(rng, 16, 96))
        return _case("run", "slabs", model, shape, rng.randint(10, 80))
    if kind == "sweep":
        n = 16 * rng.randint(3, 8)
        return _case("sweep", "skin", model, (n, n, n), rng.randint(n // 4, n // 2))
    n = _log(rng, 20, 120)
    shape = tuple(max(16, int(n * rng.uniform(0.85, 1.15))) for _ in range(3))
    return _case("adjoint", "medium", model, shape, rng.randint(8, 48), sigma=rng.random() < 0.5)


def _shape(case):
    return case["nx"], case["ny"], case["nz"]


def _sweep_sizes(case):
    """Cube edges 32, 48, ... up to the case's, and the steps of each in proportion to its edge."""
    sizes = list(range(32, case["nx"] + 1, 16))
    return [(n, max(1, case["steps"] * n // case["nx"])) for n in sizes]


# --- inputs ------------------------------------------------------------------------------------
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _skin(model, shape, rng, device):
    """Section IV-B: a plane wave imposed on the plane z = 0, a conductor from nz / 4 on."""
    nx, ny, nz = shape
    sigma = torch.zeros((nz, ny, nx), device=device)
    sigma[nz // 4:] = rng.uniform(0.002, 0.02) if nx * ny == 1 else rng.uniform(0.05, 0.2)
    e0 = rng.uniform(0.5, 2.0) * 1e-4
    src = wl.Source("impose", np.arange(nx * ny), wl.TimeFunction("sin", 1.0, rng.uniform(0.8, 1.6) * max(nz / 8, 24.0)),
                    E0=(e0, 0.0, 0.0), B0=(0.0, e0 / wl.LIGHT_SPEED[model], 0.0))
    return {"sigma": sigma.reshape(-1)}, [src]


def _waves(model, shape, rng, device, count=3, amplitude=1e-4):
    """E and B of a few plane waves that fit the periodic lattice: fields of a run under way."""
    nx, ny, nz = shape
    x, y, z = (torch.arange(m, device=device, dtype=torch.float64) * (2 * math.pi / m) for m in shape)
    E = torch.zeros((3, nz, ny, nx), device=device)
    B = torch.zeros_like(E)
    for _ in range(count):
        k = [rng.randint(0, max(1, m // 12)) for m in shape]
        k[rng.randrange(3)] += 1
        kv = np.array([ki / m for ki, m in zip(k, shape)])
        a = np.cross(kv, [rng.uniform(-1, 1) for _ in range(3)])
        a *= amplitude / max(np.linalg.norm(a), 1e-30)
        b = np.cross(kv / np.linalg.norm(kv), a) / wl.LIGHT_SPEED[model]
        phase = k[0] * x[None, None, :] + k[1] * y[None, :, None] + k[2] * z[:, None, None] + rng.uniform(0, 6.28)
        wave = torch.cos(phase)
        for c in range(3):
            E[c] += a[c] * wave
            B[c] += b[c] * wave
    return E.reshape(3, -1), B.reshape(3, -1)


def _inputs(case, seed):
    """What the caller holds: media (float32 per cell), sources, and E and B or populations."""
    rng = random.Random(int(seed))
    dev = _device()
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed))
    model, shape = case["model"], _shape(case)
    nx, ny, nz = shape
    n = nx * ny * nz
    media, sources, E, B, f = {}, [], torch.zeros((3, n), device=dev), torch.zeros((3, n), device=dev), None
    if case["setup"] == "skin":
        media, sources = _skin(model, shape, rng, dev)
    elif case["setup"] == "pulse":  # Section IV-A: a Gaussian pulse and a dielectric slab
        z = torch.arange(nz, device=dev, dtype=torch.float64)
        eps = torch.ones(nz, device=dev)
        eps[int(0.39 * nz):int(0.69 * nz)] = rng.uniform(1.5, 4.0)
        g = 1e-4 * torch.exp(-((z - rng.uniform(0.15, 0.25) * nz) / (rng.uniform(0.015, 0.03) * nz)) ** 2 / 2)
        E[0], B[1] = g, g / wl.LIGHT_SPEED[model]
        media = {"eps_r": eps}
    elif case["setup"] == "dipole":  # Section IV-C's current in a lattice with waves under way
        E, B = _waves(model, shape, rng, dev)
        cells, w = wl.dipole_cells(shape, tuple(m // 2 for m in shape))
        sources = [wl.Source("current", cells, wl.TimeFunction("sin", 1e-4, rng.uniform(16.0, 48.0), rng.uniform(0, 6.28)), w=w)]
    elif case["setup"] == "slabs":  # a plane pulse through 64 dielectric slabs along x
        per = np.array([rng.uniform(1.0, 8.0) for _ in range(64)])
        x = torch.arange(nx, device=dev)
        eps = torch.as_tensor(per, device=dev)[torch.clamp(x * 64 // nx, max=63)]
        g = 1e-4 * torch.exp(-((x - nx / 8) / (rng.uniform(0.02, 0.04) * nx)) ** 2 / 2)
        row = lambda v: v.to(torch.float32)[None, :].expand(ny * nz, nx).reshape(-1)  # noqa: E731
        E[1], B[2] = row(g), row(g * eps.sqrt() / wl.LIGHT_SPEED[model])
        media = {"eps_r": row(eps)}
    elif case["setup"] == "materials":  # five materials, a current and an imposed source, any state
        table = torch.tensor([[rng.uniform(1.0, 4.0), rng.uniform(1.0, 2.0), s] for s in (0.0, 0.0, 0.05, 0.1, 0.2)], device=dev)
        block = torch.randint(0, 5, (nz // 8 + 1, ny // 8 + 1, nx // 8 + 1), generator=gen, device=dev)
        for axis in range(3):
            block = block.repeat_interleave(8, axis)
        ids = block[:nz, :ny, :nx].reshape(-1)
        media = {"eps_r": table[ids, 0].contiguous(), "mu_r": table[ids, 1].contiguous(), "sigma": table[ids, 2].contiguous()}
        f = 1e-2 * torch.randn((wl.POPULATIONS[model], n), generator=gen, device=dev)
        cells = np.sort(np.array(rng.sample(range(n), 40)))
        fn = lambda: wl.TimeFunction("sin", rng.uniform(0.5, 2.0), rng.uniform(10.0, 40.0), rng.uniform(0, 6.28))  # noqa: E731
        w = np.array([[rng.gauss(0, 1e-2) for _ in range(3)] for _ in range(20)])
        sources = [wl.Source("current", cells[:20], fn(), w=w),
                   wl.Source("impose", cells[20:], fn(), E0=(1e-2, -2e-2, 1e-2), B0=(2e-2, 1e-2, -1e-2))]
    elif case["setup"] == "medium":  # a smooth random permittivity around a dipole
        E, B = _waves(model, shape, rng, dev)
        low = 1.0 + 3.0 * torch.rand((1, 1, nz // 8 + 2, ny // 8 + 2, nx // 8 + 2), generator=gen, device=dev)
        eps = torch.nn.functional.interpolate(low, size=(nz, ny, nx), mode="trilinear", align_corners=True)
        media = {"eps_r": eps.reshape(-1).contiguous()}
        cells, w = wl.dipole_cells(shape, tuple(m // 2 for m in shape))
        sources = [wl.Source("current", cells, wl.TimeFunction("sin", 1e-4, rng.uniform(16.0, 32.0)), w=w)]
    for s in sources:  # the library keeps weights and amplitudes in 32 bits
        if s.w is not None:
            s.w = np.asarray(s.w, np.float32)
        s.E0, s.B0 = (tuple(float(np.float32(v)) for v in q) for q in (s.E0, s.B0))
    return {"media": media, "sources": sources, "E": E, "B": B, "f": f, "t": rng.randint(1, 500) if f is not None else 0}


def _plane(case):
    """The loss plane: constant x, a quarter of the way in (away from the source in the middle)."""
    return 0, case["nx"] // 8


# --- one pass ----------------------------------------------------------------------------------
def _lattice(case, inp, stream=None):
    L = Lattice(case["model"], _shape(case), **inp["media"], storage=case["storage"], storage_scale=SCALE[case["storage"]],
                stream=stream)
    for s in inp["sources"]:
        L.add_source(s)
    return L


def prepare(case, seed):
    if case["kind"] == "sweep":  # a batch replays a captured graph on a stream of its own
        stream = torch.cuda.Stream()
        lats, steps, ins = [], [], []
        for k, (n, s) in enumerate(_sweep_sizes(case)):
            sub = dict(case, nx=n, ny=n, nz=n)
            ins.append(_inputs(sub, seed * 64 + k))
            lats.append(_lattice(sub, ins[-1], stream))
            steps.append(s)
        return {"case": case, "ins": ins, "lats": lats, "steps": steps, "batch": Batch(lats)}
    inp = _inputs(case, seed)
    state = {"case": case, "in": inp, "lat": _lattice(case, inp)}
    if case["kind"] == "samples":
        state["cells"] = torch.arange(case["nx"] * case["ny"] * case["nz"], device=_device())
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "sweep":
        for L, inp in zip(state["lats"], state["ins"]):
            L.init_fields(inp["E"], inp["B"])
        state["batch"].step(state["steps"])
        return [L.fields("EB") for L in state["lats"]]
    L, inp = state["lat"], state["in"]
    if case["kind"] == "restart":
        L.set_populations(inp["f"], inp["t"])
        L.step(case["steps"])
        return L.populations()
    L.init_fields(inp["E"], inp["B"])
    if case["kind"] == "samples":
        L.step(case["steps"] - case["window"])
        rows = []
        for _ in range(case["window"]):
            L.step(1)
            rows.append(L.fields("E")["E"][0].index_select(0, state["cells"]))
        return torch.stack(rows)
    if case["kind"] == "adjoint":
        loss, g_eps, g_sigma = L.adjoint(case["steps"], *_plane(case), sigma=case["sigma"])
        return {"loss": loss, "eps_r": g_eps} if g_sigma is None else {"loss": loss, "eps_r": g_eps, "sigma": g_sigma}
    L.step(case["steps"])
    return L.fields("EB")


def work(case):
    """Bytes: the caller's inputs and outputs, and the populations and media read and the populations
    written once by the call that steps (an adjoint: the populations and their adjoints). Operations:
    every cell update (an adjoint: a forward and a backward one)."""
    parts = [(n ** 3, s) for n, s in _sweep_sizes(case)] if case["kind"] == "sweep" else [(math.prod(_shape(case)), case["steps"])]
    cells = sum(n for n, _ in parts)
    updates = sum(n * s for n, s in parts)
    state = POPULATIONS[case["model"]] * VALUE_BYTES[case["storage"]]
    media = {"dipole": 0, "medium": 12}.get(case["setup"], 1)
    per_cell = 24 + 2 * state + media + 24  # E and B in, the populations in and out, E and B out
    if case["kind"] == "restart":
        per_cell = 2 * 4 * wl.POPULATIONS[case["model"]] + 2 * state + media
    elif case["kind"] == "samples":
        per_cell = 24 + 2 * state + media + 4 * case["window"]
    elif case["kind"] == "adjoint":
        per_cell = 24 + 4 * state + media + (8 if case["sigma"] else 4)
    flops = FLOPS[case["model"]] * updates * (2 if case["kind"] == "adjoint" else 1)
    return {"bytes": per_cell * cells, "flops": flops}


# --- the same in 64 bits, from the paper's formulas ----------------------------------------------
class _Exact:
    """One lattice in float64: populations before the collision, as tensors (.., nz, ny, nx).

    MM (Section II): f[r, d, j] with the 12 edge velocities v_d, e_d1 = -e_d0, b_dj = v_d x e_dj.
    HV (Section III): f[r, i, c] with the 6 axis velocities, r = 0 electric and 1 magnetic."""

    def __init__(self, case, inp):
        self.model, (self.nx, self.ny, self.nz) = case["model"], _shape(case)
        dev = _device()
        grid = (self.nz, self.ny, self.nx)
        m = {k: v.to(torch.float64).reshape(grid) for k, v in inp["media"].items()}
        one = torch.ones((), dtype=torch.float64, device=dev)
        self.er, self.mr, self.sg = m.get("eps_r", one), m.get("mu_r", one), m.get("sigma", 0 * one)
        self.sources, self.grid, self.dev = inp["sources"], grid, dev
        self.where = [torch.as_tensor(np.asarray(s.cells), dtype=torch.long, device=dev) for s in self.sources]
        self.w = [None if s.w is None else torch.as_tensor(s.w, device=dev).double().T.contiguous() for s in self.sources]
        self.v, self.e = [], []
        if self.model == "mm":
            for a, b in ((0, 1), (0, 2), (1, 2)):  # planes xy, xz, yz
                ring = []
                for i in range(1, 5):
                    u = [0, 0, 0]
                    u[a], u[b] = (round(math.sqrt(2) * f((2 * i - 1) * math.pi / 4)) for f in (math.cos, math.sin))
                    ring.append(np.array(u))
                self.v += ring
                self.e += [ring[(i + 2) % 4] / 2 for i in range(1, 5)]  # e_i0 = v_{[(i+2) mod 4]+1} / 2
            self.b = [np.cross(v, e) for v, e in zip(self.v, self.e)]
        else:
            self.v = [np.array(u) for u in ((1, 0, 0), (0, 1, 0), (-1, 0, 0), (0, -1, 0), (0, 0, -1), (0, 0, 1))]
        self.t = 0

    @staticmethod
    def _dot(a, X):
        out = 0
        for c in range(3):
            if a[c]:
                out = out + float(a[c]) * X[c]
        return out

    @staticmethod
    def _cross(v, X):
        """v x X for an axis vector v (3 tensors; 0 where a component vanishes)."""
        return [v[1] * X[2] - v[2] * X[1], v[2] * X[0] - v[0] * X[2], v[0] * X[1] - v[1] * X[0]]

    def _s(self, k, t):
        fn = self.sources[k].fn
        return fn.amplitude * math.sin(2 * math.pi * t / fn.period + fn.phase)

    def _current(self, t):
        J = None
        for k, s in enumerate(self.sources):
            if s.kind == "current":
                J = torch.zeros((3, math.prod(self.grid)), dtype=torch.float64, device=self.dev) if J is None else J
                J.index_add_(1, self.where[k], self.w[k] * self._s(k, t))
        return None if J is None else J.reshape((3,) + self.grid)

    def fields(self, f, t, er=None, sg=None):
        """E, B and J of the populations f at time t (the current of iteration t + 1)."""
        er, sg = self.er if er is None else er, self.sg if sg is None else sg
        J = self._current(t + 1)
        J = [0, 0, 0] if J is None else J
        if self.model == "mm":
            de, db = f[0, :, 0] - f[0, :, 1], f[1, :, 0] - f[1, :, 1]
            E, B = [], []
            for c in range(3):
                D = sum(float(self.e[d][c]) * de[d] for d in range(12) if self.e[d][c])
                E.append((D / er - J[c] / (2 * er)) / (1 + sg / (2 * er)))  # mu0 = 2
                B.append(sum(float(self.b[d][c]) * db[d] for d in range(12) if self.b[d][c]))
        else:
            D, B = f[0].sum(0), list(f[1].sum(0))
            E = [D[c] / (3 * er) for c in range(3)]
        return E, B, [sg * E[c] + J[c] for c in range(3)]

    def equilibrium(self, E, B, J, er, mr):
        if self.model == "mm":
            out = []
            for v, e, b in zip(self.v, self.e, self.b):
                s, ee, bb = self._dot(v, J) / 16, self._dot(e, E), self._dot(b, B)
                alpha, beta = er / 4 * ee + bb / (8 * mr), ee / 4 + bb / 8
                out.append(((s + alpha, s - alpha), (s + beta, s - beta)))
            return [[[out[d][r][j] for j in (0, 1)] for d in range(12)] for r in (0, 1)]
        D, H = [3 * er * E[c] for c in range(3)], [B[c] / (3 * mr) for c in range(3)]
        eq = [[], []]
        for v in self.v:
            vH, vE = self._cross(v, H), self._cross(v, E)
            eq[0].append([D[c] / 6 - vH[c] / 2 for c in range(3)])
            eq[1].append([B[c] / 6 + vE[c] / 2 for c in range(3)])
        return eq

    def start(self, E, B):
        E, B = (list(X.double().reshape((3,) + self.grid)) for X in (E, B))
        eq = self.equilibrium(E, B, [0 * E[0]] * 3, self.er, self.mr)
        return torch.stack([torch.stack([torch.stack([x + 0 * E[0] for x in q]) for q in r]) for r in eq])

    def from_canonical(self, p):
        if self.model == "mm":
            return p[:48].double().reshape((2, 12, 2) + self.grid)
        return p.double().reshape((2, 6, 3) + self.grid)

    def to_canonical(self, f):
        f = f.reshape(-1, math.prod(self.grid))
        if self.model == "mm":  # the rest populations are not kept
            f = torch.cat([f, torch.zeros((2, f.shape[1]), dtype=f.dtype, device=f.device)])
        return f

    def step(self, f, t, er=None, sg=None):
        """Iteration t + 1 of populations f: collision, imposed cells, advection."""
        er_, sg_ = self.er if er is None else er, self.sg if sg is None else sg
        E, B, J = self.fields(f, t, er_, sg_)
        eq = self.equilibrium(E, B, J, er_, self.mr)
        imposed = [k for k, s in enumerate(self.sources) if s.kind == "impose"]
        fixed, cells = None, None
        if imposed:
            vals = torch.zeros((6, math.prod(self.grid)), dtype=torch.float64, device=self.dev)
            for k in imposed:
                eb = torch.tensor(list(self.sources[k].E0) + list(self.sources[k].B0), dtype=torch.float64, device=self.dev)
                vals.index_add_(1, self.where[k], (eb * self._s(k, t + 1))[:, None].expand(6, self.where[k].numel()).contiguous())
            cells = torch.unique(torch.cat([self.where[k] for k in imposed]))
            at = vals[:, cells]
            pick = lambda x: x.reshape(-1)[cells] if x.ndim else x  # noqa: E731
            fixed = self.equilibrium(list(at[:3]), list(at[3:]), [0 * at[0]] * 3, pick(er_), pick(self.mr))
        out = [[], []]
        for r in (0, 1):
            for d, v in enumerate(self.v):
                new = []
                for j in range(f.shape[2]):
                    x = 2 * eq[r][d][j] - f[r, d, j]
                    if self.model == "hv" and r == 0 and v[j]:  # T_i = -(J . v_i) v_i / 2
                        x = x - J[j] / 2
                    if fixed is not None:
                        x = x.reshape(-1).index_copy(0, cells, fixed[r][d][j] + 0 * at[0]).reshape(self.grid)
                    new.append(x)
                out[r].append(torch.roll(torch.stack(new), (int(v[2]), int(v[1]), int(v[0])), (1, 2, 3)))
        return torch.stack([torch.stack(o) for o in out])

    def read(self, f, t):
        E, B, _ = self.fields(f, t)
        return {"E": torch.stack(E).reshape(3, -1), "B": torch.stack(B).reshape(3, -1)}


def _exact_adjoint(case, inp):
    """Loss and gradients by reverse accumulation through the steps, each recomputed from its state."""
    X = _Exact(case, inp)
    er = X.er.detach().clone().requires_grad_(True)
    sg = torch.zeros_like(er, requires_grad=True)
    axis, index = _plane(case)
    dim = 2 - axis
    with torch.no_grad():
        states = [X.start(inp["E"], inp["B"])]
        for t in range(case["steps"]):
            states.append(X.step(states[-1], t))
    loss, back, grads = 0.0, None, [torch.zeros_like(er), torch.zeros_like(er)]

    def plane_loss(f, t):
        E, _, _ = X.fields(f, t, er, sg)
        return sum((e.select(dim, index) ** 2).sum() for e in E)

    for t in range(case["steps"], -1, -1):  # dL / d(state t), and the medium's share of it
        f = states.pop().requires_grad_(True)
        parts = []
        if t >= 1:
            parts.append(plane_loss(f, t))
            loss += float(parts[0].detach())
        if back is not None:
            parts.append((X.step(f, t, er, sg) * back).sum())
        back, *g = torch.autograd.grad(sum(parts), [f, er, sg], allow_unused=True)
        for total, part in zip(grads, g):
            if part is not None:
                total += part
    out = {"loss": loss, "eps_r": grads[0].reshape(-1)}
    if case["sigma"]:
        out["sigma"] = grads[1].reshape(-1)
    return out


def exact(case, seed):
    if case["steps"] > 6000:  # minutes of small launches
        return None
    with torch.no_grad():
        if case["kind"] == "sweep":  # uniform in x and y: one column of each cube, spread over it
            out = []
            for k, (n, s) in enumerate(_sweep_sizes(case)):
                cube = _inputs(dict(case, nx=n, ny=n, nz=n), seed * 64 + k)
                src = cube["sources"][0]
                col = dict(cube, media={"sigma": cube["media"]["sigma"][:: n * n].contiguous()},
                           sources=[wl.Source(src.kind, np.array([0]), src.fn, E0=src.E0, B0=src.B0)])
                X = _Exact(dict(case, nx=1, ny=1, nz=n), col)
                f = X.start(torch.zeros((3, n), device=_device()), torch.zeros((3, n), device=_device()))
                for t in range(s):
                    f = X.step(f, t)
                out.append({q: v[:, :, None].expand(3, n, n * n).reshape(3, -1) for q, v in X.read(f, s).items()})
            return out
        inp = _inputs(case, seed)
        if case["kind"] != "adjoint":
            X = _Exact(case, inp)
            t0, steps = inp["t"], case["steps"]
            f = X.from_canonical(inp["f"]) if case["kind"] == "restart" else X.start(inp["E"], inp["B"])
            rows = []
            for t in range(t0, t0 + steps):
                f = X.step(f, t)
                if case["kind"] == "samples" and t + 1 > t0 + steps - case["window"]:
                    rows.append(X.fields(f, t + 1)[0][0].reshape(-1))
            if case["kind"] == "samples":
                return torch.stack(rows)
            return X.to_canonical(f) if case["kind"] == "restart" else X.read(f, t0 + steps)
    return _exact_adjoint(case, inp)
