"""Timed cases of the framework: foam runs through its public entry points.

A case is a dict of plain values. `prepare` builds what a user's program holds
before the call (a box with its initial state, or a batch of boxes); `run`
advances it by the case's number of time steps and reads the result back as
torch CUDA tensors, as a program that keeps working on the GPU does; `exact`
computes the same outputs in FP64 with plain torch operations, from the
equations alone.

Kinds:
  box       one box, sim.step(steps), the populations read back (the state a
            run resumes from), with the blocked-edge mask where the film
            barrier is on
  grow      the same with the growth source (gas released every step)
  two       a two-component box (melt and gas lattices)
  batch     many boxes advanced together, their densities read back
  diagnose  every diagnostic of a state: bubble statistics with a size
            histogram, the bubbles' areas, densities, velocities, pressure,
            labels
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_1708_01613_gb300 import Batch, Simulation, make_config

# Coexisting liquid and gas densities at G = -5.5 (psi = 1 - exp(-rho), tau = 1).
RHO_L, RHO_G = 2.306865, 0.104158
G, WIDTH, ZONE, EPS, THRESHOLD = -5.5, 4.0, 4, 1e-6, math.log(2.0)
G_MG = 1.0  # two components: melt-gas coupling
GAS_IN, GAS_OUT = 0.305, 0.005  # two components: gas density inside and outside bubbles


def _box(name, nx, ny, steps, *, kind="box", storage="f32", barrier=True, every=10, tau=1.0, scene="foam",
         bubbles=0, rmin=8.0, rmax=64.0):
    return {"name": name, "kind": kind, "nx": nx, "ny": ny, "steps": steps, "storage": storage, "barrier": barrier,
            "every": every, "tau": tau, "scene": scene, "bubbles": bubbles, "rmin": rmin, "rmax": rmax}


def listed():
    return [
        # phase separation of a noisy density in a small box, the parameter-study run: one
        # launch after another, each a few microseconds of work
        _box("spinodal_128", 128, 128, 100, barrier=False, scene="noise"),
        # two bubbles and the film between them at the paper's cadence (the barrier is found
        # anew every step): the smallest barrier run, launches only
        _box("film_160x80_every_step", 160, 80, 20, every=1, scene="pair", bubbles=2, rmin=20.0, rmax=20.0),
        # clustered foam of touching bubbles, the ordinary single run; the state fits the L2
        _box("foam_1024_f16", 1024, 1024, 50, storage="f16", scene="cluster", bubbles=20, rmin=10.0, rmax=40.0),
        # the growth source on an ordinary run (gas released every step to the gas points of
        # the latest census)
        _box("grow_1024", 1024, 1024, 20, kind="grow", every=5, scene="cluster", bubbles=20, rmin=10.0, rmax=40.0),
        # a served request of any integer side: rows that start on no 16-byte boundary
        _box("request_1531_f16", 1531, 1531, 40, storage="f16", bubbles=60, rmin=4.0, rmax=48.0),
        # plain Shan-Chen in BF16 with a relaxation time other than one (another viscosity)
        _box("relax_2000x1504_bf16", 2000, 1504, 40, storage="bf16", barrier=False, tau=0.8, bubbles=30),
        # melt and gas lattices
        _box("two_component_2048", 2048, 2048, 10, kind="two", bubbles=25),
        # the paper's cadence on a large box: half of the time goes to the barrier
        _box("foam_4096_every_step", 4096, 4096, 4, every=1, bubbles=100),
        # the headline box, both storages of the headline
        _box("foam_8192_f32", 8192, 8192, 10, bubbles=400),
        _box("foam_8192_f16", 8192, 8192, 10, storage="f16", bubbles=400),
        # independent boxes of mixed integer sides advanced together
        _batch("batch_16_f16", 16, 256, 2048, 50),
        # what a run reads out at its checkpoints
        _box("diagnose_4096", 4096, 4096, 10, kind="diagnose", bubbles=100),
    ]


def _batch(name, count, lo, hi, steps, *, storage="f16", every=10, rates=False):
    return {"name": name, "kind": "batch", "count": count, "lo": lo, "hi": hi, "steps": steps, "storage": storage,
            "every": every, "rates": rates}


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the listed ranges: any kind, sides log-uniform from 100 to 8192 (any integer, every second
    a multiple of 16), at most the largest listed box's cost."""
    kind = rng.choice(["box", "box", "box", "box", "grow", "two", "batch", "diagnose"])
    if kind == "batch":
        c = _batch("", rng.randint(4, 20), 256, _log(rng, 500, 2048), 10 * rng.randint(2, 5),
                   storage=rng.choice(["f16", "f16", "f32"]), rates=rng.random() < 0.5)
        del c["name"]
        return c
    hi = {"box": 8192, "grow": 2500, "two": 4096, "diagnose": 4500}[kind]
    nx = _log(rng, 100, hi)
    ny = max(100, min(hi, int(nx * math.exp(rng.uniform(-0.7, 0.7)))))
    if rng.random() < 0.5:
        nx = max(112, nx // 16 * 16)
    storage = rng.choice(["f32", "f16", "bf16"]) if kind == "box" else "f32"
    barrier = kind != "box" or rng.random() < 0.75
    every = rng.choice([1, 5, 10, 10])
    most = {"box": 4.0e8, "grow": 1.2e8, "two": 1.2e8, "diagnose": 2.0e8}[kind] / (2 if every == 1 else 1)
    steps = max(4, min(100, int(most / (nx * ny)), rng.randint(10, 100)))
    scene = rng.choice(["foam", "cluster"]) if kind != "box" or barrier else rng.choice(["foam", "noise"])
    small = min(nx, ny)
    c = _box("", nx, ny, steps, kind=kind, storage=storage, barrier=barrier, every=every,
             tau=rng.choice([1.0, 1.0, 0.8]) if kind == "box" else 1.0, scene=scene,
             bubbles=0 if scene == "noise" else max(2, min(400, int(nx * ny / rng.uniform(5e4, 1.7e5)))),
             rmin=8.0, rmax=float(min(64, small // 6)))
    if c["kind"] == "diagnose":
        c["steps"] = min(c["steps"], 10)
    del c["name"]
    return c


# ----------------------------------------------------------------- inputs
def _bubbles(nx, ny, n, rmin, rmax, scene, seed):
    """(n, 3) centres and radii on the torus, no two closer than 2 cells: anywhere ("foam"), each 2 to 6
    cells off an earlier one where that fits ("cluster"), or two with a film of 3 cells ("pair")."""
    r = random.Random(seed)
    if scene == "pair":
        x, y, rad = r.uniform(0, nx), r.uniform(0, ny), rmin
        return np.array([[x, y, rad], [(x + 2 * rad + 3.0) % nx, y, rad]])
    size = np.array([nx, ny], np.float64)
    out = np.empty((n, 3))
    k = 0
    for attempt in range(400 * n):
        if k == n:
            break
        rad = math.exp(r.uniform(math.log(rmin), math.log(max(rmin, rmax))))
        c = np.array([r.uniform(0, nx), r.uniform(0, ny)])
        if scene == "cluster" and k:
            j, a = r.randrange(k), r.uniform(0, 2 * math.pi)
            c = (out[j, :2] + (out[j, 2] + rad + r.uniform(2.0, 6.0)) * np.array([math.cos(a), math.sin(a)])) % size
        d = np.abs(out[:k, :2] - c)
        d = np.minimum(d, size - d)
        if 2 * rad + 2 < min(nx, ny) and (np.hypot(d[:, 0], d[:, 1]) - out[:k, 2] - rad >= 2.0).all():
            out[k] = c[0], c[1], rad
            k += 1
    return out[:k].copy()


def _noise(nx, ny, seed, device):
    g = torch.Generator(device="cpu").manual_seed(seed)
    u = torch.rand(ny, nx, generator=g, dtype=torch.float64)
    return (0.7 * (1.0 + 0.01 * (2.0 * u - 1.0))).to(device)


def _profile(nx, ny, bubbles, device):
    """tanh profile of the nearest bubble's surface, FP64."""
    s = torch.full((ny, nx), float("inf"), dtype=torch.float64, device=device)
    for cx, cy, r in bubbles.tolist():
        reach = int(r + 20 * WIDTH / 2) + 3  # beyond 20 half-widths tanh is 1 in FP64
        whole = 2 * reach + 1 >= min(nx, ny)
        xs = torch.arange(nx) if whole else torch.arange(int(cx) - reach, int(cx) + reach + 1) % nx
        ys = torch.arange(ny) if whole else torch.arange(int(cy) - reach, int(cy) + reach + 1) % ny
        xs, ys = xs.to(device), ys.to(device)
        dx, dy = (xs.double() - cx).abs(), (ys.double() - cy).abs()
        dx, dy = torch.minimum(dx, nx - dx), torch.minimum(dy, ny - dy)
        d = torch.sqrt(dx[None, :] ** 2 + dy[:, None] ** 2) - r
        s[ys[:, None], xs[None, :]] = torch.minimum(s[ys[:, None], xs[None, :]], d)
    return 0.5 * (RHO_L + RHO_G) + 0.5 * (RHO_L - RHO_G) * torch.tanh(s / (WIDTH / 2))


def _density(case, seed, device):
    if case["scene"] == "noise":
        return _noise(case["nx"], case["ny"], seed, device)
    return _profile(case["nx"], case["ny"], _scene(case, seed), device)


def _scene(case, seed):
    return _bubbles(case["nx"], case["ny"], case["bubbles"], case["rmin"], case["rmax"], case["scene"], seed)


def _nuclei(case, seed):
    r = random.Random(seed + 1)
    return np.array([[r.uniform(0, case["nx"]), r.uniform(0, case["ny"]), r.uniform(3.0, 8.0)] for _ in range(12)])


GROWTH_RATE, GROWTH_BUDGET = 1.0, 1e4  # gas mass per step, in all


def _members(case, seed):
    """The boxes of a batch: the same sides for every seed, bubbles of the seed."""
    r = random.Random(1000 * case["count"] + case["hi"])
    out = []
    for k in range(case["count"]):
        side = _log(r, case["lo"], case["hi"])
        n = max(2, min(_log(r, 5, 200), side * side // 4000))
        rmax = max(6.0, min(48.0, 0.33 * side / math.sqrt(n)))
        out.append({"nx": side, "ny": side, "scene": "foam", "bubbles": n, "rmin": 6.0, "rmax": rmax,
                    "steps": _log(r, max(1, case["steps"] // 8), case["steps"]) if case["rates"] else case["steps"],
                    "seed": 1009 * seed + k})
    return out


def _gas_of(rho_m):
    return GAS_OUT + (GAS_IN - GAS_OUT) * (RHO_L - rho_m) / (RHO_L - RHO_G)


# ----------------------------------------------------------------- prepare and run
class _State:
    pass


def _simulation(case, **kw):
    return Simulation(make_config(case["nx"], case["ny"], storage=case["storage"], barrier=case["barrier"],
                                  relabel_every=case["every"], tau=case["tau"],
                                  rho_ref=0.7 if case["scene"] == "noise" else RHO_L, G=G, **kw))


def prepare(case, seed):
    st = _State()
    st.case = case
    kind = case["kind"]
    if kind == "batch":
        st.members = _members(case, seed)
        st.sims = []
        for m in st.members:
            sim = Simulation(make_config(m["nx"], m["ny"], storage=case["storage"], barrier=True,
                                         relabel_every=case["every"], rho_ref=RHO_L, G=G))
            sim.init_bubbles(_scene(m, m["seed"]), RHO_L, RHO_G, WIDTH)
            st.sims.append(sim)
        st.batch = Batch(st.sims)
        st.rates = [m["steps"] for m in st.members]
        return st
    if kind == "two":
        st.sim = _simulation(case, components=2, G_mg=G_MG)
        rho = _density(case, seed, "cuda").float().double()
        st.sim.init_density(rho.cpu().numpy(), _gas_of(rho).cpu().numpy())
        return st
    st.sim = _simulation(case, growth=kind == "grow")
    if case["scene"] == "noise":
        st.sim.init_density(_noise(case["nx"], case["ny"], seed, "cuda"))
    else:
        st.sim.init_bubbles(_scene(case, seed), RHO_L, RHO_G, WIDTH)
    if kind == "grow":
        st.sim.nucleate(_nuclei(case, seed), RHO_G)
        st.sim.set_growth(GROWTH_RATE, GROWTH_BUDGET)
    if kind == "diagnose":
        st.sim.step(case["steps"])
        st.sim.sync()
    return st


def run(state):
    case = state.case
    kind = case["kind"]
    if kind == "batch":
        if case["rates"]:
            state.batch.step_each(state.rates)
        else:
            state.batch.step(case["steps"])
        return [s.read("rho", device=True)["rho"] for s in state.sims]
    if kind == "diagnose":
        out = state.sim.read("rho", "ux", "uy", "p", "label", "owner", "mask", "open", device=True)
        st = state.sim.stats(nbins=32, dmin=4.0, dmax=256.0)
        out["labels"], out["areas"] = state.sim.bubble_areas()
        out.update(n_bubbles=st["n_bubbles"], n_open=st["n_open"], n_merges=st["n_merges"], hist=st["hist"],
                   gas_fraction=st["gas_fraction"], mean_diameter=st["mean_diameter"], mass=st["mass"])
        return out
    state.sim.step(case["steps"])
    return state.sim.read(*(("pops", "mask") if case["barrier"] else ("pops",)), device=True)


# Floating-point operations of one cell and time step (moments 27, psi 4, force 20, equilibrium and
# collision 60, with the barrier's and the stores' conversions left out).
_CELL_FLOPS = 110


def work(case):
    """Per time step each population is read once and written once (with the barrier also one mask byte per
    cell); what is read back is one pass over the populations and the output written."""
    kind = case["kind"]
    if kind == "batch":
        eb = 4 if case["storage"] == "f32" else 2
        m = _members(case, 0)
        cells = sum(b["nx"] * b["ny"] for b in m)
        steps = sum(b["nx"] * b["ny"] * b["steps"] for b in m)
        return {"bytes": steps * (18 * eb + 1) + cells * (9 * eb + 4), "flops": steps * _CELL_FLOPS}
    cells = case["nx"] * case["ny"]
    eb = 4 if case["storage"] == "f32" else 2
    planes = 18 if kind == "two" else 9
    if kind == "diagnose":  # the populations and the mask read once, each field written once, owner, mask and open copied
        return {"bytes": cells * (9 * eb + 1 + 5 * 4 + 2 * 6), "flops": cells * 80}
    mask = 1 if case["barrier"] else 0
    return {"bytes": case["steps"] * cells * (2 * planes * eb + mask) + cells * (planes * (eb + 4) + 2 * mask),
            "flops": case["steps"] * cells * _CELL_FLOPS * planes / 9}


# ----------------------------------------------------------------- FP64 in plain torch
_EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
_EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
_W = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
_OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)


def _at(a, i):
    """a(x + e_i) on the torus."""
    return torch.roll(a, (-_EY[i], -_EX[i]), (0, 1)) if i else a


def _psi(rho):
    return 1.0 - torch.exp(-rho)


def _labels(gas):
    """4-connected gas components on the torus, each by its smallest row-major index; -1 elsewhere."""
    ny, nx = gas.shape
    none = nx * ny
    label = torch.where(gas, torch.arange(none, device=gas.device).reshape(ny, nx), none)
    for _ in range(4 * (nx + ny)):
        low = label
        for i in (1, 2, 3, 4):
            low = torch.minimum(low, _at(label, i))
        low = torch.where(gas, low, none)
        flat = torch.cat([low.reshape(-1), low.new_full((1,), none)])
        for _ in range(3):  # a label's own label is a smaller index of the same component
            flat = torch.cat([torch.minimum(flat[:-1], flat[flat[:-1]]), flat[-1:]])
        low = flat[:-1].reshape(ny, nx)
        if torch.equal(low, label):
            break
        label = low
    return torch.where(gas, label, -1)


class _Exact:
    """One box in FP64: `f` holds the incoming populations, [components][9][ny][nx]."""

    def __init__(self, rho, *, barrier, every, tau, growth=0.0, budget=0.0):
        self.f = torch.stack([torch.stack([w * r for w in _W]) for r in rho])
        self.barrier, self.every, self.tau, self.rate, self.budget = barrier, every, tau, growth, budget
        self.t, self.released = 0, 0.0
        ny, nx = rho[0].shape
        self.g = ((G,),) if len(rho) == 1 else ((G, G_MG), (G_MG, 0.0))
        self.mask = torch.zeros(ny, nx, dtype=torch.uint8, device=rho[0].device)
        self.open = torch.zeros_like(self.mask, dtype=torch.bool)
        self.sign = torch.zeros_like(self.mask, dtype=torch.int8)
        self.gas = None

    def pressure(self, rho, psi):
        p = sum(rho) / 3.0
        for a in range(len(rho)):
            for b in range(len(rho)):
                p = p + self.g[a][b] * psi[a] * psi[b] / 6.0
        return p

    def relabel(self, rho):
        self.gas = rho[0] < THRESHOLD
        if not self.barrier:
            return
        label = _labels(self.gas)
        owner = label.clone()
        found = label >= 0
        near = {}
        for dy in range(-ZONE, ZONE + 1):
            for dx in range(-ZONE, ZONE + 1):
                if 0 < dx * dx + dy * dy <= ZONE * ZONE:
                    near.setdefault(dx * dx + dy * dy, []).append((dx, dy))
        big = label.numel()
        for d2 in sorted(near):
            lo = torch.full_like(label, big)
            hi = torch.full_like(label, -1)
            for dx, dy in near[d2]:
                n = torch.roll(label, (-dy, -dx), (0, 1))
                lo = torch.minimum(lo, torch.where(n >= 0, n, big))
                hi = torch.maximum(hi, n)
            here = ~found & (hi >= 0)
            owner = torch.where(here, torch.where(lo == hi, lo, -2), owner)
            found |= here
        p = self.pressure(rho, [_psi(r) for r in rho])
        second, chosen = torch.zeros_like(p), torch.zeros_like(self.open)
        for i in range(1, 9):
            n = _at(owner, i)
            here = ~chosen & (owner != -1) & (n != -1) & (n != owner)
            second = torch.where(here, _at(p, i) - 2.0 * p + _at(p, _OPP[i]), second)
            chosen |= here
        sign = torch.where(chosen, torch.sign(second), torch.zeros_like(second)).to(torch.int8)
        self.open |= chosen & ((second.abs() <= EPS) | ((self.sign != 0) & (sign != self.sign)))
        self.sign = sign
        self.mask.zero_()
        for i in range(1, 9):
            n = _at(owner, i)
            cut = (owner != -1) & (n != -1) & (n != owner) & ~self.open & ~_at(self.open, i)
            self.mask |= cut.to(torch.uint8) << (i - 1)

    def blocked(self, i):
        return ((self.mask >> (i - 1)) & 1).bool()

    def moments(self):
        rho = [f.sum(0) for f in self.f]
        jx = [sum(_EX[i] * f[i] for i in range(9) if _EX[i]) for f in self.f]
        jy = [sum(_EY[i] * f[i] for i in range(9) if _EY[i]) for f in self.f]
        return rho, jx, jy

    def forces(self, rho):
        psi = [_psi(r) for r in rho]
        sums = []
        for p in psi:
            sx, sy = torch.zeros_like(p), torch.zeros_like(p)
            for i in range(1, 9):
                n = torch.where(self.blocked(i), p, _at(p, i)) if self.barrier else _at(p, i)
                sx, sy = sx + _W[i] * _EX[i] * n, sy + _W[i] * _EY[i] * n
            sums.append((sx, sy))
        return [tuple(-psi[a] * sum(self.g[a][b] * sums[b][d] for b in range(len(rho))) for d in (0, 1))
                for a in range(len(rho))]

    def step(self):
        rho, jx, jy = self.moments()
        if self.t % self.every == 0:
            self.relabel(rho)
        force = self.forces(rho)
        den = sum(rho)
        ux, uy = sum(jx) / den, sum(jy) / den  # equal relaxation times
        for a in range(len(rho)):
            vx, vy = ux + self.tau * force[a][0] / rho[a], uy + self.tau * force[a][1] / rho[a]
            base = 1.0 - 1.5 * (vx * vx + vy * vy)
            out = torch.empty_like(self.f[a])
            for i in range(9):
                e = _EX[i] * vx + _EY[i] * vy
                out[i] = self.f[a][i] + (_W[i] * rho[a] * (base + 3.0 * e + 4.5 * e * e) - self.f[a][i]) / self.tau
            if self.rate:
                n = int(self.gas.sum())
                give = min(self.rate, self.budget - self.released) if n else 0.0
                self.released += give
                for i in range(9):
                    out[i] += torch.where(self.gas, _W[i] * give / max(n, 1), 0.0)
            for i in range(9):
                self.f[a][i] = _at(out[i], _OPP[i])
                if self.barrier and i:  # what would cross a blocked edge returns to its own cell
                    self.f[a][i] = torch.where(self.blocked(_OPP[i]), out[_OPP[i]], self.f[a][i])
        self.t += 1


def exact(case, seed):
    """What run() returns on a fresh state, in FP64; no value for labels, masks and the rupture state."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    kind = case["kind"]
    if dev == "cpu" and kind != "batch" and case["nx"] * case["ny"] * case["steps"] > 2e7:
        return None
    if kind == "batch":
        out = []
        for m in _members(case, seed):
            e = _Exact([_density(m, m["seed"], dev)], barrier=True, every=case["every"], tau=1.0)
            for _ in range(m["steps"]):
                e.step()
            out.append(e.f[0].sum(0))
        return out
    rho = _density(case, seed, dev)
    if kind == "two":
        rho = rho.float().double()
        rho = [rho, _gas_of(rho)]
    else:
        rho = [rho]
    if kind == "grow":
        x = torch.arange(case["nx"], device=dev).double()
        y = torch.arange(case["ny"], device=dev).double()
        for cx, cy, r in _nuclei(case, seed).tolist():
            dx, dy = (x - cx).abs(), (y - cy).abs()
            dx, dy = torch.minimum(dx, case["nx"] - dx), torch.minimum(dy, case["ny"] - dy)
            rho[0][dx[None, :] ** 2 + dy[:, None] ** 2 <= r * r] = RHO_G
    e = _Exact(rho, barrier=case["barrier"], every=case["every"], tau=case["tau"],
               growth=GROWTH_RATE if kind == "grow" else 0.0, budget=GROWTH_BUDGET)
    for _ in range(case["steps"]):
        e.step()
    if kind != "diagnose":
        out = {"pops": e.f.reshape(-1, case["ny"], case["nx"])}
        if case["barrier"]:
            out["mask"] = None
        return out
    (r,), (jx,), (jy,) = e.moments()
    (fx, fy), = e.forces([r])
    gas = r < THRESHOLD
    label = _labels(gas)
    areas = torch.unique(label[gas], return_counts=True)[1].double()
    return {"rho": r, "ux": (jx + 0.5 * fx) / r, "uy": (jy + 0.5 * fy) / r, "p": e.pressure([r], [_psi(r)]),
            "label": None, "owner": None, "mask": None, "open": None, "labels": None, "areas": areas,
            "n_bubbles": None, "n_open": None, "n_merges": None, "hist": None,
            "gas_fraction": float(gas.double().mean()),
            "mean_diameter": float((2.0 * torch.sqrt(areas / math.pi)).mean()) if areas.numel() else 0.0,
            "mass": float(r.sum())}
