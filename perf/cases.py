"""The work that users of this framework have it do, as cases that can be timed and checked.

Every case runs through the public entry points (``Simulation``, ``Batch``, ``EndpointProblem``
and the connectivity functions) on seeded synthetic inputs.  The sizes are the five benchmark
configurations' own, the connectivity workload's, and generic ones between and beside them
(odd sides, rate maps, the SNR rule).  A case is a dict of plain values; ``kind`` says which
entry point it goes through:

  step   a few coupled steps of a running simulation (no reset: it goes on from where it is)
  run    a whole run from the initial state, which the caller keeps on the device
  batch  a batch of uneven instances, tuned once, run from its initial state
  grad   loss and gradients of the endpoint problem (autograd), ``loss``: its loss alone
  graph  bin the neurons, connect the cones, adjacency list, breadth-first levels

``exact`` is the model in 64 bits, written here with torch tensors only.
"""
import math

import numpy as np
import torch

from paper_1405_3331_gb300 import autograd as A
from paper_1405_3331_gb300 import batch as B
from paper_1405_3331_gb300 import cue
from paper_1405_3331_gb300 import graph as G
from paper_1405_3331_gb300 import workloads as W

DEV = "cuda:0"
SNR = dict(gain=8.0, width=2.0, kd=1.5, c_min=0.05, c_max=50.0, turn=math.pi / 30)


def _sim(kind, name, dim, nx, ny, nz=1, *, steps, cones, sources, stop=0.0, clamp=False, rate_map=False, snr=False,
         clustered=False, start="zeros"):
    c = dict(kind=kind, dim=dim, nx=nx, ny=ny, nz=nz, steps=steps, cones=cones, sources=sources, stop=stop,
             clamp=clamp, rate_map=rate_map, snr=snr, clustered=clustered, start=start)
    return dict(c, name=name) if name else c


def listed():
    return [
        # an interactive viewer or a coupled host model: one step at a time of a small culture
        _sim("step", "step-2d-128", 2, 128, 128, steps=1, cones=64, sources=4, clamp=True),
        # the small configuration: 128^2, 64 cones, a whole run
        _sim("run", "run-2d-128", 2, 128, 128, steps=500, cones=64, sources=4),
        # the SNR steering rule on a middle-sized dish, cones turned back at its walls
        _sim("run", "snr-2d-512x384", 2, 512, 384, steps=500, cones=2000, sources=8, clamp=True, snr=True,
             start="smooth"),
        # a grid of 2^k + 1 nodes per side, as finite-difference users choose them: odd rows
        _sim("run", "run-2d-1025x769", 2, 1025, 769, steps=500, cones=4096, sources=24, stop=1.5),
        # the large 2D configuration, a whole run
        _sim("run", "run-2d-2048", 2, 2048, 2048, steps=5000, cones=16384, sources=64, stop=2.0),
        # the largest 2D grid, beyond the L2 cache
        _sim("run", "run-2d-8192", 2, 8192, 8192, steps=200, cones=16384, sources=64, stop=2.0),
        # the 3D configuration, a whole run
        _sim("run", "run-3d-256", 3, 256, 256, 256, steps=2000, cones=65536, sources=128),
        # a ragged 3D tissue block
        _sim("run", "run-3d-129x97x65", 3, 129, 97, 65, steps=300, cones=5000, sources=16),
        # a parameter sweep: 512 uneven instances
        dict(name="batch-512", kind="batch", instances=512, lo=64, hi=1024, steps=200, sizes=3),
        # fitting the physics: the loss alone, as a line search evaluates it ...
        dict(name="loss-2d-1024", kind="loss", n=1024, cones=4096, sources=32, steps=2000, every=64),
        # ... and the loss with its gradients, as an optimiser's step takes it
        dict(name="grad-2d-1024", kind="grad", n=1024, cones=4096, sources=32, steps=2000, every=64),
        # which neurons the grown cones reach
        dict(name="graph-262144", kind="graph", neurons=262144, per_neuron=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "run2", "run2", "run2", "run2", "run3", "run3", "batch", "loss", "grad", "graph"])
    if kind in ("step", "run2"):
        nx, ny = _log(rng, 64, 4096), _log(rng, 64, 4096)
        if rng.random() < 0.6:
            nx = max(64, nx // 4 * 4)                    # most users round their rows
        # cones in proportion to the grid's area within what the configurations have
        cones = _log(rng, 16, max(64, min(16384, nx * ny // 64)))
        snr = rng.random() < 0.15
        clamp = snr or rng.random() < 0.5
        most = max(20, min(5000, int(2e10 / (nx * ny + 2e5))))
        steps = _log(rng, 1, 16) if kind == "step" else _log(rng, min(64, most), most)
        return _sim("step" if kind == "step" else "run", None, 2, nx, ny, steps=steps, cones=cones,
                    sources=rng.randint(1, 64), stop=0.0 if clamp else rng.choice([0.0, 1.5, 2.0]), clamp=clamp,
                    rate_map=rng.random() < 0.25, snr=snr, clustered=clamp and rng.random() < 0.3,
                    start=rng.choice(["zeros", "smooth"]) if nx * ny < 1 << 20 else "zeros")
    if kind == "run3":
        nx, ny, nz = (_log(rng, 24, 256) for _ in range(3))
        if rng.random() < 0.5:
            nx = max(24, nx // 4 * 4)
        return _sim("run", None, 3, nx, ny, nz, steps=_log(rng, 20, 300), cones=_log(rng, 64, 65536),
                    sources=rng.randint(1, 128), stop=rng.choice([0.0, 2.0]))
    if kind == "batch":
        return dict(kind="batch", instances=rng.randint(4, 128), lo=64, hi=rng.choice([192, 512, 1024]),
                    steps=rng.randint(40, 200), sizes=rng.randint(0, 1 << 20))
    if kind in ("loss", "grad"):
        n = _log(rng, 64, 1024)
        n = n // 4 * 4 if rng.random() < 0.7 else n
        return dict(kind=kind, n=n, cones=_log(rng, 64, 4096), sources=rng.randint(1, 32),
                    steps=rng.randint(50, 600), every=rng.choice([16, 64, 100]))
    return dict(kind="graph", neurons=_log(rng, 2000, 262144), per_neuron=rng.randint(1, 4))


# ------------------------------------------------------------------ inputs
def _workload(c, seed):
    three = c["dim"] == 3
    w = W.make("case", c["dim"], c["nx"], c["ny"], c["nz"], D=1.0, lam=0.01 if three else 0.005,
               dt=0.15 if three else 0.2, n_src=c["sources"], emit=(0.5, 2.0), n_axons=c["cones"],
               stop_radius=c["stop"], wall_mode=1 if c["clamp"] else 0, nsteps=c["steps"], seed=seed,
               src_map="random" if c["rate_map"] else False, C0=None if c["start"] == "zeros" else c["start"])
    if c["clustered"]:                                   # the cones start together, in a square of 48 nodes
        rng = np.random.default_rng(seed + 1)
        side = min(48.0, c["nx"] / 2, c["ny"] / 2)
        centre = np.array([[rng.uniform(side / 2, c["nx"] - 1 - side / 2)],
                           [rng.uniform(side / 2, c["ny"] - 1 - side / 2)]])
        w.pos = (centre + rng.uniform(-side / 2, side / 2, w.pos.shape)).astype(np.float32)
    return w


def _batch_workloads(c, seed):
    """The batched configuration's distributions at the case's count and sides (the sizes are the
    case's own, the inputs the seed's)."""
    rng, sizes = np.random.default_rng(seed), np.random.default_rng(c["sizes"])
    out = []
    for b in range(c["instances"]):
        nx, ny = (int(v) for v in sizes.integers(c["lo"], c["hi"] + 1, 2))
        n_axons = int(sizes.integers(256, 4097))
        D, lam = float(rng.uniform(0.5, 2.0)), float(10.0 ** rng.uniform(-3.0, -1.0))
        out.append(W.make(f"case{b}", 2, nx, ny, D=D, lam=lam, dt=0.2 / D, n_src=int(rng.integers(4, 65)),
                          emit=(0.5, 2.0), n_axons=n_axons, nsteps=c["steps"],
                          seed=int(rng.integers(0, 2**31 - 1)), philox_seed=4 + 16 * b))
    return out


def _endpoint_workload(c, seed):
    return W.config_c5(seed=seed, n=c["n"], n_src=c["sources"], n_axons=c["cones"], nsteps=c["steps"])


def _graph_workload(c, seed):
    # the connectivity workload's density of neurons at the case's count
    extent = 2048.0 * math.sqrt(c["neurons"] / 262144.0)
    return W.config_graph(seed=seed, extent=extent, n_neurons=c["neurons"], cones_per_neuron=c["per_neuron"])


class _State:
    def __init__(self, case):
        self.case = case


def prepare(case, seed):
    s, kind = _State(case), case["kind"]
    if kind in ("step", "run"):
        s.sim = cue.Simulation(_workload(case, seed), device=DEV)
        if case["snr"]:
            s.sim.set_steering(SNR)
        s.start = [t.clone() for t in (s.sim.fields[0], s.sim.pos, s.sim.dir, s.sim.active)]
    elif kind == "batch":
        b = s.batch = B.Batch(_batch_workloads(case, seed), device=DEV)
        b.autotune(16)
        b.set_option(B.CUE_BOPT_GRAPH, 1)
        b.reset_state(0, 0)
        s.now = [f[0] for f in b.fields] + list(b.pos) + list(b.dir)
        s.start = [t.clone() for t in s.now]
        s.active = [t.clone() for t in b.active]
    elif kind in ("loss", "grad"):
        w = _endpoint_workload(case, seed)
        s.problem = A.EndpointProblem(w, w.targets, case["steps"], case["every"], device=DEV)
        grad = kind == "grad"
        s.inputs = [torch.tensor(w.D, device=DEV, requires_grad=grad), torch.tensor(w.lam, device=DEV, requires_grad=grad),
                    torch.as_tensor(w.src_emit, device=DEV).clone().requires_grad_(grad),
                    torch.as_tensor(w.src_map, device=DEV).clone().requires_grad_(grad)]
    else:
        w = s.w = _graph_workload(case, seed)
        s.npos, s.pos = torch.as_tensor(w.npos, device=DEV), torch.as_tensor(w.pos, device=DEV)
        s.owner, s.active = torch.as_tensor(w.owner, device=DEV), torch.as_tensor(w.active, device=DEV)
    return s


def run(s):
    kind = s.case["kind"]
    if kind in ("step", "run"):
        sim = s.sim
        if kind == "run":                                # the run starts from the initial state on the device
            for t, t0 in zip((sim.fields[0], sim.pos, sim.dir, sim.active), s.start):
                t.copy_(t0)
            cue.cue_set_state(sim.h, 0, 0, 0)
        sim.sim_run(s.case["steps"])
        return {"field": sim.field(), "pos": sim.pos, "dir": sim.dir, "active": sim.active}
    if kind == "batch":
        b = s.batch
        with torch.cuda.stream(b.stream):
            torch._foreach_copy_(s.now, s.start)
            torch._foreach_copy_(b.active, s.active)
        b.reset_state(0, 0)
        b.run(s.case["steps"])
        with torch.cuda.stream(b.stream):                # a sweep's results, instances end to end
            cur = b.get_option(B.CUE_BINFO_CUR)
            return {"field": torch.cat([f[cur][:, : w.nx].reshape(-1) for f, w in zip(b.fields, b.w)]),
                    "pos": torch.cat([p.reshape(-1) for p in b.pos]), "dir": torch.cat([d.reshape(-1) for d in b.dir]),
                    "active": torch.cat(b.active)}
    if kind == "loss":
        with torch.no_grad():
            loss = s.problem(*s.inputs)
        sim = s.problem.sim                              # with where it led: the field and the cones at the end
        return {"loss": loss, "field": sim.field(), "pos": sim.pos, "dir": sim.dir}
    if kind == "grad":
        for t in s.inputs:
            t.grad = None
        loss = s.problem(*s.inputs)
        loss.backward()
        return {"loss": loss.detach(), **{k: t.grad for k, t in zip(("D", "lam", "emit", "map"), s.inputs)}}
    w = s.w
    binned = G.bin_points(s.npos, w.cell, w.grid)
    src, dst, count = G.connect(s.pos, s.owner, s.active, s.npos, w.radius, w.cell, w.grid, binned, cap=4 * w.n_cones)
    row, col, m = G.csr(w.n_neurons, src, dst, count)
    level = G.bfs(row, col, w.source)
    col[int(m) :] = -1                                   # an array of one size whatever was connected
    return {"count": count, "sorted": binned[1], "row": row, "col": col, "level": level}


def work(case):
    """A grid is read once and written once per pass when it fits the card's on-chip memories
    (up to 2^25 nodes), else once per 16 steps, the deepest blocking the framework takes; a node
    update is 7 operations in 2D and 9 in 3D, a cone step about 150."""
    kind = case["kind"]
    if kind in ("step", "run"):
        nodes = case["nx"] * case["ny"] * case["nz"]
        passes = 1 if nodes <= 1 << 25 else -(-case["steps"] // 16)
        cones = case["cones"]
        per_cone = 8 * case["dim"] + 1
        return {"bytes": passes * (8 * nodes + 2 * per_cone * cones) + (4 * nodes if case["rate_map"] else 0) + 8 * case["sources"],
                "flops": float(case["steps"]) * ((7 if case["dim"] == 2 else 9) * nodes + 150 * cones)}
    if kind == "batch":
        side = 0.5 * (case["lo"] + case["hi"])
        nodes, cones = case["instances"] * side * side, case["instances"] * 2176
        return {"bytes": -(-case["steps"] // 16) * (8 * nodes + 34 * cones), "flops": case["steps"] * (7 * nodes + 150 * cones)}
    if kind in ("loss", "grad"):
        nodes, cones, n = case["n"] ** 2, case["cones"], case["steps"]
        if kind == "loss":
            return {"bytes": 16 * nodes + 17 * cones, "flops": n * (9 * nodes + 150 * cones)}
        # forward and backward: the parameters' products read the field of every step, kept or recomputed
        return {"bytes": 8 * nodes * n, "flops": n * (30 * nodes + 600 * cones)}
    n, e = case["neurons"], case["neurons"] * case["per_neuron"]
    return {"bytes": 8 * n + 4 * n + 13 * e + 8 * n + 12 * e, "flops": 40.0 * e}


# ------------------------------------------------------------------ the model in 64 bits
def _mulhi(a, c):
    """High and low words of a 32-bit constant times a 32-bit word, in int64 tensors."""
    lo16, hi16 = c & 0xFFFF, c >> 16
    t = a * lo16
    u = a * hi16 + (t >> 16)
    return u >> 16, ((u & 0xFFFF) << 16) | (t & 0xFFFF)


def _noise(seed, ids, step, comps):
    """Philox-4x32-10 (key: the seed's words, counter: cone, step, 0, 0), then Box-Muller."""
    c = [ids.clone(), torch.full_like(ids, step), torch.zeros_like(ids), torch.zeros_like(ids)]
    k0, k1 = seed & 0xFFFFFFFF, seed >> 32
    for _ in range(10):
        ha, la = _mulhi(c[0], 0xD2511F53)
        hb, lb = _mulhi(c[2], 0xCD9E8D57)
        c = [hb ^ c[1] ^ k0, lb, ha ^ c[3] ^ k1, la]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    u = [(c[0] >> 8).double().add(1.0) * 2.0**-24, (c[1] >> 8).double() * 2.0**-24]
    r = torch.sqrt(-2.0 * torch.log(u[0]))
    xi = [r * torch.cos(2 * math.pi * u[1]), r * torch.sin(2 * math.pi * u[1])]
    if comps == 3:
        u = [(c[2] >> 8).double().add(1.0) * 2.0**-24, (c[3] >> 8).double() * 2.0**-24]
        xi.append(torch.sqrt(-2.0 * torch.log(u[0])) * torch.cos(2 * math.pi * u[1]))
    return torch.stack(xi)


class _Exact:
    """One grid, or several 2D grids stacked with their instance as the slowest axis."""

    def __init__(self, ws, snr=None):
        f32 = lambda v: float(np.float32(v))             # the entry points take their parameters in 32 bits
        w0, self.snr = ws[0], snr
        self.dim, self.n = w0.dim, len(ws)
        ext = [[w.nx, w.ny, w.nz][: w0.dim] for w in ws]
        self.full = [max(e[a] for e in ext) for a in range(w0.dim)]
        t = lambda v, d=torch.float64: torch.as_tensor(np.asarray(v), dtype=d, device=DEV)
        one = [1] * w0.dim
        col = lambda v: t([f32(x) for x in v]).reshape([-1] + one)
        self.D, self.lam, self.dt = (col([getattr(w, k) for w in ws]) for k in ("D", "lam", "dt"))
        self.h = f32(w0.h)
        # between neighbours i and i + 1 of an axis there is flux where both are in the grid
        self.inside = []
        for a in range(w0.dim):
            m = torch.arange(1, self.full[a], device=DEV)[None] < t([e[a] for e in ext], torch.int64)[:, None]
            self.inside.append(m.double().reshape([self.n] + [-1 if k == w0.dim - 1 - a else 1 for k in range(w0.dim)]))
        shape = [self.n] + self.full[::-1]
        self.C = torch.zeros(shape, dtype=torch.float64, device=DEV)
        self.map = torch.zeros(shape, dtype=torch.float64, device=DEV) if w0.src_map is not None else None
        where, emit, src = [], [], []
        for i, w in enumerate(ws):
            sl = (i,) + tuple(slice(0, e) for e in ext[i][::-1])
            if w.C0 is not None:
                self.C[sl] = t(w.C0)
            if self.map is not None:
                self.map[sl] = t(w.src_map)
            cell = t(w.src_cell, torch.int64)
            xyz = [cell % w.nx, (cell // w.nx) % w.ny, cell // (w.nx * w.ny)][: self.dim]
            where.append(self._flat(torch.full_like(cell, i), xyz))
            emit.append(t(w.src_emit))
            src.append(torch.stack(xyz).double() * self.h)
        self.where, self.emit, self.src = torch.cat(where), torch.cat(emit), src
        self.count = [w.n_axons for w in ws]
        self.of = torch.repeat_interleave(torch.arange(self.n, device=DEV), t(self.count, torch.int64))
        self.ids = torch.cat([torch.arange(k, device=DEV) for k in self.count])
        self.seeds = [int(w.seed) for w in ws]
        self.pos, self.dir = (torch.cat([t(getattr(w, k)) for w in ws], 1) for k in ("pos", "dir"))
        self.active = torch.cat([t(w.active, torch.bool) for w in ws])
        self.ext = t(ext, torch.int64)[self.of].T.contiguous()      # extents at each cone
        self.par = {k: f32(getattr(w0, k)) for k in ("w_prev", "w_grad", "w_noise", "step_len", "stop_radius", "grad_eps")}
        self.clamp = w0.wall_mode == 1

    def _flat(self, i, xyz):
        f = i
        for a in range(self.dim - 1, -1, -1):
            f = f * self.full[a] + xyz[a]
        return f

    def field_step(self):
        C = self.C
        lap = torch.zeros_like(C)
        for a in range(self.dim):
            ax = C.dim() - 1 - a
            d = (C.narrow(ax, 1, C.shape[ax] - 1) - C.narrow(ax, 0, C.shape[ax] - 1)) * self.inside[a]
            pad = [0, 0] * a
            lap = lap + torch.nn.functional.pad(d, pad + [0, 1]) - torch.nn.functional.pad(d, pad + [1, 0])
        C = C + (self.D * self.dt / self.h**2) * lap - self.lam * self.dt * C
        C = C.reshape(-1).index_add(0, self.where, self.emit).reshape(C.shape)
        self.C = C if self.map is None else C + self.dt * self.map

    def _sense(self, p):
        """Cue value and gradient at p: multilinear over the cell's nodes and their central differences."""
        s = p / self.h
        lo = torch.minimum(torch.clamp(torch.floor(s.detach()), min=0).long(), self.ext - 2)
        fr = s - lo
        flat, top = self.C.reshape(-1), self.ext - 1
        at = lambda xyz: flat[self._flat(self.of, xyz)]
        val, g = 0.0, [0.0] * self.dim
        for corner in range(1 << self.dim):
            bit = [(corner >> a) & 1 for a in range(self.dim)]
            w, node = 1.0, [lo[a] + bit[a] for a in range(self.dim)]
            for a in range(self.dim):
                w = w * (fr[a] if bit[a] else 1.0 - fr[a])
            if self.snr:
                val = val + w * at(node)
            for a in range(self.dim):
                hi, low = list(node), list(node)
                hi[a], low[a] = torch.minimum(node[a] + 1, top[a]), torch.clamp(node[a] - 1, min=0)
                g[a] = g[a] + w * (at(hi) - at(low)) / (2.0 * self.h)
        return val, torch.stack(g)

    def _xi(self, step):
        xi, k = [], 0
        for seed, n in zip(self.seeds, self.count):
            if k and seed == self.seeds[0] and len(set(self.seeds)) == 1:
                break
            xi.append(_noise(seed, self.ids[k : k + n], step, self.dim))
            k += n
        return torch.cat(xi, 1)

    def cone_step(self, step):
        q, p, d = self.par, self.pos, self.dir
        val, g = self._sense(p)
        xi = self._xi(step)
        if self.snr:
            s = self.snr
            gn = g.norm(dim=0)
            gamma = val / s["kd"]
            ok = (gn > 0) & (val > 0)
            safe_v, safe_g = torch.where(ok, val, 1.0), torch.where(ok, gn, 1.0)
            ratio = s["gain"] * s["width"] * gn / safe_v * torch.sqrt(torch.clamp(gamma, min=0) / (1 + gamma) ** 3)
            ratio = torch.where(ok, ratio * (d[1] * g[0] - d[0] * g[1]) / safe_g, 0.0)
            sn = torch.where(ratio + xi[0] > 0, -math.sin(s["turn"]), math.sin(s["turn"]))
            cs = math.cos(s["turn"])
            turned = torch.stack([d[0] * cs - d[1] * sn, d[0] * sn + d[1] * cs])
            turned = turned / turned.norm(dim=0)
            dn = torch.where((val >= s["c_min"]) & (val <= s["c_max"]), turned, d)
        else:
            g2 = (g * g).sum(0)
            some = g2 > q["grad_eps"] ** 2
            unit = torch.where(some, g * torch.where(some, g2, 1.0).rsqrt(), 0.0)
            v = q["w_prev"] * d + q["w_grad"] * unit + q["w_noise"] * xi
            v2 = (v * v).sum(0)
            dn = torch.where(v2 > 1e-30, v * torch.where(v2 > 1e-30, v2, 1.0).rsqrt(), d)
        pn = p + q["step_len"] * dn
        hi = (self.ext - 1).double() * self.h
        out = ((pn < 0) | (pn > hi)).any(0)
        pn = torch.minimum(torch.clamp(pn, min=0.0), hi)
        move = self.active if self.clamp else self.active & ~out
        stop = torch.zeros_like(move)
        if q["stop_radius"] > 0:
            k = 0
            for i, n in enumerate(self.count):
                for s in range(self.src[i].shape[1]):
                    e = pn[:, k : k + n] - self.src[i][:, s : s + 1]
                    stop[k : k + n] |= (e * e).sum(0) <= q["stop_radius"] ** 2
                k += n
        self.pos, self.dir = torch.where(move, pn, p), torch.where(move, dn, d)
        self.active = move & ~stop


def exact(case, seed):
    kind = case["kind"]
    if kind in ("step", "run"):
        w = _workload(case, seed)
        # a cone's path amplifies rounding: past some hundred steps its state has no exact value to
        # compare with (a cone that circles a source, a turn that noise decides); the field does
        # not read the cones and has one at any length
        cones = case["steps"] <= 16 and not case["snr"]
        e = _Exact([w], SNR if case["snr"] else None)
        for n in range(case["steps"]):
            if cones:
                e.cone_step(n)
            e.field_step()
        return {"field": e.C[0].clone(), "pos": e.pos if cones else None, "dir": e.dir if cones else None, "active": None}
    if kind == "batch":
        ws = _batch_workloads(case, seed)
        e = _Exact(ws)
        for n in range(case["steps"]):
            e.field_step()
        return {"field": torch.cat([e.C[i, : w.ny, : w.nx].reshape(-1) for i, w in enumerate(ws)]), "pos": None,
                "dir": None, "active": None}
    if kind == "grad":
        if case["steps"] > 100 or case["n"] > 512:       # longer paths: their derivative amplifies rounding without bound
            return None
        w = _endpoint_workload(case, seed)
        e = _Exact([w])
        leaves = [e.D.requires_grad_(True), e.lam.requires_grad_(True), e.emit.requires_grad_(True), e.map.requires_grad_(True)]
        for n in range(case["steps"]):
            e.cone_step(n)
            e.field_step()
        t = torch.as_tensor(w.targets, dtype=torch.float64, device=DEV)
        loss = ((e.pos - t) ** 2).sum() / w.n_axons
        gD, gl, ge, gm = torch.autograd.grad(loss, leaves)
        return {"loss": loss.detach(), "D": gD.reshape(()), "lam": gl.reshape(()), "emit": ge, "map": gm[0]}
    if kind == "loss":
        w = _endpoint_workload(case, seed)
        e = _Exact([w])
        cones = case["steps"] <= 100
        for n in range(case["steps"]):
            if cones:
                e.cone_step(n)
            e.field_step()
        t = torch.as_tensor(w.targets, dtype=torch.float64, device=DEV)
        return {"loss": ((e.pos - t) ** 2).sum() / w.n_axons if cones else None, "field": e.C[0], "pos": None, "dir": None}
    return None                                          # the connectivity stage's outputs are whole numbers
