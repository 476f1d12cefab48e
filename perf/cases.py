"""The work whose speed counts: calls of the public API (AmrLBM, AmrBatch, Mlp)
over the sizes, storages and options the workloads of this repository use.

listed() names the cases, draw() gives more of the same ranges, prepare() makes
what a user's program has in hand before the call, run() is one pass, work()
the bytes and operations of a pass that no implementation can do without, and
exact() the results of a pass in FP64 from a plain torch statement of the
method (no code of the package).

The meshes are built from geometric marks (distance to walls, prism, outlet or
a plane), so that they are the same for every seed and every rounding; the
seed draws the flow fields, the marks of the adaptation pass and the samples.
"""
import functools
import itertools
import math

import numpy as np
import torch

import workloads as W

DTYPE = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
BYTES = {"f64": 8, "f32": 4, "bf16": 2, "f16": 2}


def forest(name, flow, q, storage, nx, ny, nz, levels, width, steps, interp="linear", kind="step"):
    c = dict(kind=kind, flow=flow, q=q, storage=storage, nx=nx, ny=ny, nz=nz, levels=levels,
             width=width, steps=steps, interp=interp)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the 2D FP64 cavity (64x64 root cells, two extra levels): a few hundred
        # small blocks, where launches and latency count
        forest("cavity2d_f64", "cavity", 9, "f64", 64, 64, 4, 3, 8.0, 20),
        # the 2D channel past a square prism, FP64: 16 coarse steps, then the force
        forest("square2d_f64", "prism", 9, "f64", 256, 256, 4, 3, 12.0, 16),
        # the 2D FP32 cavity of the paper's MLUPS table (128x128 root cells, L_max 4)
        forest("cavity2d_f32", "cavity", 9, "f32", 128, 128, 4, 4, 16.0, 20),
        # the 3D FP32 cavity of the benchmark: 64^3 root cells, three extra levels
        forest("cavity3d_f32", "cavity", 19, "f32", 64, 64, 64, 4, 8.0, 10),
        # the same method in FP64, as comparison and oracle runs take it
        forest("cavity3d_f64", "cavity", 19, "f64", 48, 48, 48, 3, 8.0, 4),
        # the single-level periodic forest the roofline is stated on
        forest("box3d_f32", "box", 19, "f32", 256, 256, 256, 1, 0.0, 30),
        # the channel past a prism, D3Q27, 16-bit shifted storage
        forest("prism3d_f16", "prism", 27, "f16", 128, 32, 32, 4, 19.2, 5),
        # the same channel in FP32 with the cubic coarse-to-fine interpolation
        forest("prism3d_f32_cubic", "prism", 27, "f32", 128, 32, 32, 4, 19.2, 5, "cubic"),
        # one adaptation of a refined 3D cavity: refine marked leaves, read the
        # tables and populations, coarsen them again
        forest("adapt3d_f32", "cavity", 19, "f32", 64, 64, 64, 4, 8.0, 0, kind="adapt"),
        # independent cavities of uneven sizes and depths advanced together
        dict(name="batch_f32", kind="batch", members=12, small=32, large=56, levels=3,
             form="members", steps=5),
        # block summaries, MLP inference and criterion of the learned proposal
        forest("propose3d_f32", "cavity", 19, "f32", 64, 64, 64, 3, 12.0, 0, kind="propose"),
        # one training epoch of the proposal network and its check on held-out samples
        dict(name="train_mlp", kind="train", samples=32768, batch=1024, held_out=8192),
    ]


def draw(rng):
    def pick(lo, hi):          # a multiple of 4, spread over the logarithm
        return 4 * max(1, round(math.exp(rng.uniform(math.log(lo / 4), math.log(hi / 4)))))

    kind = rng.choice(["flat", "flat", "solid", "solid", "prism", "adapt", "batch", "propose", "train"])
    width = round(rng.uniform(5.0, 10.0), 2)
    if kind == "flat":         # 2D forests
        flow = rng.choice(["cavity", "box", "prism"])
        interp = rng.choice(["linear", "linear", "cubic"])
        return forest(None, flow, 9, rng.choice(["f64", "f32"]), pick(64, 384), pick(64, 384), 4,
                      rng.randint(1, 4), width, rng.randint(8, 20), interp)
    if kind == "solid":        # 3D cavities and periodic boxes
        return forest(None, rng.choice(["cavity", "box"]), rng.choice([19, 19, 27]),
                      rng.choice(["f32", "f32", "f64", "bf16", "f16"]), pick(24, 64), pick(24, 64),
                      pick(24, 64), rng.randint(1, 3), width, rng.randint(2, 6),
                      rng.choice(["linear", "linear", "cubic"]))
    if kind == "prism":
        return forest(None, "prism", 27, rng.choice(["f32", "bf16", "f16"]), pick(64, 128),
                      pick(24, 40), pick(8, 32), rng.randint(2, 4), width, rng.randint(2, 5),
                      rng.choice(["linear", "cubic"]))
    if kind in ("adapt", "propose"):
        q, storage = rng.choice([19, 27]), rng.choice(["f32", "f32", "f64"])
        return forest(None, "cavity", q, storage, pick(24, 64), pick(24, 64), pick(24, 64),
                      rng.randint(2, 3), width, 0, kind=kind)
    if kind == "batch":
        return dict(kind="batch", members=rng.randint(3, 16), small=24, large=pick(32, 52),
                    levels=rng.randint(1, 3), form=rng.choice(["members", "graph", "persistent"]),
                    steps=rng.randint(2, 6))
    return dict(kind="train", samples=int(math.exp(rng.uniform(math.log(2000), math.log(40000)))),
                batch=rng.choice([256, 500, 1024, 2048]), held_out=rng.randint(100, 8192))


# ------------------------------------------------------------ configuration
def dim_of(case):
    return 2 if case["q"] == 9 else 3


def prism_box(case):
    """(x0, x1, y0, y1) of the prism: edges on root-cell faces."""
    side = 2 * max(1, round(min(case["nx"] / 64, case["ny"] / 8)))
    cx, cy = case["nx"] // 4, case["ny"] // 2
    return cx - side // 2, cx + side // 2, cy - side // 2, cy + side // 2


@functools.lru_cache(maxsize=4)
def plan_of(items):
    return Plan(dict(items))


def plan(case):
    return plan_of(tuple(sorted((k, v) for k, v in case.items() if k != "name")))


class Plan:
    """The forest of a case: per level the block positions (block units of the
    level) and IDs in ID order, and the ID of each block's first child."""

    def __init__(self, case):
        self.case, self.dim = case, dim_of(case)
        d = self.dim
        self.root = np.array([case["nx"] // 4, case["ny"] // 4, case["nz"] // 4][:d])
        self.periodic = [case["flow"] == "box"] * d
        self.nc = 2 ** d
        self.child_off = np.array([[(c >> a) & 1 for a in range(d)] for c in range(self.nc)])
        pos = np.stack(np.meshgrid(*[np.arange(n) for n in self.root[::-1]], indexing="ij"), -1)
        pos = pos.reshape(-1, d)[:, ::-1]
        self.levels = [dict(pos=pos, ids=np.arange(len(pos)), head=np.full(len(pos), -1))]
        self.next_id = len(pos)
        for lv in range(case["levels"] - 1):
            self.refine(lv, self.wanted(lv) & self.eligible(lv))
        self.blocks = self.next_id

    def grid(self, lv, values):
        g = np.full(tuple(self.root * 2 ** lv), -1, np.int64)
        g[tuple(self.levels[lv]["pos"].T)] = values
        return g

    def neighbours(self, lv, e):
        """Index within the level of the neighbour in direction e (-1: none at
        this level, -2: outside the domain)."""
        t = self.levels[lv]
        n = self.root * 2 ** lv
        q = t["pos"] + np.asarray(e)
        out = np.zeros(len(q), bool)
        for a in range(self.dim):
            if self.periodic[a]:
                q[:, a] %= n[a]
            else:
                out |= (q[:, a] < 0) | (q[:, a] >= n[a])
        g = self.grid(lv, np.arange(len(q)))
        return np.where(out, -2, g[tuple(np.clip(q, 0, n - 1).T)])

    def eligible(self, lv):
        ok = self.levels[lv]["head"] < 0
        for e in itertools.product((-1, 0, 1), repeat=self.dim):
            ok &= self.neighbours(lv, e) != -1
        return ok

    def wanted(self, lv):
        """Blocks within width / 2^level of the lid and the x walls (cavity),
        the middle plane (box), the prism and the outlet (prism)."""
        c, h = self.case, 4.0 / 2 ** lv
        x = (self.levels[lv]["pos"] + 0.5) * h
        ext, reach = self.root * 4.0, self.case["width"] / 2 ** lv
        if c["flow"] == "box":
            return np.abs(x[:, -1] - ext[-1] / 2) < reach
        if c["flow"] == "cavity":
            return (x[:, 0] < reach) | (ext[0] - x[:, 0] < reach) | (ext[-1] - x[:, -1] < reach)
        x0, x1, y0, y1 = prism_box(c)
        dx = np.maximum(np.maximum(x0 - x[:, 0], x[:, 0] - x1), 0)
        dy = np.maximum(np.maximum(y0 - x[:, 1], x[:, 1] - y1), 0)
        return (dx * dx + dy * dy < reach * reach) | (ext[0] - x[:, 0] < reach)

    def refine(self, lv, mask):
        """Children of the blocks in mask: groups of IDs in ascending ID order."""
        t = self.levels[lv]
        which = np.nonzero(mask)[0]
        head = self.next_id + self.nc * np.arange(len(which))
        t["head"] = t["head"].copy()
        t["head"][which] = head
        self.next_id += self.nc * len(which)
        t.setdefault("marks", []).append(t["ids"][which])
        pos = (2 * t["pos"][which][:, None, :] + self.child_off).reshape(-1, self.dim)
        ids = (head[:, None] + np.arange(self.nc)).reshape(-1)
        if lv + 1 == len(self.levels):
            self.levels.append(dict(pos=np.zeros((0, self.dim), np.int64), ids=np.zeros(0, np.int64),
                                    head=np.zeros(0, np.int64)))
        u = self.levels[lv + 1]
        u["pos"] = np.concatenate([u["pos"], pos])
        u["ids"] = np.concatenate([u["ids"], ids])
        u["head"] = np.concatenate([u["head"], np.full(len(ids), -1)])

    def copy(self):
        p = Plan.__new__(Plan)
        p.__dict__.update(self.__dict__)
        p.levels = [dict(t, marks=list(t.get("marks", []))) for t in self.levels]
        return p


def config(case):
    """Workload dictionary of a forest case."""
    p = plan(case)
    d = p.dim
    room = p.blocks + 64 * p.nc
    if case["kind"] == "adapt":
        room += p.nc * len(p.levels[case["levels"] - 2]["ids"]) if case["levels"] > 1 else 0
    kw = dict(max_levels=max(1, case["levels"]), max_blocks=room)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    if case["flow"] == "box":
        cfg = W.periodic_box(dim=d, q=case["q"], n=nx, ny=ny, nz=nz, nu0=0.01, **kw)
    elif case["flow"] == "cavity":
        # Re 100 in 2D; in 3D Re 1000 at 64 root cells and the same viscosity
        # at other sizes (BGK needs it to stay stable)
        re = 100.0 if d == 2 else 1000.0 * nx / 64
        cfg = W.cavity(dim=d, q=case["q"], n=nx, ny=ny, nz=nz, re=re, **kw)
    else:
        x0, x1, y0, y1 = prism_box(case)
        cfg = W.channel_cylinder(q=case["q"], nx=nx, ny=ny, nz=nz, side=x1 - x0, cx=(x0 + x1) / 2,
                                 cy=(y0 + y1) / 2, dim=d, refine_dist=0.0,
                                 re=min(100.0, 25.0 * (x1 - x0)), **kw)
    cfg["interp"] = case["interp"]
    return cfg


def members_of(case):
    """The forest cases of a batch: uneven sizes and depths, fixed by the case."""
    g = np.random.default_rng(case["members"] + 100 * case["large"])
    out = []
    for _ in range(case["members"]):
        n = 4 * int(g.integers(case["small"] // 4, case["large"] // 4 + 1))
        out.append(forest(None, "cavity", 19, "f32", n, n, n, int(g.integers(1, case["levels"] + 1)),
                          8.0, case["steps"]))
    return out


# ------------------------------------------------------------------- inputs
def velocities(q):
    e = [(0, 0, 0)]
    if q == 9:
        e += [(1, 0, 0), (0, 1, 0), (-1, 0, 0), (0, -1, 0), (1, 1, 0), (-1, 1, 0), (-1, -1, 0), (1, -1, 0)]
    else:
        for a, b, c in [(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, 0, 1), (0, 1, 1), (1, -1, 0),
                        (1, 0, -1), (0, 1, -1)] + \
                ([(1, 1, 1), (1, 1, -1), (1, -1, 1), (-1, 1, 1)] if q == 27 else []):
            e += [(a, b, c), (-a, -b, -c)]
    shell = {9: [4 / 9, 1 / 9, 1 / 36], 19: [1 / 3, 1 / 18, 1 / 36],
             27: [8 / 27, 2 / 27, 1 / 54, 1 / 216]}[q]
    return e, [shell[sum(v * v for v in c)] for c in e]


def moments(f, q):
    e, _ = velocities(q)
    rho = f.sum(0)
    u = [sum(c[a] * f[p] for p, c in enumerate(e) if c[a]) / rho for a in range(2 if q == 9 else 3)]
    return rho, u


def equilibrium(rho, u, q):
    e, w = velocities(q)
    us = 1.5 * sum(v * v for v in u)
    out = torch.empty((q,) + rho.shape, dtype=rho.dtype, device=rho.device)
    for p in range(q):
        cu = sum(e[p][a] * u[a] for a in range(len(u)) if e[p][a]) if any(e[p]) else torch.zeros_like(rho)
        out[p] = w[p] * rho * (1 + 3 * cu + 4.5 * cu * cu - us)
    return out


def cell_offsets(d):
    n = 4 ** d
    return np.stack([(np.arange(n) >> (2 * a)) & 3 for a in range(d)], -1)


def start_field(case, seed, dev, p):
    """Populations [q][blocks of the plan][cells] in FP64, rounded to what the
    storage holds: the equilibrium of a smooth seeded flow (a few Fourier modes
    about the free stream), |u| <= 0.08, rho within 1 %."""
    d, q = p.dim, case["q"]
    g = np.random.default_rng(seed)
    ext = p.root * 4.0
    # one set of modes per field, drawn before any level is filled
    modes = [[(2 * math.pi * g.integers(1, 4, d) / ext, g.uniform(0, 2 * math.pi), g.uniform(0.3, 1.0))
              for _ in range(4)] for _ in range(d + 1)]
    f = torch.zeros((q, p.next_id, 4 ** d), dtype=torch.float64, device=dev)
    for lv, t in enumerate(p.levels):
        if not len(t["ids"]):
            continue
        x = torch.from_numpy((t["pos"][:, None, :] * 4 + cell_offsets(d) + 0.5) / 2.0 ** lv).to(dev)
        field = [sum(a * torch.sin(sum(float(k[i]) * x[..., i] for i in range(d)) + ph)
                     for k, ph, a in ms) / 4 for ms in modes]
        u = [0.03 * v for v in field[1:]]
        if case["flow"] == "prism":
            u[0] = u[0] + 0.05
        e = equilibrium(1 + 0.01 * field[0], u, q)
        if case["flow"] == "prism":        # solid cells are at rest
            x0, x1, y0, y1 = prism_box(case)
            solid = (x[..., 0] > x0) & (x[..., 0] < x1) & (x[..., 1] > y0) & (x[..., 1] < y1)
            rest = torch.tensor(velocities(q)[1], dtype=torch.float64, device=dev).view(-1, 1, 1)
            e = torch.where(solid, rest, e)
        f[:, torch.from_numpy(t["ids"]).to(dev)] = e
    if case["storage"] in ("f64", "f32"):
        return f.to(DTYPE[case["storage"]]).double()
    w = torch.tensor(velocities(q)[1], dtype=torch.float64, device=dev).view(-1, 1, 1)
    return (f - w).to(DTYPE[case["storage"]]).double() + w


def make_forest(case, seed):
    from paper_2308_08085_gb300 import amr
    cfg, p = config(case), plan(case)
    sim = amr.AmrLBM(cfg, storage=case["storage"])
    for lv in range(len(p.levels) - 1):
        for ids in p.levels[lv].get("marks", []):
            marks = torch.zeros(sim.cap, dtype=torch.int8, device=sim.device)
            marks[torch.from_numpy(ids).to(sim.device)] = 1
            sim.adapt(marks)
    f = torch.zeros((case["q"], sim.cap, sim.m), dtype=torch.float64, device=sim.device)
    f[:, :p.next_id] = start_field(case, seed, sim.device, p)
    rc = sim.lib.amr_set_fields(sim.h, amr.AMR_F, f.data_ptr(), f.numel() * 8, 1)
    if rc != amr.AMR_OK:
        raise amr.AmrError(rc, "amr_set_fields")
    return sim


def adapt_marks(case, seed):
    """A seeded tenth of the refinable leaves of the second-finest level."""
    p = plan(case)
    lv = case["levels"] - 2
    can = p.eligible(lv)
    return lv, can & (np.random.default_rng(seed).random(len(can)) < 0.1)


def train_inputs(case, seed, dev):
    """(samples, labels, weights): 27 summaries of unit scale, a rule with noise
    for the labels, Glorot-sized weights."""
    g = torch.Generator(device=dev).manual_seed(int(seed))
    n = case["samples"] + case["held_out"]
    x = torch.randn(n, 27, generator=g, device=dev)
    rule = torch.randn(27, generator=g, device=dev)
    y = ((x @ rule + 2 * torch.randn(n, generator=g, device=dev)) > 6).float()
    shapes = [(64, 27), (64,), (64, 64), (64,), (64,), (1,)]
    w = [torch.rand(s, generator=g, device=dev) * 2 - 1 for s in shapes]
    scale = [math.sqrt(6 / 91), 0.1, math.sqrt(6 / 128), 0.1, math.sqrt(6 / 65), 0.1]
    return x, y, torch.cat([(v * s).reshape(-1) for v, s in zip(w, scale)])


def prepare(case, seed):
    from paper_2308_08085_gb300 import amr
    dev = torch.device("cuda", torch.cuda.current_device())
    s = dict(case=case, amr=amr)
    if case["kind"] == "train":
        x, y, w = train_inputs(case, seed, dev)
        n = case["samples"]
        s.update(mlp=amr.Mlp(dev), x=x[:n].contiguous(), y=y[:n].contiguous(), held=x[n:].contiguous())
        s["mlp"].params.copy_(w)
        return s
    if case["kind"] == "batch":
        s["members"] = [make_forest(c, seed + 1000 * i) for i, c in enumerate(members_of(case))]
        s["batch"] = amr.AmrBatch(s["members"])
        if case["form"] == "persistent":
            s["batch"].configure("persistent", threads=128, tile_blocks=8)
        else:
            s["batch"].configure(case["form"], threads=64)
        return s
    s["sim"] = make_forest(case, seed)
    if case["kind"] == "adapt":
        lv, mask = adapt_marks(case, seed)
        ids = torch.from_numpy(plan(case).levels[lv]["ids"][mask]).to(dev)
        s["plus"] = torch.zeros(s["sim"].cap, dtype=torch.int8, device=dev)
        s["plus"][ids] = 1
        s["minus"] = -s["plus"]
    if case["kind"] == "propose":
        s["mlp"] = amr.Mlp(dev, seed=seed)
    return s


# --------------------------------------------------------------------- pass
def state_of(sim, amr):
    """The advanced state as a program reads it: density and velocity (after
    the level synchronisation) and the populations, in the storage's type."""
    t = DTYPE[sim.storage]
    return dict(rho_u=sim.fields_device(amr.AMR_RHO_U, torch.float64).to(t),
                f=sim.fields_device(amr.AMR_F, torch.float64).to(t))


def run(s):
    case, amr = s["case"], s["amr"]
    if case["kind"] == "train":
        m = s["mlp"]
        loss = m.train_epoch(s["x"], s["y"], batch=case["batch"], lr=2e-3, pos_weight=4.0, seed=3)
        return dict(loss=np.float32(loss), params=m.params, adam_m=m.m, adam_v=m.v, half=m.half,
                    prob=m.infer(s["held"]))
    if case["kind"] == "batch":
        s["batch"].step(case["steps"])
        return [state_of(m, amr) for m in s["members"]]
    sim = s["sim"]
    if case["kind"] == "propose":
        # the marks first: features() reads the same synchronised state
        return dict(marks=sim.propose_marks(s["mlp"].half, 0.5), features=sim.features())
    if case["kind"] == "adapt":
        sim.adapt(s["plus"])
        out = dict(blocks=sim.fields_device(amr.AMR_BLOCKS, torch.int32),
                   nbr=sim.fields_device(amr.AMR_NBR, torch.int32),
                   f=sim.fields_device(amr.AMR_F, torch.float64).to(DTYPE[case["storage"]]))
        sim.adapt(s["minus"])
        return out
    sim.step(case["steps"])
    out = state_of(sim, amr)
    if case["flow"] == "prism":
        out["force"] = torch.from_numpy(sim.force()).to(DTYPE[case["storage"]])
    return out


# --------------------------------------------------------------------- work
def work(case):
    if case["kind"] == "train":
        n, m = case["samples"], case["held_out"]
        layer = 27 * 64 + 64 * 64 + 64
        steps = -(-n // case["batch"])
        return dict(bytes=4.0 * (n * 28 + m * 28) + 4.0 * 6017 * 8 * steps,
                    flops=2.0 * layer * (3 * n + m))
    if case["kind"] == "batch":
        parts = [work(c) for c in members_of(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    p = plan(case)
    if case["kind"] == "adapt":
        lv, mask = adapt_marks(case, 0)
        p = p.copy()
        p.refine(lv, mask)
    d, q, size = p.dim, case["q"], BYTES[case["storage"]]
    m = 4 ** d
    blocks, leaves = p.next_id, 0.0
    for lv, t in enumerate(p.levels):
        leaves += 2.0 ** lv * m * np.count_nonzero(t["head"] < 0)
    out = blocks * m * (q + 1 + d) * size                # the results
    if case["kind"] == "propose":
        return dict(bytes=float(blocks * (m * q * size + 27 * 4 + 1)),
                    flops=float(blocks * (m * 120 + 2 * (27 * 64 + 64 * 64 + 64))))
    if case["kind"] == "adapt":
        # read and write the tables and the populations of the children that
        # come and go, read the state once, write the results
        return dict(bytes=float(blocks * (m * q * size * 2 + 2 * 148)), flops=float(blocks * m * 120))
    return dict(bytes=float(case["steps"] * leaves * 2 * q * size + out),
                flops=float((case["steps"] * leaves + blocks * m) * 10 * q))


# ------------------------------------------------------- the method in FP64
class Exact:
    """The method on a plan's forest in FP64: f[level] is [q, blocks * cells],
    the pre-collision populations."""

    def __init__(self, case, seed, dev):
        self.case, self.p, self.dev = case, plan(case).copy(), dev
        self.q, self.d = case["q"], self.p.dim
        self.m, self.nc = 4 ** self.d, 2 ** self.d
        self.cfg = config(case)
        self.e, self.w = velocities(self.q)
        self.opp = [self.e.index(tuple(-v for v in c)) for c in self.e]
        f = start_field(case, seed, dev, self.p)
        self.f = [f[:, torch.from_numpy(t["ids"]).to(dev)].reshape(self.q, -1) for t in self.p.levels]
        self.tau = [0.5 + 2.0 ** lv * 3.0 * self.cfg["nu0"] for lv in range(len(self.p.levels) + 1)]
        self.link()

    def link(self):
        p, d, dev = self.p, self.d, self.dev
        off = cell_offsets(d)
        faces, rank = self.cfg["faces"], {"noslip": 1, "moving": 2, "outlet": 3, "periodic": 0}
        self.solid, self.src, self.face, self.cls, self.par = [], [], [], [], []
        for lv, t in enumerate(p.levels):
            cells = (t["pos"][:, None, :] * 4 + off).reshape(-1, d)
            solid = np.zeros(len(cells), bool)
            if self.cfg.get("solid") is not None:
                x = (cells + 0.5) / 2.0 ** lv
                x0, x1, y0, y1 = self.cfg["solid"]
                solid = (x[:, 0] > x0) & (x[:, 0] < x1) & (x[:, 1] > y0) & (x[:, 1] < y1)
            self.solid.append(torch.from_numpy(solid).to(dev))
            block_at = torch.from_numpy(p.grid(lv, np.arange(len(t["ids"])))).to(dev)
            n = [int(v) for v in p.root * 2 ** lv]
            cells = torch.from_numpy(cells).to(dev)
            src, face = [], []
            for c in self.e:
                y = [cells[:, a] - c[a] for a in range(d)]
                which = torch.full_like(y[0], -1)
                best = torch.zeros_like(y[0])
                for a in range(d):
                    for side, beyond in ((0, y[a] < 0), (1, y[a] >= 4 * n[a])):
                        r = rank[faces[2 * a + side][0]]
                        take = beyond & (best < r)
                        which[take], best[take] = 2 * a + side, r
                    y[a] = y[a] % (4 * n[a])
                b = block_at[tuple(v // 4 for v in y)]
                at = b * self.m + sum((v % 4) * 4 ** a for a, v in enumerate(y))
                gone = (b < 0) | (which >= 0)
                gone |= self.solid[lv][at.clamp(min=0)] & ~gone
                src.append(torch.where(gone, torch.full_like(at, -1), at))
                face.append(torch.where(which >= 0, which, torch.full_like(which, -1)))
            self.src.append(src)
            self.face.append(face)
            # cell classes: Chebyshev distance to the nearest missing block
            dist = np.full((len(t["ids"]), self.m), 99)
            for e in itertools.product((-1, 0, 1), repeat=d):
                miss = p.neighbours(lv, e) == -1
                far = np.zeros(self.m, int)
                for a in range(d):
                    if e[a]:
                        far = np.maximum(far, off[:, a] + 1 if e[a] < 0 else 4 - off[:, a])
                dist[miss] = np.minimum(dist[miss], far)
            self.cls.append(torch.from_numpy(np.where(dist <= 2, 2, np.where(dist <= 4, 1, 0))).to(dev))
            if lv:
                up = p.levels[lv - 1]
                at = p.grid(lv - 1, np.arange(len(up["ids"])))[tuple((t["pos"] // 2).T)]
                kid = ((t["pos"] % 2) * 2 ** np.arange(d)).sum(-1)
                self.par.append((torch.from_numpy(at).to(dev), torch.from_numpy(kid).to(dev)))
            else:
                self.par.append(None)

    def relax(self, f, r):
        """f_eq + (f - f_eq) r."""
        e = equilibrium(*moments(f, self.q), self.q)
        return e + (f - e) * r

    def interpolate(self, lv, all_from=None):
        """Ghost cells of level lv + 1 from level lv; all_from: every cell of the
        blocks from that index on instead."""
        at, kid = self.par[lv + 1]
        lo = 0 if all_from is None else all_from
        need = torch.nonzero((self.cls[lv + 1] == 2).any(1) if all_from is None else
                             torch.arange(len(at), device=self.dev) >= lo)[:, 0]
        if not len(need):
            return
        q = self.q
        g = self.relax(self.f[lv], self.tau[lv + 1] / (2 * self.tau[lv])).reshape(q, -1, self.m)
        g = g[:, at[need]].reshape((q, -1) + (4,) * self.d)
        wt = np.zeros((2, 4, 4))                       # [child half][cell][parent cell]
        for c, i in itertools.product(range(2), range(4)):
            if self.case["interp"] == "linear":
                x = -0.25 + 0.5 * i
                wt[c, i, 2 * c], wt[c, i, 2 * c + 1] = 1 - x, x
            else:
                x = (2 * (i + 4 * c) - 1) / 4          # nodes 0, 1, 2, 3
                for k in range(4):
                    wt[c, i, k] = np.prod([(x - j) / (k - j) for j in range(4) if j != k])
        wt = torch.from_numpy(wt).to(self.dev)
        for a in range(self.d):                        # axis a is dimension -1 - a
            half = (kid[need] >> a) & 1
            g = torch.einsum("nij,qn...j->qn...i", wt[half], g.transpose(-1, -1 - a)).transpose(-1, -1 - a)
        g = g.reshape(q, -1, self.m)
        fine = self.f[lv + 1].reshape(q, -1, self.m)
        put = (self.cls[lv + 1][need] == 2) if all_from is None else torch.ones_like(g[0], dtype=torch.bool)
        put &= ~self.solid[lv + 1].reshape(-1, self.m)[need]
        fine[:, need] = torch.where(put, g, fine[:, need])

    def average(self, lv, sync):
        """Level lv + 1 into level lv: interface cells, or with sync every cell
        that is not a ghost."""
        q, d = self.q, self.d
        at, kid = self.par[lv + 1]
        if not len(at):
            return
        g = self.relax(self.f[lv + 1], 2 * self.tau[lv] / self.tau[lv + 1])
        g = g.reshape((q, -1) + (2, 2) * d)
        g = g.mean(dim=tuple(3 + 2 * a for a in range(d))).reshape(q, -1, self.nc)
        cls = self.cls[lv + 1].reshape((-1,) + (2, 2) * d)
        for a in range(d):
            cls = cls.select(2 + a, 0)
        cls = cls.reshape(-1, self.nc)
        grp = torch.arange(self.nc, device=self.dev)
        cell = sum((2 * ((kid[:, None] >> a) & 1) + ((grp >> a) & 1)) * 4 ** a for a in range(d))
        to = at[:, None] * self.m + cell
        put = ((cls != 2) if sync else (cls == 1)) & ~self.solid[lv][to]
        self.f[lv][:, to[put]] = g[:, put]

    def collide(self, lv):
        """f* and the velocities it was computed with."""
        rho, u = moments(self.f[lv], self.q)
        return self.f[lv] + (equilibrium(rho, u, self.q) - self.f[lv]) / self.tau[lv], u

    def step_level(self, lv):
        fine = lv + 1 < len(self.p.levels) and len(self.p.levels[lv + 1]["ids"]) > 0
        if fine:
            self.interpolate(lv)
        fs, u = self.collide(lv)
        us = 1.5 * sum(v * v for v in u)
        new = torch.empty_like(fs)
        for p in range(self.q):
            s, face, o = self.src[lv][p], self.face[lv][p], self.opp[p]
            back = fs[o].clone()
            for k, fc in enumerate(self.cfg["faces"]):
                at = face == k
                if fc[0] == "moving":
                    back[at] += -6 * self.w[o] * sum(self.e[o][a] * fc[1][a] for a in range(self.d))
                elif fc[0] == "outlet":
                    cu = sum(self.e[o][a] * u[a][at] for a in range(self.d))
                    back[at] = -back[at] + 2 * self.w[o] * (1 + 4.5 * cu * cu - us[at])
            new[p] = torch.where(s >= 0, fs[p][s.clamp(min=0)], back)
        self.f[lv] = torch.where(self.solid[lv], self.f[lv], new)
        if fine:
            self.step_level(lv + 1)
            self.step_level(lv + 1)
            self.average(lv, self.case["interp"] == "cubic")

    def sync(self):
        for lv in reversed(range(len(self.p.levels) - 1)):
            self.average(lv, True)
        for lv in range(len(self.p.levels) - 1):
            self.interpolate(lv)

    def refine(self, lv, mask):
        """Adapt: synchronise, then new children with every cell interpolated."""
        self.sync()
        old = len(self.p.levels[lv + 1]["ids"]) if lv + 1 < len(self.p.levels) else 0
        self.p.refine(lv, mask)
        new = self.p.levels[lv + 1]
        if lv + 1 == len(self.f):
            self.f.append(torch.empty((self.q, 0), dtype=torch.float64, device=self.dev))
        more = (len(new["ids"]) - old) * self.m
        self.f[lv + 1] = torch.cat([self.f[lv + 1], self.f[lv + 1].new_zeros((self.q, more))], 1)
        self.link()
        self.interpolate(lv, all_from=old)

    def by_id(self, per_level, width):
        """[cap][width] from per-level [blocks][width]."""
        out = torch.zeros((self.cfg["max_blocks"], width), dtype=torch.float64, device=self.dev)
        for t, v in zip(self.p.levels, per_level):
            out[torch.from_numpy(t["ids"]).to(self.dev)] = v.reshape(-1, width)
        return out

    def populations(self):
        return torch.stack([self.by_id([f[k] for f in self.f], self.m) for k in range(self.q)])

    def state(self):
        out = []
        for f in self.f:
            rho, u = moments(f, self.q)
            out.append(torch.stack([rho] + u, -1))
        return dict(rho_u=self.by_id(out, self.m * (1 + self.d)).reshape(-1),
                    f=self.populations().reshape(-1))

    def force(self):
        total = torch.zeros(3, dtype=torch.float64, device=self.dev)
        for lv, t in enumerate(self.p.levels):
            leaf = torch.from_numpy(t["head"] < 0).to(self.dev).repeat_interleave(self.m)
            fs, _ = self.collide(lv)
            dx = self.cfg["length_x"] / (self.cfg["nx"] * 2 ** lv)
            shape = [int(v) for v in self.p.root * 2 ** lv]
            block_at = torch.from_numpy(self.p.grid(lv, np.arange(len(t["ids"])))).to(self.dev)
            cells = torch.from_numpy((t["pos"][:, None, :] * 4 + cell_offsets(self.d)).reshape(-1, self.d)).to(self.dev)
            for p, c in enumerate(self.e):
                y = [cells[:, a] + c[a] for a in range(self.d)]
                ok = leaf & ~self.solid[lv]
                for a in range(self.d):
                    ok = ok & (y[a] >= 0) & (y[a] < 4 * shape[a])
                    y[a] = y[a].clamp(0, 4 * shape[a] - 1)
                b = block_at[tuple(v // 4 for v in y)]
                at = b * self.m + sum((v % 4) * 4 ** a for a, v in enumerate(y))
                ok = ok & (b >= 0) & self.solid[lv][at.clamp(min=0)]
                for a in range(3):
                    total[a] += 2 * dx ** (self.d - 1) * c[a] * fs[p][ok].sum()
        return total

    def features(self):
        """The 27 block summaries."""
        lmax, per = self.case["levels"], []

        def squash(v):
            return torch.sign(v) * torch.log1p(v.abs())

        for lv, f in enumerate(self.f):
            rho, u = moments(f, self.q)
            inv_dx = self.cfg["nx"] * 2 ** lv / self.cfg["length_x"]
            rho = rho.reshape(-1, 64)
            u = [v.reshape(-1, 4, 4, 4) for v in u]
            grad = []
            for v in u:
                for a in range(3):
                    g = v.diff(dim=3 - a)
                    last = g.select(3 - a, 2).unsqueeze(3 - a)
                    grad.append(torch.cat([g, last], 3 - a).reshape(-1, 64) * inv_dx)
            u = [v.reshape(-1, 64) for v in u]
            om = ((grad[7] - grad[5]) ** 2 + (grad[2] - grad[6]) ** 2 + (grad[3] - grad[1]) ** 2).sqrt()
            speed = (u[0] ** 2 + u[1] ** 2 + u[2] ** 2).sqrt()
            col = [squash(g.mean(1)) for g in grad] + [squash(g.abs().amax(1)) for g in grad]
            col += [(rho.mean(1) - 1) * 100, (rho.amax(1) - rho.amin(1)) * 100]
            col += [v.mean(1) * 20 for v in u] + [speed.amax(1) * 20, squash(om.mean(1)), squash(om.amax(1))]
            col.append(torch.full_like(col[0], lv / lmax))
            per.append(torch.stack(col, -1))
        return self.by_id(per, 27)


def exact_train(case, seed, dev):
    x, y, w = train_inputs(case, seed, dev)
    x, y, w = x.double(), y.double(), w.double()
    n = case["samples"]

    def splitmix(z):
        k = (1 << 64) - 1
        z = (z + 0x9E3779B97F4A7C15) & k
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & k
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & k
        return z ^ (z >> 31)

    def net(w, x):
        a = [w[:1728].reshape(64, 27), w[1728:1792], w[1792:5888].reshape(64, 64), w[5888:5952],
             w[5952:6016], w[6016]]
        h = torch.relu(x @ a[0].T + a[1])
        return torch.relu(h @ a[2].T + a[3]) @ a[4] + a[5]

    mul = (splitmix(3) % n) | 1
    while math.gcd(mul, n) != 1:
        mul += 2
    order = (torch.arange(n, device=dev) * mul + splitmix(4) % n) % n
    m, v, total = torch.zeros_like(w), torch.zeros_like(w), 0.0
    for t, at in enumerate(order.split(case["batch"]), 1):
        w.requires_grad_(True)
        z = net(w, x[at])
        loss = (4.0 * y[at] * torch.nn.functional.softplus(-z) +
                (1 - y[at]) * torch.nn.functional.softplus(z)).sum()
        g, = torch.autograd.grad(loss, w)
        g, w, total = g / len(at), w.detach(), total + float(loss)
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        w = w - 2e-3 * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8)
    # inference reads FP16 weights
    return dict(loss=np.float64(total / n), params=w, adam_m=m, adam_v=v, half=w,
                prob=torch.sigmoid(net(w.half().double(), x[n:])))


def exact(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    if case["kind"] == "train":
        return exact_train(case, seed, dev)
    if case["kind"] == "batch":
        out = []
        for i, c in enumerate(members_of(case)):
            x = Exact(c, seed + 1000 * i, dev)
            for _ in range(case["steps"]):
                x.step_level(0)
            x.sync()
            out.append(x.state())
        return out
    x = Exact(case, seed, dev)
    if case["kind"] == "propose":
        x.sync()
        return dict(marks=None, features=x.features())
    if case["kind"] == "adapt":
        lv, mask = adapt_marks(case, seed)
        x.refine(lv, mask)
        return dict(blocks=None, nbr=None, f=x.populations().reshape(-1))
    for _ in range(case["steps"]):
        x.step_level(0)
    x.sync()
    out = x.state()
    if case["flow"] == "prism":
        out["force"] = x.force()
    return out
