"""Performance cases of the GB300 Delaunay library: what its users run, through its public calls.

Every case is one whole use of the package: points in, canonical tetrahedra out (the form in which
two triangulations can be compared), or a training run of the learned scheduler's network. The
sizes follow the repository's own workloads (uniform clouds, the degenerate mix, the cube + slab,
batches of clouds, box refinement, the learned schedule), from a cloud of a few dozen points up to
the benchmark's 1e7.

Kinds ("kind" of a case):
  insert   one cloud through a handle that is kept: clear, insert, canonical tetrahedra;
  append   a mesh that grows: a first insert, then further chunks into the same handle;
  host     the same as insert from and to page-locked host memory (the end-to-end call);
  batch    many independent clouds in one call, rows into page-locked host memory;
  refine   Delaunay refinement of a unit cube from its surface lattice;
  train    the learned scheduler's network: Adam steps on logged features.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1805_08831_gb300 as dt
from paper_1805_08831_gb300 import learned, synth


def listed():
    return [
        # a mesher's smallest call: a cloud of one BRIO round less one point; launches and host
        # latency are all of it
        {"name": "uniform_2047", "kind": "insert", "cloud": "uniform", "n": 2047},
        # a mid-sized cloud, the repository's first configuration
        {"name": "uniform_1e5", "kind": "insert", "cloud": "uniform", "n": 100_000},
        # the benchmark's headline cloud
        {"name": "uniform_1e7", "kind": "insert", "cloud": "uniform", "n": 10_000_000},
        # scanned or CAD-like data: points on a sphere, in clusters and on a lattice, with
        # duplicates and exactly degenerate configurations
        {"name": "degenerate_1e6", "kind": "insert", "cloud": "degenerate", "n": 1_000_000},
        # strongly varying density: cube plus thin slab, an odd count
        {"name": "slab_3000001", "kind": "insert", "cloud": "slab", "n": 3_000_001},
        # the same with the trained schedule
        {"name": "slab_learned_1e6", "kind": "insert", "cloud": "slab", "n": 1_000_000, "learned": True},
        # host data in, host data out
        {"name": "host_1e6", "kind": "host", "cloud": "uniform", "n": 1_000_000},
        # points that arrive in chunks
        {"name": "append_3e5_4x50001", "kind": "append", "cloud": "uniform", "n": 300_000, "chunks": 4,
         "chunk": 50_001},
        # thousands of points to tens of thousands per cloud, many clouds
        {"name": "batch_512", "kind": "batch", "clouds": 512, "lo": 50, "hi": 50_000},
        # a few small clouds
        {"name": "batch_64_small", "kind": "batch", "clouds": 64, "lo": 50, "hi": 2_000},
        # volume mesh of a box from its boundary mesh
        {"name": "refine_48", "kind": "refine", "k": 48},
        # fitting the scheduler's network
        {"name": "train_100x4096", "kind": "train", "rows": 400_000, "batch": 4096, "steps": 100},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["insert", "insert", "insert", "append", "host", "batch", "refine", "train"])
    if kind == "insert":
        cloud = rng.choice(["uniform", "uniform", "degenerate", "slab"])
        hi = {"uniform": 10_000_000, "degenerate": 1_000_000, "slab": 3_000_000}[cloud]
        c = {"kind": kind, "cloud": cloud, "n": _log(rng, 64, hi)}
        if cloud == "slab" and c["n"] >= 10_000 and rng.random() < 0.5:
            c["learned"] = True
        return c
    if kind == "host":
        return {"kind": kind, "cloud": rng.choice(["uniform", "slab"]), "n": _log(rng, 1_000, 2_000_000)}
    if kind == "append":
        n = _log(rng, 1_000, 1_000_000)
        return {"kind": kind, "cloud": rng.choice(["uniform", "slab"]), "n": n, "chunks": rng.randint(1, 5),
                "chunk": _log(rng, 100, max(200, n // 4))}
    if kind == "batch":
        lo, hi = rng.choice([(50, 2_000), (50, 50_000), (1_000, 10_000)])
        most = {2_000: 4_096, 50_000: 512, 10_000: 1_024}[hi]
        return {"kind": kind, "clouds": _log(rng, 16, most), "lo": lo, "hi": hi}
    if kind == "refine":
        return {"kind": kind, "k": rng.randint(6, 48)}
    return {"kind": kind, "rows": _log(rng, 20_000, 400_000), "batch": _log(rng, 200, 8_192),
            "steps": rng.randint(10, 100)}


# ------------------------------------------------------------------ inputs (on the GPU, by seed)
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _uniform(n, g):
    return torch.rand((n, 3), generator=g, device="cuda", dtype=torch.float64)


def _cloud(kind, n, g):
    """The recipes of the package's synthetic clouds, drawn on the device."""
    if kind == "uniform":
        return _uniform(n, g)
    if kind == "slab":  # 70 % in the cube, 30 % in the slab |z - 1/2| < 5e-4
        m = int(round(0.3 * n))
        s = _uniform(m, g)
        s[:, 2] = 0.4995 + 1e-3 * s[:, 2]
        return torch.cat([_uniform(n - m, g), s])
    a, b = (2 * n) // 5, (2 * n) // 5  # sphere, clusters; the rest on the lattice {0..99}^3 / 99
    d = torch.randn((a, 3), generator=g, device="cuda", dtype=torch.float64)
    d = 0.5 + 0.5 * d / d.norm(dim=1, keepdim=True).clamp_min(1e-300)
    centres = _uniform(64, g)
    which = torch.arange(b, device="cuda") % 64
    e = centres[which] + 0.01 * torch.randn((b, 3), generator=g, device="cuda", dtype=torch.float64)
    ijk = torch.randint(0, 100, (n - a - b, 3), generator=g, device="cuda")
    return torch.cat([d, e, ijk.double() / 99.0]).contiguous()


def _sizes(case, seed):
    """Cloud sizes spread evenly over the logarithm, in an order of the seed's own: batches of one
    kind differ in their clouds' places and not in their total work."""
    q = (np.arange(case["clouds"]) + 0.5) / case["clouds"]
    s = np.rint(np.exp(math.log(case["lo"]) + q * (math.log(case["hi"]) - math.log(case["lo"])))).astype(np.int64)
    return np.random.default_rng(seed).permutation(s)


def _total(case):
    return int(_sizes(case, 0).sum())


def _samples(case, seed):
    """Feature rows and labels like those of logged insertions: densities, key fields, the round
    and the boundary distance in [0, 1], log2(1 + |C|) around 4.4 and rare lost conflicts."""
    g = _gen(seed)
    n = case["rows"]
    x = torch.rand((n, dt.DT_FEATURES), generator=g, device="cuda")
    noise = torch.randn((n,), generator=g, device="cuda")
    size = 4.4 + 0.8 * x[:, 2] - 0.6 * x[:, 7] + 0.3 * noise
    lost = (torch.rand((n,), generator=g, device="cuda") < 0.02 + 0.1 * x[:, 0]).float()
    return x, torch.stack([size, lost], dim=1).contiguous()


def prepare(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    if kind == "train":
        x, y = _samples(case, seed)
        return {"case": case, "x": x, "y": y, "params": torch.from_numpy(dt.init_params(seed)).cuda()}
    if case.get("learned"):
        t = dt.Triangulation(seed=seed, schedule=dt.DT_SCHED_LEARNED)
        params, _ = learned.train_scheduler([_cloud("slab", 20_000, g).cpu().numpy()], steps=100, seed=1)
        t.load_model(params)
    else:
        t = dt.Triangulation(seed=seed)
    s = {"case": case, "t": t}
    if kind == "batch":
        s["offsets"] = np.concatenate([[0], np.cumsum(_sizes(case, seed))]).astype(np.uint64)
        n = int(s["offsets"][-1])
        s["xyz"] = _uniform(n, g)
        s["out"] = torch.zeros((7 * n + 64, 4), dtype=torch.int32, pin_memory=True).numpy().view(np.uint32)
    elif kind == "refine":
        k = case["k"]
        lo = _uniform(1, g)  # the box stands anywhere in space
        s["xyz"] = torch.from_numpy(synth.box_surface(k)).cuda() + lo
        s["box"] = tuple(s["xyz"].min(dim=0).values.tolist()) + tuple(s["xyz"].max(dim=0).values.tolist())
    elif kind == "append":
        n, m = case["n"], case["chunk"]
        x = _cloud(case["cloud"], n + case["chunks"] * m, g)
        x = x[torch.randperm(len(x), generator=g, device="cuda")]  # the chunks come from all over
        s["xyz"] = [x[:n].contiguous()] + [x[n + i * m:n + (i + 1) * m].contiguous() for i in range(case["chunks"])]
    elif kind == "host":
        n = case["n"]
        s["xyz"] = _cloud(case["cloud"], n, g).cpu().pin_memory().numpy()
        s["out"] = torch.zeros((7 * n + 64, 4), dtype=torch.int32, pin_memory=True).numpy().view(np.uint32)
    else:
        s["xyz"] = _cloud(case["cloud"], case["n"], g)
    if kind in ("insert", "append", "refine"):
        n = case["k"] ** 3 + 6 * case["k"] ** 2 + 64 if kind == "refine" else _count(case)[1]
        s["tets"] = torch.zeros((7 * n + 64, 4), dtype=torch.int32, device="cuda")
        if kind == "refine":
            s["points"] = torch.zeros((n, 3), dtype=torch.float64, device="cuda")
    return s


def _kept(s, name, rows):
    """The rows in the front of a buffer that the program keeps (its end stays zero), and their
    count: another cloud of the same size has another number of tetrahedra."""
    s[name][: len(rows)].copy_(rows)
    return {"rows_" + name: len(rows), name: s[name]}


def run(s):
    kind = s["case"]["kind"]
    if kind == "train":
        params = s["params"].clone()
        losses = dt.mlp_train(params, s["x"], s["y"], s["case"]["steps"], s["case"]["batch"], 2e-3, 5)
        return {"params": params, "losses": losses}
    t = s["t"]
    if kind == "batch":
        t.batch(s["xyz"], s["offsets"])
        tets, offsets = t.tets_batch(out=s["out"])
        return {"rows": len(tets), "tets": s["out"].view(np.int32), "offsets": offsets.view(np.int64)}
    t.clear()
    if kind == "host":
        t.insert_host(s["xyz"])
        return {"rows": len(t.tets_host(out=s["out"])), "tets": s["out"].view(np.int32)}
    if kind == "append":
        for x in s["xyz"]:
            t.insert(x)
        return _kept(s, "tets", t.tets())
    t.insert(s["xyz"])
    if kind == "refine":
        t.refine(1.0 / s["case"]["k"], box=s["box"])
        return {**_kept(s, "points", t.points()), **_kept(s, "tets", t.tets())}
    return _kept(s, "tets", t.tets())


def _count(case):
    """(points given, points of the result, tetrahedra of the result), about: 6.77 tetrahedra per
    point inside a cloud, fewer towards its hull; 5.05 per point of the degenerate mix."""
    kind = case["kind"]
    inside = lambda n: max(1.0, 6.77 * n - 5.5 * n ** (2 / 3))  # noqa: E731
    if kind == "batch":
        n = _total(case)
        return n, n, sum(inside(int(m)) for m in _sizes(case, 0))
    if kind == "refine":
        k = case["k"]
        given, total = (k + 1) ** 3 - (k - 1) ** 3, 0.47 * k ** 3
        return given, total, 2.6 * k ** 3
    n = case["n"] + case.get("chunks", 0) * case.get("chunk", 0)
    return n, n, 5.05 * n if case["cloud"] == "degenerate" else inside(n)


def work(case):
    """Points read and tetrahedra written once; one insphere decision (about 120 operations) per
    facet, without which no triangulation is known to be Delaunay. Training: the sampled rows and
    the parameters with their moments, read and written each step; three multiply-adds per weight
    and sample (forward, and both products of the backward pass)."""
    if case["kind"] == "train":
        each = case["batch"] * 4 * (dt.DT_FEATURES + 2) + 6 * 4 * dt.DT_MLP_PARAMS
        return {"bytes": case["steps"] * each, "flops": case["steps"] * case["batch"] * 6 * 1344}
    given, total, tets = _count(case)
    bytes_ = 24 * given + 16 * tets + (24 * total if case["kind"] == "refine" else 0)
    return {"bytes": bytes_, "flops": 120 * 2 * tets}


def tolerance(case):
    """The triangulation is unique and its points are a fixed sequence of roundings: integers and
    coordinates are equal. Training sums in 32 bits, in no fixed order, for up to a hundred Adam
    steps, each of which moves a parameter by about the learning rate whatever its gradient."""
    if case["kind"] == "train":
        return {"rel": 1e-5, "max": 1e-3}
    return "exact"


def _mix64(z):
    with np.errstate(over="ignore"):
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return z ^ (z >> np.uint64(31))


def exact(case, seed):
    """Training in 64 bits: minibatches of a SplitMix64 stream per step, backpropagation of the
    squared error plus cross-entropy through 8 -> 32 -> 32 -> 2 with ReLU, and Adam."""
    if case["kind"] != "train":
        return None
    x, y = (v.double().cpu() for v in _samples(case, seed))
    shapes = [(8, 32), (32,), (32, 32), (32,), (32, 2), (2,)]
    p = torch.from_numpy(dt.init_params(seed)).double()
    m, v = torch.zeros_like(p), torch.zeros_like(p)
    losses = []
    k = np.arange(1, case["batch"] + 1, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15)
    for t in range(1, case["steps"] + 1):
        first = np.uint64((5 + t * 0x51ED2701) & ((1 << 64) - 1))
        with np.errstate(over="ignore"):
            idx = torch.from_numpy((_mix64(first + k) % np.uint64(case["rows"])).astype(np.int64))
        q = p.clone().requires_grad_(True)
        w = [a.reshape(s) for a, s in zip(torch.split(q, [math.prod(s) for s in shapes]), shapes)]
        h = torch.relu(x[idx] @ w[0] + w[1])
        h = torch.relu(h @ w[2] + w[3])
        o = h @ w[4] + w[5]
        loss = ((o[:, 0] - y[idx, 0]) ** 2 + torch.nn.functional.softplus(o[:, 1]) - y[idx, 1] * o[:, 1]).mean()
        (g,) = torch.autograd.grad(loss, q)
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        p = p - 2e-3 * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8)
        losses.append(loss.item())
    return {"params": p, "losses": np.array(losses)}
