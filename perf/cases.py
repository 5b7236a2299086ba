"""The workloads whose speed this package is judged by.

A case is a dict of plain values; ``prepare`` builds its inputs on the GPU
from a seed, ``run`` makes one pass through the package's public entry points
(``Context`` and ``LearnedPartitioner``) and returns everything they compute.
The graphs are the shapes the partitioner is used on: structured meshes,
power-law graphs (R-MAT, labels shuffled, isolated vertices kept) and random
geometric graphs with ids in no particular order.  Every result but the
learned form's floats is an exact integer.
"""
import math

import numpy as np
import torch

import paper_2304_13194_gb300 as jet
from paper_2304_13194_gb300 import train_lip

DEV = "cuda"
EPS = 0.03
HIDDEN, FEATS = 64, 16

# One handle per set of options for the whole process, as a program that
# partitions many graphs keeps it (its memory pool stays warm with it).
_handles = {}


def _context(two_hop=False):
    if two_hop not in _handles:
        _handles[two_hop] = jet.Context(0, flags=jet.FLAG_TWO_HOP if two_hop else 0)
    return _handles[two_hop]


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # smallest whole call: a 64 x 64 five-point mesh, 8 parts (latency and launches)
        {"name": "partition_grid64", "op": "partition", "graph": "grid2d", "a": 64, "b": 64, "k": 8},
        # the benchmark workload: a weighted seven-point mesh, 2.1M vertices, 64 parts
        {"name": "partition_mesh128w", "op": "partition", "graph": "grid3d", "a": 128, "b": 128, "c": 128,
         "weights": True, "k": 64},
        # the largest: a power-law graph of 4.2M vertices and 64M edges (a social network or web crawl)
        {"name": "partition_rmat22", "op": "partition", "graph": "rmat", "a": 22, "k": 64},
        # a power-law graph coarsened with two-hop matches: many levels, all with hub rows
        {"name": "partition_rmat17_two_hop", "op": "partition", "graph": "rmat", "a": 17, "k": 64, "two_hop": True},
        # a graph that lives in host memory, copied in and its partition copied out on each call
        {"name": "host_rgg300k", "op": "host", "graph": "rgg", "a": 300000, "k": 32},
        # many graphs of uneven size in one call, each with its own number of parts
        {"name": "batch_rgg48", "op": "batch", "count": 48, "lo": 1000, "hi": 200000},
        # repartitioning: refinement alone, from the partition the program has, ragged weighted mesh
        {"name": "refine_grid1000x777w", "op": "refine", "graph": "grid2d", "a": 1000, "b": 777, "weights": True,
         "k": 32},
        # one Jetlp pass on a small graph, composed by the caller (no allocation on the call)
        {"name": "lp_pass_rgg20k", "op": "lp_pass", "graph": "rgg", "a": 20011, "k": 16},
        # one rebalancing pass on an odd-sized mesh with oversized parts
        {"name": "rebalance_mesh61w", "op": "rebalance", "graph": "grid3d", "a": 61, "b": 53, "c": 47, "weights": True,
         "k": 48},
        # checking a partition: exact cut and part weights of a weighted power-law graph
        {"name": "cut_rmat20w", "op": "cut", "graph": "rmat", "a": 20, "weights": True, "k": 256},
        # learned initial partition: loss and gradient of a training batch of 32 coarsest graphs
        {"name": "lip_loss_grad", "op": "loss_grad", "count": 32, "lo": 320, "hi": 480, "k": 64},
        # learned initial partition in use: the whole call on a weighted mesh
        {"name": "learned_mesh48w", "op": "learned", "graph": "grid3d", "a": 48, "b": 48, "c": 48, "weights": True,
         "k": 64},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_graph(rng, nmin, nmax, scale_lo, scale_hi, kinds=("grid2d", "grid3d", "rgg", "rmat")):
    kind = rng.choice(kinds)
    n = _log_int(rng, nmin, nmax)
    if kind == "grid2d":
        a = max(3, int(math.sqrt(n) * rng.uniform(0.6, 1.6)))
        g = {"graph": kind, "a": a, "b": max(3, n // a)}
    elif kind == "grid3d":
        a = max(3, int(n ** (1 / 3) * rng.uniform(0.7, 1.3)))
        b = max(3, int(n ** (1 / 3) * rng.uniform(0.7, 1.3)))
        g = {"graph": kind, "a": a, "b": b, "c": max(3, n // (a * b))}
    elif kind == "rgg":
        g = {"graph": kind, "a": n}
    else:
        g = {"graph": kind, "a": rng.randint(scale_lo, scale_hi)}
    g["weights"] = rng.random() < 0.5
    return g


def draw(rng):
    op = rng.choice(["partition", "partition", "partition", "two_hop", "host", "batch", "refine", "lp_pass",
                     "rebalance", "cut", "loss_grad", "learned"])
    k = rng.choice([2, 3, 8, 16, 31, 64, 100, 256])
    if op in ("partition", "two_hop"):
        g = _draw_graph(rng, 1000, *((2000000, 12, 21) if op == "partition" else (300000, 12, 17)))
        # an unweighted mesh that is not coarsened is one and the same input for every seed
        g["weights"] = g["weights"] or (g["graph"].startswith("grid") and _sizes(g)[0] <= 16 * k)
        return {"op": "partition", **g, "k": k, **({"two_hop": True} if op == "two_hop" else {})}
    if op == "host":
        return {"op": op, **_draw_graph(rng, 2000, 1000000, 12, 19), "k": k}
    if op == "batch":
        return {"op": op, "count": rng.randint(2, 48), "lo": 1000, "hi": _log_int(rng, 4000, 200000)}
    if op == "refine":
        return {"op": op, **_draw_graph(rng, 1000, 2000000, 12, 20), "k": k}
    if op == "lp_pass":
        return {"op": op, **_draw_graph(rng, 1000, 262144, 10, 17), "k": k}
    if op in ("rebalance", "cut"):
        return {"op": op, **_draw_graph(rng, 1000, 4000000, 12, 21), "k": k}
    if op == "loss_grad":
        lo = _log_int(rng, 100, 4000)
        return {"op": op, "count": rng.randint(1, 32), "lo": lo, "hi": int(lo * rng.uniform(1.1, 2.0)),
                "k": rng.choice([8, 31, 64, 128])}
    return {"op": "learned", **_draw_graph(rng, 4000, 200000, 12, 16), "k": rng.choice([8, 31, 64])}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _edge_weights(gen, u, v, hi=10):
    """Weights 1..hi of the undirected edges {u, v}, equal in both directions."""
    salt = int(torch.randint(1, 1 << 30, (1,), generator=gen, device=DEV).item())
    a, b = torch.minimum(u, v), torch.maximum(u, v)
    h = a * 2654435761 + b * 40503 + salt
    h = (h ^ (h >> 15)) * 2246822519
    h = (h ^ (h >> 13)) & 0x7FFFFFFF
    return (h % hi + 1).to(torch.int32)


def _csr_from_keys(key, n):
    """CSR of the directed edges u * n + v (sorted and made unique here)."""
    key, _ = torch.sort(key)
    if key.numel():
        keep = torch.ones_like(key, dtype=torch.bool)
        keep[1:] = key[1:] != key[:-1]
        key = key[keep]
    u = torch.div(key, n, rounding_mode="floor")
    v = key - u * n
    xadj = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    xadj[1:] = torch.cumsum(torch.bincount(u, minlength=n), 0)
    return xadj, u, v


def _grid(gen, dims):
    n = dims[0] * dims[1] * dims[2]
    ids = torch.arange(n, device=DEV)
    x, y, z = ids % dims[0], ids // dims[0] % dims[1], ids // (dims[0] * dims[1])
    nb, ok, step = [], [], (1, dims[0], dims[0] * dims[1])
    for axis in (2, 1, 0):
        nb.append(ids - step[axis])
        ok.append((x, y, z)[axis] > 0)
    for axis in (0, 1, 2):
        nb.append(ids + step[axis])
        ok.append((x, y, z)[axis] < dims[axis] - 1)
    nb, ok = torch.stack(nb, 1), torch.stack(ok, 1)
    xadj = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    xadj[1:] = torch.cumsum(ok.sum(1), 0)
    return xadj, ids[:, None].expand_as(nb)[ok], nb[ok], ids.double() / n


def _rmat(gen, scale, edge_factor=16):
    n, m = 1 << scale, edge_factor << scale
    u = torch.zeros(m, dtype=torch.int64, device=DEV)
    v = torch.zeros(m, dtype=torch.int64, device=DEV)
    for _ in range(scale):                      # a = .57, b = c = .19, d = .05
        r = torch.rand(m, generator=gen, device=DEV)
        u = 2 * u + (r >= 0.76)
        v = 2 * v + (((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
    label = torch.randperm(n, generator=gen, device=DEV)
    u, v = label[u], label[v]
    off = u != v
    u, v = u[off], v[off]
    xadj, u, v = _csr_from_keys(torch.cat([u * n + v, v * n + u]), n)
    return xadj, u, v, torch.rand(n, generator=gen, device=DEV, dtype=torch.float64)


def _rgg(gen, n, degree=8.0):
    """Random points of the unit square joined within the radius that gives the mean degree."""
    p = torch.rand(n, 2, generator=gen, device=DEV, dtype=torch.float64)
    r = math.sqrt(degree / (math.pi * n))
    g = max(1, min(4096, int(1.0 / r)))
    cell = (p * g).long().clamp_(max=g - 1)
    cid = cell[:, 1] * g + cell[:, 0]
    order = torch.argsort(cid, stable=True)
    start = torch.zeros(g * g + 1, dtype=torch.int64, device=DEV)
    start[1:] = torch.cumsum(torch.bincount(cid, minlength=g * g), 0)
    us, vs = [], []
    ids = torch.arange(n, device=DEV)
    for dy in (-1, 0, 1):                       # three neighbouring cells of a row lie in one piece
        cy = cell[:, 1] + dy
        ok = (cy >= 0) & (cy < g)
        cy = cy.clamp(0, g - 1)
        b = start[cy * g + (cell[:, 0] - 1).clamp(min=0)]
        e = start[cy * g + (cell[:, 0] + 1).clamp(max=g - 1) + 1]
        cnt = torch.where(ok, e - b, torch.zeros_like(b))
        u = torch.repeat_interleave(ids, cnt)
        first = torch.cumsum(cnt, 0) - cnt
        v = order[torch.arange(u.numel(), device=DEV) - first[u] + b[u]]
        near = ((p[u] - p[v]).square().sum(1) < r * r) & (u != v)
        us.append(u[near])
        vs.append(v[near])
    xadj, u, v = _csr_from_keys(torch.cat(us) * n + torch.cat(vs), n)
    return xadj, u, v, p[:, 0]


def _graph(case, gen):
    kind = case["graph"]
    if kind == "grid2d":
        xadj, u, v, pos = _grid(gen, (case["a"], case["b"], 1))
    elif kind == "grid3d":
        xadj, u, v, pos = _grid(gen, (case["a"], case["b"], case["c"]))
    elif kind == "rmat":
        xadj, u, v, pos = _rmat(gen, case["a"])
    else:
        xadj, u, v, pos = _rgg(gen, case["a"])
    n = xadj.numel() - 1
    vw = ew = None
    if case.get("weights"):
        vw = torch.randint(1, 5, (n,), generator=gen, device=DEV, dtype=torch.int32)
        ew = _edge_weights(gen, u, v)
    return {"xadj": xadj, "adjncy": v.to(torch.int32), "vwgt": vw, "adjwgt": ew, "pos": pos, "n": n}


def _start(g, k, gen, skew=1.0, noise=0.02):
    """The partition a caller comes with: slabs of somewhat uneven width along one axis, some
    vertices misplaced; skew above 1 makes the first slabs the large ones."""
    skew = skew * (0.95 + 0.1 * torch.rand(1, generator=gen, device=DEV).item())
    part = (k * (g["pos"] ** skew)).long().clamp_(0, k - 1).to(torch.int32)
    moved = torch.rand(g["n"], generator=gen, device=DEV) < noise
    other = torch.randint(0, k, (g["n"],), generator=gen, device=DEV, dtype=torch.int32)
    return torch.where(moved, other, part)


def _union(gen, count, lo, hi):
    """Block-diagonal union of `count` connected-ish graphs of lo..hi vertices, mean degree 14
    (the coarsest levels a training batch holds)."""
    sizes = torch.randint(lo, hi + 1, (count,), generator=gen, device=DEV).tolist()
    xs, adjs, n, m = [torch.zeros(1, dtype=torch.int64, device=DEV)], [], 0, 0
    for s in sizes:
        xadj, _, v, _ = _rgg(gen, s, degree=14.0)
        xs.append(xadj[1:] + m)
        adjs.append((v + n).to(torch.int32))
        n += s
        m += v.numel()
    return torch.cat(xs), torch.cat(adjs), n


def prepare(case, seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    op, k = case["op"], case.get("k", 2)
    st = {"op": op, "k": k, "seed": seed % (1 << 31) + 1, "ctx": _context(bool(case.get("two_hop")))}
    if op == "batch":
        st["graphs"] = []
        for i in range(case["count"]):          # sizes spread over the logarithm of the range, mixed k
            n = int(case["lo"] * (case["hi"] / case["lo"]) ** ((i * 7 % case["count"] + 0.5) / case["count"]))
            xadj, _, v, _ = _rgg(gen, n)
            st["graphs"].append({"xadj": xadj, "adjncy": v.to(torch.int32), "k": 2 + 2 * (i * 13 % 32), "eps": EPS,
                                 "seed": st["seed"]})
        return st
    if op == "loss_grad":
        st["xadj"], st["adjncy"], n = _union(gen, case["count"], case["lo"], case["hi"])
        st["x"] = st["ctx"].lip_features(st["xadj"], st["adjncy"])
        # labels in step with the features (position in the greedy order), as training pairs have them
        noise = 0.02 * torch.randn(n, generator=gen, device=DEV)
        st["y"] = ((st["x"][:, 3] * case["count"] % 1.0 + noise) * k).long().clamp_(0, k - 1).to(torch.int32)
        st["params"] = train_lip.init_params(k, seed % 1000)
        st["model"] = jet.LearnedPartitioner(st["ctx"], k, st["params"])
        return st
    g = st["g"] = _graph(case, gen)
    st["args"] = (g["xadj"], g["adjncy"], g["vwgt"], g["adjwgt"])
    if op == "host":
        st["args"] = tuple(None if a is None else a.cpu().pin_memory() for a in st["args"])
        st["part"] = torch.empty(g["n"], dtype=torch.int32).pin_memory()
    elif op == "learned":
        st["model"] = jet.LearnedPartitioner(st["ctx"], k, train_lip.init_params(k, seed % 1000))
    elif op in ("refine", "cut"):
        st["part"] = _start(g, k, gen)
    elif op == "lp_pass":
        st["part"] = _start(g, k, gen)
        st["locked"] = (torch.rand(g["n"], generator=gen, device=DEV) < 0.05).to(torch.uint8)
        st["out"] = {"Pd": torch.int32, "F": torch.int32, "inX": torch.uint8, "F2": torch.int32, "inM": torch.uint8}
        st["out"] = {name: torch.empty(g["n"], dtype=t, device=DEV) for name, t in st["out"].items()}
    elif op == "rebalance":
        st["part"] = _start(g, k, gen, skew=1.4)
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(st):
    op, ctx, k = st["op"], st["ctx"], st["k"]
    if op == "partition":
        part, cut = ctx.partition(*st["args"], k=k, eps=EPS, seed=st["seed"])
        return {"part": part, "cut": cut}
    if op == "host":
        part, cut = ctx.partition_host(*st["args"], k=k, eps=EPS, seed=st["seed"], part_out=st["part"])
        return {"part": part, "cut": cut}
    if op == "batch":
        got = ctx.partition_batch(st["graphs"])
        return {"part": torch.cat([p for p, _, _, _ in got]), "cut": np.array([c for _, c, _, _ in got])}
    if op == "refine":
        part, cut = ctx.refine(*st["args"], k, st["part"], eps=EPS, seed=st["seed"])
        return {"part": part, "cut": cut}
    if op == "lp_pass":
        return ctx.lp_pass_noalloc(*st["args"], k, st["part"], locked=st["locked"], c=0.25, out=st["out"])
    if op == "rebalance":
        weak = ctx.rebalance_pass(*st["args"], k, st["part"], eps=EPS, strong=False, seed=st["seed"])
        strong = ctx.rebalance_pass(*st["args"], k, st["part"], eps=EPS, strong=True, seed=st["seed"])
        return {"weak": weak, "strong": strong}
    if op == "cut":
        cut, weights = ctx.cut(*st["args"], k, st["part"])
        return {"cut": cut, "weights": weights}
    if op == "loss_grad":
        loss, grad = st["model"].loss_grad(st["xadj"], st["adjncy"], st["x"], st["y"])
        return {"loss": loss, "grad": grad}
    part, cut, info = st["model"].partition(*st["args"], eps=EPS, seed=st["seed"])
    return {"part": part, "cut": cut, "cut_plain": info["cut_plain"], "cut_learned": info["cut_learned"]}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _sizes(case):
    """(vertices, CSR entries), the entries of a random graph by its expected degree."""
    kind = case["graph"]
    if kind == "rmat":
        n = 1 << case["a"]
        return n, int(2 * 16 * n * 0.93)
    if kind == "rgg":
        return case["a"], 8 * case["a"]
    dims = (case["a"], case["b"], case.get("c", 1))
    n = dims[0] * dims[1] * dims[2]
    return n, 2 * sum(n // d * (d - 1) for d in dims)


def work(case):
    op = case["op"]
    if op == "batch":
        mean = (case["hi"] - case["lo"]) / max(math.log(case["hi"] / case["lo"]), 1e-9)
        n = case["count"] * mean
        return {"bytes": n * (8 + 8 * 4 + 4), "flops": 0}
    if op == "loss_grad":
        n = case["count"] * (case["lo"] + case["hi"]) / 2
        k = case["k"]
        params = 2 * FEATS * HIDDEN + 2 * 2 * HIDDEN * HIDDEN + HIDDEN * k + 3 * HIDDEN + k
        dense = 2 * FEATS * HIDDEN * 2 + 2 * HIDDEN * HIDDEN * 3 * 2 + HIDDEN * k * 3
        gather = 14 * (FEATS + 2 * HIDDEN + 2 * HIDDEN)
        return {"bytes": n * (8 + 14 * 4 + FEATS * 4 + 4) + 8 * params, "flops": n * (2 * dense + gather)}
    n, nnz = _sizes(case)
    csr = 8 * n + 4 * nnz + (4 * n + 4 * nnz if case.get("weights") else 0)
    if op == "lp_pass":
        return {"bytes": csr + n * (4 + 1 + 4 + 4 + 1 + 4 + 1), "flops": 0}
    if op == "rebalance":
        return {"bytes": 2 * (csr + n * (4 + 4 + 4)), "flops": 0}
    if op == "refine":
        return {"bytes": csr + 8 * n, "flops": 0}
    return {"bytes": csr + 4 * n, "flops": 0}


# ---------------------------------------------------------------------------
# the floating results in 64 bits
# ---------------------------------------------------------------------------
def exact(case, seed):
    """Loss and gradient of the network (mean aggregation, three relu layers, softmax
    cross-entropy) in float64.  The other cases return whole numbers."""
    if case["op"] != "loss_grad":
        return None
    st = prepare(case, seed)
    k, n = case["k"], st["x"].shape[0]
    theta = torch.from_numpy(st["params"]).to(DEV).double().requires_grad_(True)
    deg = (st["xadj"][1:] - st["xadj"][:-1])
    row = torch.repeat_interleave(torch.arange(n, device=DEV), deg)
    col = st["adjncy"].long()
    h, at, din = st["x"].double(), 0, FEATS
    for _ in range(3):
        w = theta[at:at + 2 * din * HIDDEN].view(2 * din, HIDDEN)
        at += 2 * din * HIDDEN
        b = theta[at:at + HIDDEN]
        at += HIDDEN
        mean = torch.zeros_like(h).index_add(0, row, h[col]) / deg.clamp(min=1).double()[:, None]
        h = torch.relu(torch.cat([h, mean], 1) @ w + b)
        din = HIDDEN
    w = theta[at:at + HIDDEN * k].view(HIDDEN, k)
    b = theta[at + HIDDEN * k:]
    loss = torch.nn.functional.cross_entropy(h @ w + b, st["y"].long())
    (grad,) = torch.autograd.grad(loss, theta)
    return {"loss": float(loss.detach()), "grad": grad}
