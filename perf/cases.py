"""The work that programs built on libgila have it do, as cases that can be
timed and checked: inputs from a seed, one pass through the public calls,
what the pass cannot do without, and the same result in plain FP64 torch.

A graph arrives as a CSR, its k-hop lists are built once, then the layout
iterates over them. So the cases are: iterating (whole runs on the device and
from and to host arrays, single steps), building the lists anew, the quality
figures, the layout of a pruned graph (weighted repulsion), and batches of
small graphs. Whole runs use a low initial temperature, as the last and
coldest part of a layout has or a drawn graph that is relaxed again after a
small change: an iteration costs the same at every temperature, and a hot run
of many iterations is chaotic.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_1606_02162_gb300 import gila as G

FP32, FP64, FP32C = G.GILA_FP32, G.GILA_FP64, G.GILA_FP32_COMPENSATED


def listed():
    return [
        # the smallest: a 32 x 32 grid in the FP64 mode, launches and latency
        {"name": "grid32_fp64", "kind": "run", "graph": "grid", "rows": 32, "cols": 32, "k": 2,
         "precision": FP64, "iters": 100, "t0": 0.02},
        # an ordinary small graph from and to host arrays, as a program that draws it calls it
        {"name": "ba10k_k2_host", "kind": "host", "graph": "ba", "n": 10_000, "m": 3, "k": 2,
         "precision": FP32, "iters": 50, "t0": 0.05},
        # a scale-free graph of 300k edges, the default radius
        {"name": "ba100k_k2", "kind": "run", "graph": "ba", "n": 100_000, "m": 3, "k": 2,
         "precision": FP32, "iters": 20, "t0": 0.2},
        # the same graph at radius 3: long rows
        {"name": "ba100k_k3_step", "kind": "step", "graph": "ba", "n": 100_000, "m": 3, "k": 3,
         "precision": FP32},
        # a triangulated mesh of three million edges: short even rows, neighbours near in id
        {"name": "mesh1000_k3", "kind": "run", "graph": "mesh", "rows": 1000, "cols": 1000, "k": 3,
         "precision": FP32C, "iters": 10, "t0": 0.5},
        # a power-law graph whose balls hold a fifth of all vertices: the largest lists
        {"name": "chunglu120k_k3_step", "kind": "step", "graph": "chunglu", "n": 120_000,
         "mean": 8.0, "k": 3, "precision": FP32C},
        # a new graph up to its first moved placement: the lists, the plan and one step
        {"name": "rebuild_chunglu60k_k3", "kind": "rebuild", "graph": "chunglu", "n": 60_000,
         "mean": 8.0, "k": 3, "precision": FP32C},
        {"name": "rebuild_ba1m_k2", "kind": "rebuild", "graph": "ba", "n": 333_334, "m": 3, "k": 2,
         "precision": FP32},
        # quality figures of a finished placement
        {"name": "metrics_ba100k_k3", "kind": "metrics", "graph": "ba", "n": 100_000, "m": 3,
         "k": 3, "precision": FP32},
        # a sparse power-law graph with its degree-one vertices pruned: weighted repulsion
        {"name": "pruned_chunglu100k_k2", "kind": "pruned", "graph": "chunglu", "n": 99_991,
         "mean": 4.0, "k": 2, "precision": FP32, "iters": 10, "t0": 0.2},
        # many small graphs of uneven sizes in one launch, in both widths
        {"name": "batch500_fp32", "kind": "batch", "graph": "mix", "count": 500, "nmin": 50,
         "nmax": 5000, "k": 2, "precision": FP32, "iters": 50, "t0": 0.02},
        {"name": "batch250_fp64", "kind": "batch", "graph": "mix", "count": 250, "nmin": 50,
         "nmax": 5000, "k": 2, "precision": FP64, "iters": 20, "t0": 0.02},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["grid", "host", "run", "step3", "mesh", "dense", "rebuild_dense",
                       "rebuild_sparse", "metrics", "pruned", "batch"])
    if kind == "grid":
        return {"kind": "run", "graph": "grid", "rows": _log_int(rng, 8, 64),
                "cols": _log_int(rng, 8, 64), "k": rng.choice([2, 3]),
                "precision": rng.choice([FP32, FP64]), "iters": rng.randint(20, 100), "t0": 0.02}
    if kind == "host":
        return {"kind": "host", "graph": "ba", "n": _log_int(rng, 1_000, 30_000), "m": 3, "k": 2,
                "precision": rng.choice([FP32, FP32C]), "iters": rng.randint(20, 50), "t0": 0.02}
    if kind == "run":
        return {"kind": "run", "graph": rng.choice(["ba", "er"]), "n": _log_int(rng, 30_000, 333_334),
                "m": 3, "mean": 4.0, "k": 2, "precision": FP32, "iters": rng.randint(5, 20),
                "t0": 0.02}
    if kind == "step3":
        return {"kind": "step", "graph": "ba", "n": _log_int(rng, 20_000, 100_000), "m": 3, "k": 3,
                "precision": rng.choice([FP32, FP32C])}
    if kind == "mesh":
        return {"kind": "run", "graph": "mesh", "rows": _log_int(rng, 200, 1000),
                "cols": _log_int(rng, 200, 1000), "k": rng.choice([2, 3]),
                "precision": rng.choice([FP32, FP32C]), "iters": rng.randint(3, 10), "t0": 0.02}
    if kind == "dense":
        return {"kind": "step", "graph": "chunglu", "n": _log_int(rng, 20_000, 110_000),
                "mean": 8.0, "k": 3, "precision": rng.choice([FP32, FP32C])}
    if kind == "rebuild_dense":
        return {"kind": "rebuild", "graph": "chunglu", "n": _log_int(rng, 15_000, 60_000),
                "mean": 8.0, "k": 3, "precision": FP32C}
    if kind == "rebuild_sparse":
        return {"kind": "rebuild", "graph": rng.choice(["ba", "er"]),
                "n": _log_int(rng, 30_000, 333_334), "m": 3, "mean": 4.0, "k": 2,
                "precision": FP32}
    if kind == "metrics":
        return {"kind": "metrics", "graph": "ba", "n": _log_int(rng, 20_000, 100_000), "m": 3,
                "k": rng.choice([2, 3]), "precision": FP32}
    if kind == "pruned":
        return {"kind": "pruned", "graph": "chunglu", "n": _log_int(rng, 20_000, 100_000),
                "mean": 4.0, "k": 2, "precision": FP32, "iters": rng.randint(3, 10), "t0": 0.02}
    return {"kind": "batch", "graph": "mix", "count": _log_int(rng, 32, 250), "nmin": 50,
            "nmax": 5000, "k": 2, "precision": rng.choice([FP32, FP64]),
            "iters": rng.randint(5, 20), "t0": 0.02}


# ------------------------------------------------------------------- graphs

def _csr(n, a, b):
    """Symmetric simple CSR (rows ascending) of undirected edges, on the GPU."""
    keep = a != b
    a, b = a[keep], b[keep]
    key = torch.unique(torch.cat([a * n + b, b * n + a]))
    src, dst = key // n, key % n
    row = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    row[1:] = torch.cumsum(torch.bincount(src, minlength=n), 0)
    return row, dst


def _grid_edges(rows, cols, diagonals):
    ids = torch.arange(rows * cols, device="cuda").reshape(rows, cols)
    a = [ids[:, :-1].reshape(-1), ids[:-1, :].reshape(-1)]
    b = [ids[:, 1:].reshape(-1), ids[1:, :].reshape(-1)]
    if diagonals:
        a.append(ids[:-1, :-1].reshape(-1))
        b.append(ids[1:, 1:].reshape(-1))
    return torch.cat(a), torch.cat(b)


def _rand(gen, count):
    return torch.rand(count, dtype=torch.float64, device="cuda", generator=gen)


def _ba_edges(n, m, gen):
    """Preferential attachment: each new vertex draws m ends of earlier edges;
    a drawn far end is resolved by following that edge's own draw."""
    first = m * (m + 1) // 2
    pairs = torch.triu_indices(m + 1, m + 1, 1, device="cuda")
    v = torch.arange(m + 1, n, device="cuda").repeat_interleave(m)
    src = torch.cat([pairs[0], v])
    total = src.numel()
    dst = torch.full((total,), -1, dtype=torch.int64, device="cuda")
    dst[:first] = pairs[1]
    slots = 2 * (first + (v - m - 1) * m)
    r = (_rand(gen, total - first) * slots).long()
    ptr = torch.arange(total, device="cuda")
    near = (r & 1) == 0
    dst[first:] = torch.where(near, src[r >> 1], dst[first:])
    ptr[first:] = torch.where(near, ptr[first:], r >> 1)
    for _ in range(64):
        if int((dst < 0).sum()) == 0:
            break
        dst = torch.where(dst < 0, dst[ptr], dst)
        ptr = ptr[ptr]
    return src, dst


def _chunglu_edges(n, mean, gen):
    """Power-law weights (exponent 2.3), endpoints drawn in proportion to them."""
    w = torch.arange(1, n + 1, dtype=torch.float64, device="cuda") ** (-1.0 / 1.3)
    w *= mean / w.mean()
    w = torch.minimum(w, w.sum().sqrt())
    cdf = torch.cumsum(w, 0)
    cdf /= cdf[-1].clone()
    edges = int(n * mean / 2)
    a = torch.searchsorted(cdf, _rand(gen, edges)).clamp_(max=n - 1)
    b = torch.searchsorted(cdf, _rand(gen, edges)).clamp_(max=n - 1)
    return a, b


def _er_edges(n, mean, gen):
    edges = int(n * mean / 2)
    return (_rand(gen, edges) * n).long(), (_rand(gen, edges) * n).long()


def _graph(case, seed):
    """(n, row, col) on the GPU; a mix of small graphs as their disjoint union
    with the vertex offsets of its graphs."""
    gen = torch.Generator(device="cuda")
    # a pruned graph keeps another number of vertices for every graph: there
    # the seed gives the placement alone
    gen.manual_seed(17 if case["kind"] == "pruned" else 1_000_003 * seed + 17)
    kind = case["graph"]
    if kind in ("grid", "mesh"):
        n = case["rows"] * case["cols"]
        a, b = _grid_edges(case["rows"], case["cols"], kind == "mesh")
        row, col = _csr(n, a, b)
        return n, row, col, None
    if kind == "mix":
        rng = np.random.default_rng(case["count"])  # the sizes belong to the case
        sizes = np.rint(np.exp(rng.uniform(math.log(case["nmin"]), math.log(case["nmax"]),
                                           case["count"]))).astype(np.int64)
        kinds = rng.integers(0, 3, case["count"])
        rng = np.random.default_rng(seed)
        voff, us, vs = [0], [], []
        for n, what in zip(sizes.tolist(), kinds.tolist()):
            base = voff[-1]
            if what == 0:  # a random tree under a random relabelling
                p = rng.permutation(n)
                us.append(base + p[1:])
                vs.append(base + p[(rng.random(n - 1) * np.arange(1, n)).astype(np.int64)])
            elif what == 1:  # a near-square grid
                r = max(1, int(round(math.sqrt(n))))
                c = max(1, int(round(n / r)))
                n = r * c
                ids = base + np.arange(n).reshape(r, c)
                us += [ids[:, :-1].ravel(), ids[:-1, :].ravel()]
                vs += [ids[:, 1:].ravel(), ids[1:, :].ravel()]
            else:  # a sparse random graph of mean degree 4
                e = rng.binomial(n * (n - 1) // 2, min(1.0, 4.0 / (n - 1)))
                us.append(base + rng.integers(0, n, e))
                vs.append(base + rng.integers(0, n, e))
            voff.append(base + n)
        n = voff[-1]
        a = torch.from_numpy(np.concatenate(us)).cuda()
        b = torch.from_numpy(np.concatenate(vs)).cuda()
        row, col = _csr(n, a, b)
        return n, row, col, voff
    n = case["n"]
    a, b = (_ba_edges(n, case["m"], gen) if kind == "ba" else
            _chunglu_edges(n, case["mean"], gen) if kind == "chunglu" else
            _er_edges(n, case["mean"], gen))
    row, col = _csr(n, a, b)
    return n, row, col, None


def _positions(case, seed, n, voff):
    """Uniform in the square of side sqrt(n) (each graph of a mix in its own),
    with FP32 values whatever the width they are kept in."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(7_919 * seed + 5)
    x = torch.rand(n, 2, dtype=torch.float32, device="cuda", generator=gen)
    if voff is None:
        x *= math.sqrt(n)
    else:
        size = torch.tensor(np.diff(voff), device="cuda")
        x *= size.float().sqrt().repeat_interleave(size).unsqueeze(1)
    return x.double() if case["precision"] == FP64 else x


def _pruned(n, row, col):
    """Degree-one vertices dropped in one pass (of a single edge the smaller id
    stays): (kept ids, row, col of the rest, weights 1 + dropped neighbours)."""
    deg = row[1:] - row[:-1]
    src = torch.arange(n, device="cuda").repeat_interleave(deg)
    pair = (deg[src] == 1) & (deg[col] == 1) & (src < col)
    drop = deg == 1
    drop[src[pair]] = False
    w = 1.0 + torch.zeros(n, dtype=torch.float64, device="cuda").index_add_(
        0, src, drop[col].double())
    keep = ~drop
    ids = torch.nonzero(keep).reshape(-1)
    new = torch.cumsum(keep, 0) - 1
    e = keep[src] & keep[col]
    prow = torch.zeros(ids.numel() + 1, dtype=torch.int64, device="cuda")
    prow[1:] = torch.cumsum(torch.bincount(new[src[e]], minlength=ids.numel()), 0)
    return ids, prow, new[col[e]], w[ids]


# --------------------------------------------------------------------- runs

def _temperature(n):
    return 0.1 * math.sqrt(n)  # the first temperature of the linear schedule


def prepare(case, seed):
    n, row, col, voff = _graph(case, seed)
    x0 = _positions(case, seed, n, voff)
    prm = G.params(k=case["k"], iters=case.get("iters", 1), t0=case.get("t0", 0.0),
                   precision=case["precision"])
    hrow, hcol = row.cpu().numpy(), col.to(torch.int32).cpu().numpy()
    s = {"kind": case["kind"], "prm": prm, "k": case["k"]}
    if case["kind"] == "batch":
        graphs = [SimpleNamespace(n=b - a, row_ptr=hrow[a:b + 1] - hrow[a],
                                  col_idx=hcol[hrow[a]:hrow[b]] - a)
                  for a, b in zip(voff[:-1], voff[1:])]
        s["owner"] = G.Batch(graphs)
        s["h"] = s["owner"].handle
        G.gila_batch_build_khop(s["h"], case["k"])
        s["x0"], s["x"] = x0, torch.empty_like(x0)
        return s
    s["graph"] = G.Graph(n, hrow, hcol)
    s["h"] = s["graph"].handle
    if case["kind"] == "pruned":
        s["owner"] = G.Pruned(s["graph"])
        s["h"] = s["owner"].pruned_graph
        ids = _pruned(n, row, col)[0]
        x0 = x0[ids].contiguous()
    s["t"] = _temperature(x0.shape[0])
    s["x0"], s["x"], s["disp"] = x0, torch.empty_like(x0), torch.empty_like(x0)
    if case["kind"] == "host":
        s["host"] = x0.double().cpu().numpy()
    # a program in use has its lists and plan: the first step makes them
    G.gila_layout_step(s["h"], prm, s["t"], s["x0"], s["x"], s["disp"])
    return s


def run(s):
    kind, h, prm = s["kind"], s["h"], s["prm"]
    if kind in ("run", "pruned"):
        s["x"].copy_(s["x0"])
        G.gila_layout_run_device(h, prm, s["x"])
        return s["x"]
    if kind == "step":
        G.gila_layout_step(h, prm, s["t"], s["x0"], s["x"], s["disp"])
        return [s["x"], s["disp"]]
    if kind == "host":
        # drawn at single precision
        return G.gila_layout_run(h, prm, s["host"]).astype(np.float32)
    if kind == "rebuild":
        G.gila_khop_reset(h)
        nnz = G.gila_build_khop(h, s["k"])
        G.gila_layout_step(h, prm, s["t"], s["x0"], s["x"], s["disp"])
        return [nnz, s["x"], s["disp"]]
    if kind == "metrics":
        return G.gila_layout_metrics(h, prm, s["x0"])
    s["x"].copy_(s["x0"])
    G.gila_layout_batch_device(h, prm, s["x"])
    return s["x"]


# --------------------------------------------------------------------- work

def _mean_ball(n, row, col, k, samples=192):
    """Mean |N_v(k)| over evenly spaced sources, by breadth-first search."""
    row, col = row.cpu().numpy(), col.cpu().numpy()
    total, src = 0, np.linspace(0, n - 1, min(samples, n)).astype(np.int64)
    for v in src.tolist():
        seen = np.zeros(n, dtype=bool)
        seen[v] = True
        front = np.array([v])
        for _ in range(k):
            deg = row[front + 1] - row[front]
            at = np.repeat(row[front] - np.concatenate([[0], np.cumsum(deg)[:-1]]), deg)
            nxt = col[at + np.arange(deg.sum())]
            nxt = np.unique(nxt[~seen[nxt]])
            seen[nxt] = True
            front = nxt
        total += int(seen.sum()) - 1
    return total / len(src)


def work(case):
    """Per iteration: each list entry's id read once (two bytes tell it within
    a range of ids), the adjacency (four bytes an entry), per vertex a row
    offset (eight bytes) and the position read and written; eleven operations
    a k-hop pair, fourteen an edge. A rebuild writes the lists (four bytes an
    entry) besides, the quality figures read them once."""
    n, row, col, _ = _graph(case, 1)
    if case["kind"] == "pruned":
        _, row, col, _ = _pruned(n, row, col)
        n = row.numel() - 1
    pairs = n * _mean_ball(n, row, col, case["k"])
    edges = float(col.numel())
    width = 16 if case["precision"] == FP64 else 8
    step_bytes = 2 * pairs + 4 * edges + n * (8 + 2 * width)
    step_flops = 11 * pairs + 14 * edges
    if case["kind"] == "rebuild":
        return {"bytes": step_bytes + 4 * pairs + 4 * edges + 8 * n, "flops": step_flops}
    if case["kind"] == "metrics":
        return {"bytes": 2 * pairs + 4 * edges + n * (8 + width), "flops": 8 * pairs / 2 + 8 * edges}
    iters = case.get("iters", 1)
    return {"bytes": step_bytes * iters, "flops": step_flops * iters}


# -------------------------------------------------------------------- exact

def _balls(n, row, col, k, dense):
    """The k-hop lists in chunks of sources: pairs (source, vertex), by source."""
    deg = row[1:] - row[:-1]
    if dense:
        ones = torch.ones(col.numel(), dtype=torch.float32, device="cuda")
        adj = torch.sparse_csr_tensor(row, col, ones, size=(n, n))
        size = max(64, min(n, 120_000_000 // n))
        for a in range(0, n, size):
            b = min(n, a + size)
            reach = torch.zeros(n, b - a, dtype=torch.float32, device="cuda")
            ids = torch.arange(a, b, device="cuda")
            reach[ids, ids - a] = 1.0
            for _ in range(k):
                reach = ((adj @ reach + reach) > 0).float()
            reach[ids, ids - a] = 0.0
            at = torch.nonzero(reach.t())
            yield at[:, 0] + a, at[:, 1]
        return
    size = 50_000
    for a in range(0, n, size):
        b = min(n, a + size)
        src = torch.arange(a, b, device="cuda")
        own = src * n + src
        seen, front = own, own
        for _ in range(k):
            s, v = front // n, front % n
            d = deg[v]
            start = row[v] - (torch.cumsum(d, 0) - d)
            at = start.repeat_interleave(d) + torch.arange(int(d.sum()), device="cuda")
            new = torch.unique(s.repeat_interleave(d) * n + col[at])
            both = torch.unique(torch.cat([seen, new]))
            front = both[~torch.isin(both, seen, assume_unique=True)]
            seen = both
        seen = seen[seen // n != seen % n]
        yield seen // n, seen % n


def _repulsion(x, chunks, w):
    f = torch.zeros_like(x)
    for src, dst in chunks:
        for o in range(0, src.numel(), 30_000_000):
            s, v = src[o:o + 30_000_000], dst[o:o + 30_000_000]
            d = x[s] - x[v]
            r2 = (d * d).sum(1)
            c = torch.where(r2 > 0, 1.0 / r2, torch.zeros_like(r2))
            f.index_add_(0, s, d * (c if w is None else c * w[v]).unsqueeze(1))
    return f


def _move(x, chunks, w, row, col, t):
    f = _repulsion(x, chunks, w)
    src = torch.arange(x.shape[0], device="cuda").repeat_interleave(row[1:] - row[:-1])
    d = x[src] - x[col]
    f.index_add_(0, src, -d * (d * d).sum(1).sqrt().unsqueeze(1))
    norm = (f * f).sum(1).sqrt()
    return f * torch.where(norm > t, t / norm, torch.ones_like(norm)).unsqueeze(1)


def exact(case, seed):
    n, row, col, voff = _graph(case, seed)
    x = _positions(case, seed, n, voff).double()
    w = None
    if case["kind"] == "pruned":
        ids, row, col, w = _pruned(n, row, col)
        x, n = x[ids], ids.numel()
    kind = case["kind"]
    dense = case["k"] >= 3 and case["graph"] in ("ba", "chunglu")
    chunks = _balls(n, row, col, case["k"], dense)
    if kind == "step" or kind == "rebuild":
        disp = _move(x, chunks, w, row, col, _temperature(n))
        out = [x + disp, disp]
        return [None] + out if kind == "rebuild" else out
    if kind == "metrics":
        rep = 0.0
        for src, dst in chunks:
            for o in range(0, src.numel(), 30_000_000):
                d = x[src[o:o + 30_000_000]] - x[dst[o:o + 30_000_000]]
                r = (d * d).sum(1).sqrt()
                rep += float(torch.where(r > 0, 1.0 / r, torch.zeros_like(r)).sum())
        src = torch.arange(n, device="cuda").repeat_interleave(row[1:] - row[:-1])
        d = x[src] - x[col]
        r = (d * d).sum(1).sqrt()[src < col]
        mean, std, att = float(r.mean()), float(r.std(correction=0)), float((r * r).sum())
        return {"edge_mean": mean, "edge_std": std, "edge_cv": std / mean, "rep_total": rep / 2,
                "att_total": att, "rep_att_ratio": rep / 2 / att}
    chunks = list(chunks)
    for i in range(case["iters"]):
        x = x + _move(x, chunks, w, row, col, case["t0"] * (case["iters"] - i) / case["iters"])
    return x
