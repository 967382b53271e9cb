"""The work that programs have this package do, case by case, for timing.

A case is a dict of plain values; ``prepare`` turns it into what a program has
in hand on the GPU (matrices, plan, gradient of the loss, bound batch),
``run`` makes one pass through the public entry points and ``exact`` states the
same result in 64 bits with plain torch.  Inputs follow the workload classes of
the benchmark: R-MAT graphs (0.57, 0.19, 0.19, 0.05) with relabelled vertices,
Erdos-Renyi graphs with a fixed row length, and B with distinct uniform columns
per row at a given density (the fractional part rounded per row).
"""
import math
import random

import torch

from paper_2408_11988_gb300 import DeviceCSR, Plan
from paper_2408_11988_gb300.autograd import ts_spgemm
from paper_2408_11988_gb300.batched import BatchedProduct
from paper_2408_11988_gb300.force2vec import Force2Vec
from paper_2408_11988_gb300.msbfs import msbfs

DEV = "cuda"


def _product(name, mode, graph, n, deg, d, density):
    return {"name": name, "kind": "product", "mode": mode, "graph": graph, "n": n, "deg": deg, "d": d,
            "density": density}


def listed():
    return [
        # A small product in a serving loop: the Erdos-Renyi workload, captured once and replayed on new values.
        _product("er16k_replay", "replay", "er", 16384, 8, 64, 0.10),
        # The smallest training step, of odd sizes: launches and the host decide.
        _product("er3k_train", "train", "er", 3001, 5, 40, 0.125),
        # An ordinary training step of a sparse embedding (forward, then both gradients through autograd).
        _product("rmat18_train", "train", "rmat", 1 << 18, 16, 128, 0.05),
        # The benchmark's headline: the scale-22 embedding product, forward and backward.
        _product("rmat22_train", "train", "rmat", 1 << 22, 16, 256, 0.05),
        # The largest product: scale 24, 1024 columns at 1%, forward and backward.
        _product("rmat24_train", "train", "rmat", 1 << 24, 16, 1024, 0.01),
        # Inference with B 80% sparse and 128 columns, the usual shape of a sparse embedding.
        _product("rmat20_forward", "forward", "rmat", 1 << 20, 16, 128, 0.20),
        # Very many columns (the d sweep goes to 16,384), above the dense accumulators; odd number of rows.
        _product("wide_forward", "forward", "rmat", 65521, 16, 8192, 0.002),
        # Training that has to repeat bit for bit: the backward without atomics (dB_mode = 2); ragged sizes.
        _product("rmat19_repeatable", "repeatable", "rmat", 500009, 16, 100, 0.08),
        # Many uneven graphs served together: one graph replay of the batched forward and backward.
        {"name": "batched12", "kind": "batched", "count": 12, "log2n_lo": 12.0, "log2n_hi": 18.0, "shapes": 4},
        # Breadth-first search from 128 sources at once, the benchmark's graph.
        {"name": "bfs20", "kind": "bfs", "n": 1 << 20, "deg": 16, "sources": 128, "parents": False},
        # The BFS trees of a smaller search, odd numbers of vertices and sources.
        {"name": "bfs_trees", "kind": "bfs", "n": 300007, "deg": 12, "sources": 50, "parents": True},
        # One minibatch of sparse Force2Vec training (80% sparse, 5 negative samples).
        {"name": "force2vec", "kind": "force2vec", "n": 1 << 18, "deg": 16, "d": 128, "k": 26, "batch": 4096,
         "negatives": 5},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _size(rng, lo, hi):
    return max(int(lo), min(int(hi), int(round(_log(rng, lo, hi)))))


def draw(rng):
    kind = rng.choice(["small", "train", "train", "forward", "forward", "wide", "repeatable", "batched", "bfs", "bfs",
                       "force2vec"])
    if kind == "bfs":
        return {"kind": "bfs", "n": _size(rng, 5000, 1 << 20), "deg": rng.randint(8, 16),
                "sources": rng.randint(1, 128), "parents": rng.random() < 0.5}
    if kind == "force2vec":
        d = rng.choice([64, 100, 128])
        return {"kind": "force2vec", "n": _size(rng, 20000, 500000), "deg": rng.randint(8, 16), "d": d,
                "k": rng.randint(d // 10, d // 5), "batch": _size(rng, 256, 4096), "negatives": rng.randint(3, 6)}
    if kind == "batched":
        return {"kind": "batched", "count": rng.randint(3, 12), "log2n_lo": 12.0,
                "log2n_hi": round(rng.uniform(14.0, 18.0), 2), "shapes": rng.randint(10, 1 << 30)}
    graph = rng.choice(["er", "rmat", "rmat"])
    deg = rng.randint(4, 24)
    if kind == "small":
        n, d, mode = _size(rng, 1000, 30000), _size(rng, 8, 256), rng.choice(["replay", "train", "forward"])
        per_row = _log(rng, 1, 0.25 * d)
    elif kind == "wide":
        n, d, mode = _size(rng, 5000, 100000), _size(rng, 4097, 16384), "forward"
        per_row = _log(rng, 4, 32)
    elif kind == "repeatable":
        n, d, mode = _size(rng, 20000, 1 << 20), _size(rng, 16, 256), "repeatable"
        per_row = _log(rng, 1, min(24, 0.25 * d))
    elif kind == "forward":
        n, d, mode = _size(rng, 30000, 1 << 21), _size(rng, 4, 1024), "forward"
        per_row = _log(rng, 1, min(96 if d <= 256 else 48, 0.8 * d))
    else:
        n, d, mode = _size(rng, 30000, 1 << 22), _size(rng, 16, 1024), "train"
        per_row = _log(rng, 1, min(32, 0.3 * d))
    density = float("%.3g" % (per_row / d))
    while n * deg * density * d > 8e8:  # products: less than the largest listed case
        n //= 2
    return {"kind": "product", "mode": mode, "graph": graph, "n": n, "deg": deg, "d": d, "density": density}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) & 0x7FFFFFFF)
    return g


def _distinct(n, d, m, g):
    """n rows of m distinct uniform columns of [0, d), ascending (Floyd's sampling, all rows at once)."""
    if m > 48:  # many of few columns: the m smallest of d random keys
        out = torch.empty(n, m, dtype=torch.int32, device=DEV)
        step = max(1, (1 << 27) // d)
        for r in range(0, n, step):
            keys = torch.rand(min(step, n - r), d, generator=g, device=DEV)
            out[r:r + step] = keys.topk(m, dim=1, largest=False, sorted=False).indices.to(torch.int32)
    else:
        cols = torch.empty(m, n, dtype=torch.int32, device=DEV)
        for j in range(m):
            top = d - m + j
            t = torch.rand(n, generator=g, device=DEV, dtype=torch.float64).mul_(top + 1).to(torch.int32).clamp_(max=top)
            seen = torch.zeros(n, dtype=torch.bool, device=DEV)
            for i in range(j):
                seen |= cols[i] == t
            cols[j] = torch.where(seen, torch.full_like(t, top), t)
        out = cols.t().contiguous()
    return out.sort(dim=1).values


def _tall_skinny(n, d, density, g, perm):
    """rowptr and columns of B: density * d columns per row, the fraction rounded per row at random; row v of
    the pattern goes to row perm[v]."""
    want = min(density * d, float(d))
    m = int(math.ceil(want - 1e-9))
    cols = _distinct(n, d, m, g)
    keep = torch.ones(n, m, dtype=torch.bool, device=DEV)
    if m > want:
        drop = torch.rand(n, generator=g, device=DEV) < m - want
        at = torch.randint(0, m, (n,), generator=g, device=DEV)
        keep[torch.arange(n, device=DEV), at] = ~drop
    inverse = torch.empty_like(perm)
    inverse[perm] = torch.arange(n, device=DEV)
    cols, keep = cols[inverse], keep[inverse]
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(keep.sum(1), 0, out=rowptr[1:])
    return rowptr, cols[keep]


def _rmat(n, deg, g, perm, symmetric=False):
    """rowptr and columns of an R-MAT graph: deg * n edges, self-loops and duplicates removed, vertex v
    relabelled perm[v]."""
    scale = max(1, (n - 1).bit_length())
    parts, have, want = [], 0, deg * n
    while have < want:
        m = want if n == 1 << scale else int(1.5 * (want - have)) + 1024
        src = torch.zeros(m, dtype=torch.int64, device=DEV)
        dst = torch.zeros(m, dtype=torch.int64, device=DEV)
        for _ in range(scale):
            u = torch.rand(m, generator=g, device=DEV)
            down = u >= 0.76  # quadrants 0.57, 0.19 above, 0.19, 0.05 below
            src.mul_(2).add_(down)
            dst.mul_(2).add_(torch.where(down, u >= 0.95, u >= 0.57))
        if n != 1 << scale:
            ok = (src < n) & (dst < n)
            src, dst = src[ok][:want - have], dst[ok][:want - have]
        parts.append((perm[src], perm[dst]))
        have += int(src.numel())
    src, dst = (torch.cat([p[i] for p in parts]) if len(parts) > 1 else parts[0][i] for i in (0, 1))
    ok = src != dst
    src, dst = src[ok], dst[ok]
    if symmetric:
        src, dst = torch.cat([src, dst]), torch.cat([dst, src])
    key = torch.unique(src * n + dst)
    del src, dst
    rows = torch.div(key, n, rounding_mode="floor")
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(torch.bincount(rows, minlength=n), 0, out=rowptr[1:])
    return rowptr, (key - rows * n).to(torch.int32)


def _graph(case, g, perm, symmetric=False):
    n = case["n"]
    if case.get("graph", "rmat") == "er":
        k = min(case["deg"], n)
        cols = torch.empty(n, k, dtype=torch.int32, device=DEV)
        cols[perm] = perm[_distinct(n, n, k, g).long()].to(torch.int32)
        return torch.arange(n + 1, device=DEV, dtype=torch.int64) * k, cols.sort(dim=1).values.reshape(-1).contiguous()
    return _rmat(n, case["deg"], g, perm, symmetric)


def _matrices(case, seed):
    """A with U(0,1) values and B with N(0,1) values.  The patterns of one case are the same up to a relabelling
    of the vertices, which the seed draws with the values: A * B then has equally many entries for every seed."""
    g, fixed = _gen(seed), _gen(240811988)
    perm = torch.randperm(case["n"], generator=g, device=DEV)
    rp, ci = _graph(case, fixed, perm)
    A = DeviceCSR(case["n"], case["n"], rp, ci, torch.rand(ci.numel(), generator=g, device=DEV))
    rp, ci = _tall_skinny(case["n"], case["d"], case["density"], fixed, perm)
    B = DeviceCSR(case["n"], case["d"], rp, ci, torch.randn(ci.numel(), generator=g, device=DEV))
    return A, B, g


def _gradient(A, B, g):
    """dC, N(0,1) on the pattern of A * B."""
    return torch.randn(Plan(A, B).symbolic(A, B)[1], generator=g, device=DEV)


def _instances(case):
    """The shapes of a batch: n log-uniform, d and density uneven, the same for every seed of the inputs."""
    rng = random.Random(case["shapes"])
    out = []
    for _ in range(case["count"]):
        n = int(2.0 ** rng.uniform(case["log2n_lo"], case["log2n_hi"]))
        d = rng.choice([32, 64, 128, 256])
        out.append({"n": n, "deg": rng.randint(8, 32), "d": d, "density": float("%.3g" % _log(rng, 0.01, 0.50))})
    return out


def _negatives(case, g):
    return torch.randint(0, case["n"], (case["batch"] * case["negatives"],), generator=g, device=DEV, dtype=torch.int32)


def _embedding(case, g):
    n, k = case["n"], case["k"]
    col = _distinct(n, case["d"], k, g).reshape(-1).contiguous()
    return DeviceCSR(n, case["d"], torch.arange(n + 1, device=DEV, dtype=torch.int64) * k, col,
                     0.1 * torch.randn(n * k, generator=g, device=DEV))


def prepare(case, seed):
    if case["kind"] == "product":
        A, B, g = _matrices(case, seed)
        if case["mode"] in ("forward", "replay"):
            plan = Plan(A, B)
            state = {"case": case, "A": A, "B": B, "plan": plan}
            if case["mode"] == "replay":
                state["graph"], state["C"] = plan.capture_forward(A, B)
            return state
        dC = _gradient(A, B, g)
        plan = Plan(A, B, tuning={"dB_mode": 2}) if case["mode"] == "repeatable" else Plan(A, B)
        return {"case": case, "A": A, "B": B, "plan": plan, "dC": dC, "A_val": A.val.requires_grad_(),
                "B_val": B.val.requires_grad_()}
    if case["kind"] == "batched":
        As, Bs, dCs = [], [], []
        for i, shape in enumerate(_instances(case)):
            A, B, g = _matrices(shape, 1000 * seed + i)
            As.append(A)
            Bs.append(B)
            dCs.append(_gradient(A, B, g))
        batch = BatchedProduct(As, Bs)
        batch.bind_grads(dCs)
        return {"case": case, "batch": batch, "graph": batch.capture(backward=True), "nnz": [t.numel() for t in dCs]}
    g = _gen(seed)
    rp, ci = _rmat(case["n"], case["deg"], g, torch.randperm(case["n"], generator=g, device=DEV), symmetric=True)
    A = DeviceCSR(case["n"], case["n"], rp, ci)
    if case["kind"] == "bfs":
        with_edges = torch.nonzero(rp[1:] > rp[:-1]).reshape(-1)
        pick = torch.randperm(with_edges.numel(), generator=g, device=DEV)[:case["sources"]]
        return {"case": case, "A": A, "sources": with_edges[pick].to(torch.int32)}
    Z = _embedding(case, g)
    return {"case": case, "Z": Z, "neg": _negatives(case, g),
            "model": Force2Vec(A, Z, case["k"], negatives=case["negatives"], batch=case["batch"])}


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(state):
    case = state["case"]
    if case["kind"] == "product":
        A, B, plan = state["A"], state["B"], state["plan"]
        if case["mode"] == "replay":
            state["graph"].replay()
            C = state["C"]
            return [C.rowptr, C.col, C.val]
        if case["mode"] == "forward":
            C = plan.forward(A, B)
            return [C.rowptr, C.col, C.val]
        C = ts_spgemm(A, B, state["A_val"], state["B_val"], plan)
        dA, dB = torch.autograd.grad(C.val, (state["A_val"], state["B_val"]), state["dC"])
        return [C.rowptr, C.col, C.val.detach(), dA, dB]
    if case["kind"] == "batched":
        state["graph"].replay()
        b = state["batch"]
        return [[C.rowptr, C.col[:m], C.val[:m], dA, dB]
                for C, m, dA, dB in zip(b.Cs, state["nnz"], b.dAs, b.dBs)]
    if case["kind"] == "bfs":
        r = msbfs(state["A"], state["sources"], parents=case["parents"])
        return {"levels": r.levels, "parents": r.parents}
    U = state["model"].step(case["n"] // 3, state["neg"], want_u=True)
    return {"U": U, "Z_col": state["Z"].col, "Z_val": state["Z"].val}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _expected(case):
    """Stored entries of A, B and C and products that inputs of this shape have (C's from A's row lengths)."""
    n, d, m = case["n"], case["d"], min(case["density"] * case["d"], case["d"])
    rp, _ = _graph(case, _gen(1), torch.arange(n, device=DEV))
    deg = (rp[1:] - rp[:-1]).double()
    nnz_c = float((d * -torch.expm1(deg * math.log1p(-min(m / d, 1 - 1e-12)))).sum())
    return n, float(rp[-1]), n * m, nnz_c, float(rp[-1]) * m


def work(case):
    if case["kind"] in ("product", "batched"):
        total, flops = 0.0, 0.0
        train = case["kind"] == "batched" or case["mode"] in ("train", "repeatable")
        for c in (_instances(case) if case["kind"] == "batched" else [case]):
            n, a, b, nnz_c, products = _expected(c)
            total += 8 * 3 * (n + 1) + 8 * (a + b + nnz_c)  # A and B read, C written
            flops += 2 * products
            if train:  # dC read; dA and dB written
                total += 4 * (nnz_c + a + b)
                flops += 4 * products
        return {"bytes": total, "flops": flops}
    n, edges = case["n"], 2.0 * case["deg"] * case["n"]
    if case["kind"] == "bfs":  # the graph read, levels (and parents) written; one OR an edge and source
        s = case["sources"]
        return {"bytes": 8 * (n + 1) + 4 * edges + 4 * n * s * (2 if case["parents"] else 1), "flops": edges * s}
    b, k, d = case["batch"], case["k"], case["d"]
    terms = b * (edges / n + case["negatives"])  # rows of Z met by the minibatch
    return {"bytes": 12 * b + 4 * terms + 8 * k * (2 * b + min(terms, n)) + 4 * b * d, "flops": 4.0 * terms * k}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------

def _product64(A, B, dC=None):
    """C's values on its pattern (ascending columns), and dA and dB for dC, in 64 bits: row blocks of A,
    every product on its own."""
    n, d = A.nrows, B.ncols
    acol = A.col.long()
    blen = (B.rowptr[1:] - B.rowptr[:-1])
    per = blen[acol]  # products of each entry of A
    before = torch.zeros(per.numel() + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(per, 0, out=before[1:])
    row_products = before[A.rowptr].cpu()
    aptr = A.rowptr.cpu()
    bval, aval = B.val.detach().double(), A.val.detach().double()
    C = []
    dA = torch.zeros(per.numel(), dtype=torch.float64, device=DEV) if dC is not None else None
    dB = torch.zeros(B.nnz, dtype=torch.float64, device=DEV) if dC is not None else None
    r, at = 0, 0
    while r < n:
        most = min(n, r + max(1, (1 << 28) // d))
        e = int(torch.searchsorted(row_products, int(row_products[r]) + (1 << 26), right=True)) - 1
        e = max(r + 1, min(most, e))
        a0, a1 = int(aptr[r]), int(aptr[e])
        k, m = acol[a0:a1], per[a0:a1]
        entry = torch.repeat_interleave(torch.arange(a1 - a0, device=DEV), m)
        p = B.rowptr[k][entry] + torch.arange(entry.numel(), device=DEV) - (before[a0:a1] - before[a0])[entry]
        row = torch.repeat_interleave(torch.arange(e - r, device=DEV), A.rowptr[r + 1:e + 1] - A.rowptr[r:e])
        key = row[entry] * d + B.col[p]
        dense = torch.zeros((e - r) * d, dtype=torch.float64, device=DEV)
        hit = torch.zeros((e - r) * d, dtype=torch.bool, device=DEV)
        dense.scatter_add_(0, key, aval[a0:a1][entry] * bval[p])
        hit[key] = True
        C.append(dense[hit])
        if dC is not None:
            g = torch.zeros_like(dense)
            g[hit] = dC[at:at + C[-1].numel()].double()
            t = g[key]
            dA[a0:a1].scatter_add_(0, entry, t * bval[p])
            dB.scatter_add_(0, p, t * aval[a0:a1][entry])
        at += C[-1].numel()
        r = e
    return torch.cat(C), dA, dB


def exact(case, seed):
    if case["kind"] == "bfs":
        return None
    if case["kind"] == "product":
        A, B, g = _matrices(case, seed)
        dC = _gradient(A, B, g) if case["mode"] in ("train", "repeatable") else None
        C, dA, dB = _product64(A, B, dC)
        return [None, None, C] + ([dA, dB] if dC is not None else [])
    if case["kind"] == "batched":
        out = []
        for i, shape in enumerate(_instances(case)):
            A, B, g = _matrices(shape, 1000 * seed + i)
            out.append([None, None, *_product64(A, B, _gradient(A, B, g))])
        return out
    g = _gen(seed)
    rp, ci = _rmat(case["n"], case["deg"], g, torch.randperm(case["n"], generator=g, device=DEV), symmetric=True)
    Z = _embedding(case, g)
    neg = _negatives(case, g).long().view(case["batch"], case["negatives"])
    n, r0, b = case["n"], case["n"] // 3, case["batch"]
    dense = torch.zeros(n, case["d"], dtype=torch.float64, device=DEV)
    dense.scatter_(1, Z.col.long().view(n, -1), Z.val.double().view(n, -1))
    a0, a1 = int(rp[r0]), int(rp[r0 + b])
    row = torch.repeat_interleave(torch.arange(b, device=DEV), rp[r0 + 1:r0 + b + 1] - rp[r0:r0 + b])
    row = torch.cat([row, torch.arange(b, device=DEV).repeat_interleave(case["negatives"])])
    other = torch.cat([ci[a0:a1].long(), neg.reshape(-1)])
    s = torch.sigmoid((dense[r0 + row] * dense[other]).sum(1))
    w = torch.where(torch.arange(row.numel(), device=DEV) < a1 - a0, 1 - s, -s)
    U = dense[r0:r0 + b].clone().index_add_(0, row, 0.02 * w[:, None] * dense[other])
    return {"U": U, "Z_col": None, "Z_val": None}
