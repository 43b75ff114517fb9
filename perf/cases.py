"""The workloads that the framework's speed is judged by.

Each case is one call (or one plan run) through the public Python entry points, on
graphs of the families and sizes that the benchmark, the tests and the batched
workload use: G(n, m), R-MAT-ER / G / B with edge factor 8, 2-D meshes and random
geometric graphs, from ten thousand to sixteen million vertices.

Graphs are generated on the GPU with torch from the seed alone: edges are sampled,
ids shuffled, loops and duplicates dropped, rows sorted.  A case's ``n`` need not be a
power of two: an R-MAT graph of n vertices keeps the first n shuffled ids of the next
power of two.

The asynchronous form (``color_async``) is not a case: its colors depend on the
schedule, so two correct runs have no common answer to compare.
"""
import math
import random

import torch

import paper_1205_3809_gb300 as gc

RMAT = {"er": (0.25, 0.25, 0.25, 0.25), "g": (0.45, 0.15, 0.15, 0.25), "b": (0.55, 0.15, 0.15, 0.15)}
PARAMS = gc.MLP_PARAMS


def listed():
    return [
        # the benchmark's smallest graph: launches, round trips and host work
        {"name": "color_gnm_10k", "do": "color", "family": "gnm", "n": 10000, "ef": 5, "keys": "none", "validate": 0},
        # a mesh of a simulation, 949 x 1051, checked by the library on entry (untrusted input)
        {"name": "color_mesh_1m_checked", "do": "color", "family": "mesh", "n": 997399, "ef": 2, "keys": "none",
         "validate": 1},
        # the benchmark's uniform graph
        {"name": "color_er_s22", "do": "color", "family": "er", "n": 1 << 22, "ef": 8, "keys": "none", "validate": 0},
        # an ordinary skewed graph of odd size with the caller's own order (largest degree first)
        {"name": "color_g_1m_keys", "do": "color", "family": "g", "n": 1000003, "ef": 8, "keys": "degree",
         "validate": 0},
        # the headline graph
        {"name": "color_b_s24", "do": "color", "family": "b", "n": 1 << 24, "ef": 8, "keys": "none", "validate": 0},
        # the learned form end to end: features, network, keys, coloring
        {"name": "learned_g_s23", "do": "learned", "family": "g", "n": 1 << 23, "ef": 8},
        # a graph in pinned host memory, colors back in host memory
        {"name": "host_b_s22", "do": "host", "family": "b", "n": 1 << 22, "ef": 8},
        # a planned batch of the mixed workload: 1,024 graphs of 1,000 to 200,000 vertices
        {"name": "batch_1024", "do": "batch", "count": 1024, "lo": 1000, "hi": 200000},
        # a one-call batch of small graphs: planned, run and freed in the call
        {"name": "batch_once_96", "do": "batch_once", "count": 96, "lo": 500, "hi": 20000},
        # the features alone (training data of the network, or keys kept for later)
        {"name": "features_b_s22", "do": "features", "family": "b", "n": 1 << 22, "ef": 8},
        # the network alone, on an odd number of rows
        {"name": "forward_4m", "do": "forward", "n": 4194301},
        # one training step at the shipped model's batch size
        {"name": "train_64k", "do": "train", "n": 65536},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    do = rng.choice(["color", "color", "color", "color", "learned", "host", "batch", "batch_once", "features",
                     "forward", "train"])
    if do == "color":
        family = rng.choice(["gnm", "mesh", "rgg", "er", "g", "b"])
        n = _log(rng, 8000, {"mesh": 4e6, "rgg": 2e6, "gnm": 4e6, "er": 8e6, "g": 1.2e7, "b": 1.4e7}[family])
        ef = {"mesh": 2, "rgg": 4, "gnm": rng.choice([3, 5, 8])}.get(family, 8 if n > 3e6 else rng.choice([4, 8, 16]))
        return {"do": do, "family": family, "n": n, "ef": ef, "keys": rng.choice(["none", "none", "degree", "random"])
                if n < 4e6 else "none", "validate": rng.choice([0, 0, 1])}
    if do in ("learned", "features"):
        return {"do": do, "family": rng.choice(["g", "b", "er", "mesh"]), "n": _log(rng, 8000, 4e6), "ef": 8}
    if do == "host":
        return {"do": do, "family": rng.choice(["g", "b", "gnm"]), "n": _log(rng, 8000, 4e6), "ef": 8}
    if do == "batch":
        return {"do": do, "count": _log(rng, 150, 1024), "lo": rng.choice([200, 1000]), "hi": _log(rng, 5000, 200000)}
    if do == "batch_once":
        return {"do": do, "count": _log(rng, 8, 256), "lo": 500, "hi": _log(rng, 2000, 20000)}
    if do == "forward":
        return {"do": do, "n": _log(rng, 1000, 1.6e7)}
    return {"do": do, "n": _log(rng, 4096, 262144)}


# ------------------------------------------------------------------ graphs

def _gen(seed, salt=0):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + 7919 * salt + 12345) & 0x7FFFFFFFFFFFFFFF)
    return g


def _csr(n, u, v):
    """Symmetric int32 CSR (rows sorted, no loops, no duplicates) of an undirected edge list."""
    keep = u != v
    u, v = u[keep].long(), v[keep].long()
    key = torch.cat([u * n + v, v * n + u])
    del u, v
    key = key.sort().values
    if key.numel():
        keep = torch.ones_like(key, dtype=torch.bool)
        torch.ne(key[1:], key[:-1], out=keep[1:])
        key = key[keep]
    row = key // n
    colidx = (key - row * n).to(torch.int32)
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(torch.bincount(row, minlength=n), 0, out=rowptr[1:])
    return rowptr.to(torch.int32), colidx


def _rmat_pairs(levels, m, abcd, g):
    """m vertex pairs of 2**levels ids by R-MAT's recursive quadrants."""
    a, b, c, _ = abcd
    u = torch.zeros(m, dtype=torch.int32, device="cuda")
    v = torch.zeros(m, dtype=torch.int32, device="cuda")
    for _ in range(levels):
        r = torch.rand(m, device="cuda", generator=g)
        low = r >= a + b                       # quadrants c, d: the lower half of the rows
        right = ((r >= a) & ~low) | (r >= a + b + c)
        u.mul_(2).add_(low)
        v.mul_(2).add_(right)
    return u, v


def _rgg_pairs(sizes, g):
    """Edges of random geometric graphs of the given sizes (average degree 8), on union ids."""
    dev = "cuda"
    n = torch.tensor(sizes, dtype=torch.int64, device=dev)
    gid = torch.repeat_interleave(torch.arange(len(sizes), device=dev), n)
    r = torch.sqrt(8.0 / (math.pi * n.double())).clamp(max=1.0)
    cells = torch.clamp((1.0 / r).long(), min=1)
    base = torch.cumsum(cells * cells, 0) - cells * cells
    total = int((cells * cells).sum())
    x = torch.rand(gid.numel(), device=dev, generator=g, dtype=torch.float64)
    y = torch.rand(gid.numel(), device=dev, generator=g, dtype=torch.float64)
    nc = cells[gid]
    cx = torch.minimum((x * nc).long(), nc - 1)
    cy = torch.minimum((y * nc).long(), nc - 1)
    cell = base[gid] + cy * nc + cx
    order = cell.argsort()
    start = torch.zeros(total + 1, dtype=torch.int64, device=dev)
    torch.cumsum(torch.bincount(cell, minlength=total), 0, out=start[1:])
    us, vs = [], []
    place = torch.arange(gid.numel(), device=dev)     # position in cell order
    x, y, cx, cy, nc, cell, gid = x[order], y[order], cx[order], cy[order], nc[order], cell[order], gid[order]
    r2 = (r * r)[gid]
    for dx, dy in ((0, 0), (1, 0), (-1, 1), (0, 1), (1, 1)):
        ok = (cx + dx >= 0) & (cx + dx < nc) & (cy + dy < nc)
        other = torch.where(ok, cell + dy * nc + dx, torch.zeros_like(cell))
        lo = place + 1 if (dx, dy) == (0, 0) else start[other]
        cnt = torch.where(ok, start[other + 1] - lo, torch.zeros_like(lo)).clamp(min=0)
        i = torch.repeat_interleave(place, cnt)
        first = torch.cumsum(cnt, 0) - cnt
        j = lo[i] + torch.arange(i.numel(), device=dev) - first[i]
        near = (x[i] - x[j]) ** 2 + (y[i] - y[j]) ** 2 <= r2[i]
        us.append(order[i[near]])
        vs.append(order[j[near]])
    return torch.cat(us), torch.cat(vs)


def _graph(case, seed):
    family, n, ef = case["family"], case["n"], case["ef"]
    g = _gen(seed)
    if family == "gnm":
        m = n * ef
        u = torch.randint(n, (m,), device="cuda", generator=g)
        v = torch.randint(n, (m,), device="cuda", generator=g)
        return _csr(n, u, v)
    if family == "mesh":
        cols = max(1, int(round(math.sqrt(1.1075 * n))))  # the last row may be ragged
        ids = torch.arange(n, device="cuda")
        perm = torch.randperm(n, device="cuda", generator=g)
        right = ids[(ids % cols != cols - 1) & (ids + 1 < n)]
        down = ids[ids + cols < n]
        return _csr(n, torch.cat([perm[right], perm[down]]), torch.cat([perm[right + 1], perm[down + cols]]))
    if family == "rgg":
        u, v = _rgg_pairs([n], g)
        perm = torch.randperm(n, device="cuda", generator=g)
        return _csr(n, perm[u], perm[v])
    levels = max(1, (n - 1).bit_length())
    u, v = _rmat_pairs(levels, ef << levels, RMAT[family], g)
    perm = torch.randperm(1 << levels, device="cuda", generator=g).to(torch.int32)
    u, v = perm[u.long()], perm[v.long()]
    if n < 1 << levels:
        keep = (u < n) & (v < n)
        u, v = u[keep], v[keep]
    return _csr(n, u, v)


def _batch_shapes(case):
    """(family, vertices, detail) of every graph: the mixed workload's sizes and families, the
    same for every seed (which changes the graphs)."""
    rng = random.Random("%d %d %d" % (case["count"], case["lo"], case["hi"]))
    out = []
    for _ in range(case["count"]):
        n = _log(rng, case["lo"], case["hi"])
        kind = rng.choice(["grid", "rgg", "rmat"])
        if kind == "grid":
            rows = max(1, int(round(math.sqrt(n))))
            cols = max(1, int(round(n / rows)))
            out.append((kind, rows * cols, cols))
        elif kind == "rgg":
            out.append((kind, n, 0))
        else:
            s = max(1, int(round(math.log2(n))))
            out.append((kind, 1 << s, s))
    return out


def _batch(case, seed):
    """(rowptr_cat, colidx_cat, vertex offsets, edge offsets) of a batch, made as one union."""
    dev = "cuda"
    shapes = _batch_shapes(case)
    g = _gen(seed, 1)
    sizes = torch.tensor([s[1] for s in shapes], dtype=torch.int64)
    voff = torch.zeros(len(shapes) + 1, dtype=torch.int64)
    torch.cumsum(sizes, 0, out=voff[1:])
    N = int(voff[-1])
    voff_d = voff.to(dev)
    us, vs = [], []
    for kind in ("grid", "rgg", "rmat"):
        idx = [i for i, s in enumerate(shapes) if s[0] == kind]
        if not idx:
            continue
        off = voff_d[torch.tensor(idx, device=dev)]
        nk = torch.tensor([shapes[i][1] for i in idx], dtype=torch.int64, device=dev)
        if kind == "grid":
            cols = torch.tensor([shapes[i][2] for i in idx], dtype=torch.int64, device=dev)
            k = torch.repeat_interleave(torch.arange(len(idx), device=dev), nk)
            loc = torch.arange(k.numel(), device=dev) - (torch.cumsum(nk, 0) - nk)[k]
            right = loc % cols[k] != cols[k] - 1
            down = loc + cols[k] < nk[k]
            at = off[k] + loc
            us += [at[right], at[down]]
            vs += [at[right] + 1, (at + cols[k])[down]]
        elif kind == "rgg":
            u, v = _rgg_pairs([shapes[i][1] for i in idx], g)
            k = torch.repeat_interleave(torch.arange(len(idx), device=dev), nk)
            at = off[k] + torch.arange(k.numel(), device=dev) - (torch.cumsum(nk, 0) - nk)[k]
            us.append(at[u])
            vs.append(at[v])
        else:
            lev = torch.tensor([shapes[i][2] for i in idx], dtype=torch.int32, device=dev)
            k = torch.repeat_interleave(torch.arange(len(idx), device=dev), 8 * nk)
            a, b, c, _ = RMAT["g"]
            u = torch.zeros(k.numel(), dtype=torch.int64, device=dev)
            v = torch.zeros(k.numel(), dtype=torch.int64, device=dev)
            for level in range(max(shapes[i][2] for i in idx)):
                r = torch.rand(k.numel(), device=dev, generator=g)
                on = (lev > level)[k]
                low = r >= a + b
                right = ((r >= a) & ~low) | (r >= a + b + c)
                u = torch.where(on, u * 2 + low, u)
                v = torch.where(on, v * 2 + right, v)
            us.append(off[k] + u)
            vs.append(off[k] + v)
    gid = torch.repeat_interleave(torch.arange(len(shapes), device=dev), sizes.to(dev))
    # ids shuffled inside every graph
    order = ((gid << 31) + torch.randint(1 << 31, (N,), device=dev, generator=g)).argsort()
    perm = torch.empty_like(order)
    perm[order] = torch.arange(N, device=dev)
    rowptr, colidx = _csr(N, perm[torch.cat(us)], perm[torch.cat(vs)])
    del us, vs
    rowptr = rowptr.long()
    eoff = rowptr[voff_d]
    row_graph = torch.repeat_interleave(torch.arange(len(shapes), device=dev), eoff[1:] - eoff[:-1])
    colidx -= voff_d[row_graph].to(torch.int32)
    del row_graph
    # every graph's own rowptr (n_g + 1 entries, from 0)
    rowptr_cat = torch.empty(N + len(shapes), dtype=torch.int32, device=dev)
    rowptr_cat[torch.arange(N, device=dev) + gid] = (rowptr[:-1] - eoff[gid]).to(torch.int32)
    rowptr_cat[voff_d[1:] + torch.arange(len(shapes), device=dev)] = (eoff[1:] - eoff[:-1]).to(torch.int32)
    return rowptr_cat, colidx, voff.numpy(), eoff.cpu().numpy()


# ------------------------------------------------------------------- cases

def _mlp_inputs(n, seed):
    """Feature rows as graphs give them: degree-like counts on a log scale, most of them small."""
    g = _gen(seed, 2)
    x = torch.rand(n, 6, device="cuda", generator=g)
    x = x * x * 16.0
    x[:, 1] = x[:, 0].floor()
    return x


def prepare(case, seed):
    do = case["do"]
    if do == "forward":
        return {"do": do, "params": gc.load_priority_model(device="cuda"), "x": _mlp_inputs(case["n"], seed)}
    if do == "train":
        x = _mlp_inputs(case["n"], seed)
        t = 20.0 - x[:, 0] + torch.rand(case["n"], device="cuda", generator=_gen(seed, 3))
        return {"do": do, "trainer": gc.MlpTrainer(gc.load_priority_model(device="cuda")), "x": x, "t": t}
    if do in ("batch", "batch_once"):
        packed = _batch(case, seed)
        s = {"do": do, "packed": packed}
        if do == "batch":
            s["plan"] = gc.Batch(*packed)
        return s
    rowptr, colidx = _graph(case, seed)
    s = {"do": do, "rowptr": rowptr, "colidx": colidx}
    if do == "color":
        s["keys"] = None
        if case["keys"] == "degree":
            deg = rowptr[1:] - rowptr[:-1]
            s["keys"] = deg.max() - deg
        elif case["keys"] == "random":
            s["keys"] = torch.randint(1 << 31, (case["n"],), dtype=torch.int32, device="cuda", generator=_gen(seed, 4))
        s["options"] = {"validate": 1} if case["validate"] else None
        s["out"] = torch.empty(case["n"], dtype=torch.int32, device="cuda")
    elif do == "learned":
        s["params"] = gc.load_priority_model(device="cuda")
    elif do == "host":
        s["rowptr"] = rowptr.cpu().pin_memory()
        s["colidx"] = colidx.cpu().pin_memory()
        s["out"] = torch.empty(case["n"], dtype=torch.int32).pin_memory()
    return s


def run(s):
    do = s["do"]
    if do == "color":
        r = gc.color(s["rowptr"], s["colidx"], s["keys"], out=s["out"], options=s["options"])
        return {"colors": r.colors, "ncolors": r.ncolors, "rounds": r.rounds}
    if do == "learned":
        r = gc.color_learned(s["rowptr"], s["colidx"], s["params"])
        return {"colors": r.colors, "ncolors": r.ncolors, "rounds": r.rounds}
    if do == "host":
        r = gc.color_host(s["rowptr"], s["colidx"], out=s["out"])
        return {"colors": r.colors, "ncolors": r.ncolors, "rounds": r.rounds}
    if do == "batch":
        b = s["plan"]
        b.run()
        return {"colors": b.colors, "ncolors": b.ncolors, "rounds": b.rounds}
    if do == "batch_once":
        colors, ncolors, rounds = gc.color_batched(*s["packed"])
        return {"colors": colors, "ncolors": ncolors, "rounds": rounds}
    if do == "features":
        return gc.features(s["rowptr"], s["colidx"])
    if do == "forward":
        return gc.mlp_forward(s["params"], s["x"])
    t = s["trainer"]
    sse = t.step(s["x"], s["t"])
    return {"sse": sse, "grad": t.grad, "params": t.params, "m": t.m, "v": t.v}


def work(case):
    """The graph read once, the results written once; the network's multiply-adds."""
    do = case["do"]
    if do == "forward":
        return {"bytes": case["n"] * 28 + PARAMS * 4, "flops": 2.0 * 1248 * case["n"]}
    if do == "train":
        # forward, the error carried back through layers 2 and 3, every weight's gradient
        return {"bytes": case["n"] * 28 + PARAMS * 28, "flops": 2.0 * (1248 + 1056 + 1248) * case["n"]}
    if do in ("batch", "batch_once"):
        # expected sizes of the mix: mean of a log-uniform size, 20/3 edges per vertex over the families
        lo, hi = case["lo"], case["hi"]
        n = case["count"] * (hi - lo) / math.log(hi / lo)
        return {"bytes": n * 8 + n * 9.3 * 4, "flops": 0}
    n, nnz = case["n"], 2.0 * case["ef"] * case["n"]
    if do == "features":
        return {"bytes": 4 * n + 4 * nnz + 24 * n, "flops": 0}
    keys = 4 * n if case.get("keys", "none") != "none" else 0
    network = 2.0 * 1248 * n if do == "learned" else 0
    return {"bytes": 4 * n + 4 * nnz + 4 * n + keys, "flops": network}


def tolerance(case):
    """Colors, counts and features are whole numbers (features: whole multiples of 2^-16): the
    same for every correct implementation.  The network's scores and gradients are 32-bit sums
    with bf16 operands: an activation on the edge of two bf16 values may round either way when
    a sum is taken in another order (measured against 64 bits: 7.5e-6 in the scores), and Adam's
    1 - 0.999 is 1.3e-5 off in 32 bits."""
    if case["do"] == "forward":
        return {"rel": 3e-5}
    if case["do"] == "train":
        return {"rel": 5e-5}
    return "exact"


# ------------------------------------------------- the same results in 64 bits

def _bf16(x):
    return x.to(torch.float32).to(torch.bfloat16).to(torch.float64)


def _network(params, x):
    p = params.double()
    w1, b1 = _bf16(p[0:192]).reshape(32, 6), p[192:224]
    w2, b2 = _bf16(p[224:1248]).reshape(32, 32), p[1248:1280]
    w3, b3 = _bf16(p[1280:1312]), p[1312]
    a0 = _bf16(x)
    a1 = _bf16(torch.relu(a0 @ w1.T + b1))
    a2 = _bf16(torch.relu(a1 @ w2.T + b2))
    return a0, a1, a2, a2 @ w3 + b3, w2, w3


def _log2_1p(x):
    """The piecewise-linear log2(1 + x) of the features: exponent plus mantissa cut to 16 bits."""
    m = x.to(torch.int64) + 1
    e = torch.frexp(m.double())[1].to(torch.int64) - 1
    r = m - (torch.ones_like(m) << e)
    frac = torch.where(e >= 16, r >> (e - 16).clamp(min=0), r << (16 - e).clamp(min=0))
    return (e * 65536 + frac).double() / 65536.0


def exact(case, seed):
    do = case["do"]
    if do == "forward":
        s = prepare(case, seed)
        return torch.cat([_network(s["params"], x)[3] for x in s["x"].split(1 << 20)])
    if do == "train":
        s = prepare(case, seed)
        p, n = s["trainer"].params.double(), case["n"]
        a0, a1, a2, y, w2, w3 = _network(s["trainer"].params, s["x"])
        err = y - s["t"].double()
        dy = 2.0 / n * err
        d2 = torch.where(a2 > 0, dy[:, None] * w3, torch.zeros_like(a2))
        d1 = torch.where(a1 > 0, d2 @ w2, torch.zeros_like(a1))
        grad = torch.cat([(d1.T @ a0).reshape(-1), d1.sum(0), (d2.T @ a1).reshape(-1), d2.sum(0), dy @ a2,
                          dy.sum().reshape(1)])
        m, v = 0.1 * grad, 0.001 * grad * grad
        params = p - 3e-3 * (m / 0.1) / (torch.sqrt(v / 0.001) + 1e-8)
        return {"sse": (err * err).sum().reshape(1), "grad": grad, "params": params, "m": m, "v": v}
    if do == "features":
        s = prepare(case, seed)
        rowptr, colidx, n = s["rowptr"].long(), s["colidx"].long(), case["n"]
        d = rowptr[1:] - rowptr[:-1]
        row = torch.repeat_interleave(torch.arange(n, device="cuda"), d)
        dn = d[colidx]
        total = torch.zeros(n, dtype=torch.int64, device="cuda").index_add_(0, row, dn)
        most = torch.zeros(n, dtype=torch.int64, device="cuda").scatter_reduce_(0, row, dn, "amax")
        least = torch.full((n,), 1 << 40, device="cuda").scatter_reduce_(0, row, dn, "amin")
        some = d > 0
        zero = torch.zeros(n, dtype=torch.float64, device="cuda")
        whole = torch.frexp((d + 1).double())[1].double() - 1
        pick = lambda q: torch.where(some, _log2_1p(torch.where(some, q, torch.zeros_like(q))), zero)  # noqa: E731
        return torch.stack([_log2_1p(d), whole, pick(total // d.clamp(min=1)), pick(most), pick(total), pick(least)], 1)
    return None
