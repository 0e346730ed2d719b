"""The cases that this framework's speed is measured on: typed-graphlet counts through the public calls.

A case names a call (`op`), a graph family with its sizes, the number of node types L and the graphlet size k.

op    one pass
full  tg_build + tg_count + free from a CSR and into buffers on the device (the benchmark's step)
host  the same with a pinned host CSR and pinned host outputs (the benchmark's end-to-end step)
count tg_count on a kept handle (a server's resident graph)
batch tg_count_batch on a kept handle of many graphs (the captured CUDA graph is replayed)
pa    tg_count_position_aware on a kept handle
dir   tg_build_directed + tg_count_directed3 + free
et    tg_build_edge_typed + tg_count_edge_typed3 + free

Graphs are drawn on the device from the seed: Erdos-Renyi (er), Chung-Lu (cl: weights (i + i0)^(-1/(gamma-1)),
largest weight wmax) and a typed block model (sbm: 20 times more edges between blocks than inside, block = type).
Types of er and cl are Zipf(zipf) over L (0: uniform); shuffle: node ids in random order instead of by weight.
"""
import itertools
import math

import numpy as np
import torch

import paper_2010_14058_gb300 as tg


def listed():
    return [
        # the smallest graphs a user counts one at a time: launches and latency
        {"name": "er_small", "op": "full", "graph": "er", "n": 2_000, "m": 10_000, "L": 3, "k": 4},
        # a small request on a resident graph, many types, ids as a user's file has them
        {"name": "resident_small", "op": "count", "graph": "cl", "n": 8_101, "m": 40_503, "L": 8, "k": 4,
         "gamma": 2.2, "wmax": 900.0, "zipf": 0.0, "shuffle": True},
        # a large request on a resident graph (the serving pool's upper end)
        {"name": "resident_1m", "op": "count", "graph": "cl", "n": 199_999, "m": 1_000_003, "L": 7, "k": 4,
         "gamma": 2.2, "wmax": 6_000.0, "zipf": 0.0, "shuffle": True},
        # the ordinary size: a skewed graph of two million edges, built and counted once
        {"name": "cl_mid", "op": "full", "graph": "cl", "n": 200_000, "m": 2_000_000, "L": 5, "k": 4,
         "gamma": 2.1, "wmax": 1.2e4, "zipf": 1.2, "shuffle": False},
        # the headline benchmark's shape: 20 M edges, hubs of degree 37,000
        {"name": "cl_large", "op": "full", "graph": "cl", "n": 2_000_000, "m": 20_000_000, "L": 5, "k": 4,
         "gamma": 2.1, "wmax": 5.0e4, "zipf": 1.2, "shuffle": False},
        # no hubs, few triangles, the largest edge count
        {"name": "sbm_typed", "op": "full", "graph": "sbm", "n": 1_000_000, "m": 30_000_000, "L": 4, "k": 4},
        # 3-node counts alone on a large graph
        {"name": "k3_large", "op": "full", "graph": "cl", "n": 1_000_000, "m": 10_000_000, "L": 5, "k": 3,
         "gamma": 2.1, "wmax": 3.2e4, "zipf": 1.2, "shuffle": False},
        # many small graphs at once (ego networks: 100 to 400,000 edges, dense)
        {"name": "ego_batch", "op": "batch", "graph": "cl", "n": 0, "m": 400_000, "m_min": 100, "graphs": 256, "L": 6,
         "k": 4, "gamma": 2.3, "wmax": 2.0e3, "zipf": 0.0, "shuffle": True},
        # position-aware counts: longer rows, more classes
        {"name": "position_aware", "op": "pa", "graph": "cl", "n": 200_000, "m": 2_000_000, "L": 5, "k": 4,
         "gamma": 2.1, "wmax": 1.2e4, "zipf": 1.2, "shuffle": True},
        # directed and edge-typed 3-node counts
        {"name": "directed", "op": "dir", "graph": "cl", "n": 500_000, "m": 5_000_000, "L": 5, "k": 3,
         "gamma": 2.1, "wmax": 2.1e4, "zipf": 1.2, "shuffle": False},
        {"name": "edge_typed", "op": "et", "graph": "cl", "n": 500_000, "m": 5_000_000, "L": 5, "k": 3, "X": 4,
         "gamma": 2.1, "wmax": 2.1e4, "zipf": 1.2, "shuffle": False},
        # end to end from and to host memory
        {"name": "host_mid", "op": "host", "graph": "cl", "n": 100_000, "m": 1_000_000, "L": 5, "k": 4,
         "gamma": 2.1, "wmax": 7.8e3, "zipf": 1.2, "shuffle": False},
    ]


def draw(rng):
    op = rng.choice(["full", "full", "full", "count", "count", "host", "batch", "pa", "dir", "et"])
    graph = rng.choice(["cl", "cl", "cl", "sbm", "er"]) if op not in ("batch", "pa") else "cl"
    top = {"full": 1.0e7, "count": 4.0e6, "host": 1.0e6, "batch": 4.0e5, "pa": 2.0e6, "dir": 1.0e7, "et": 1.0e7}[op]
    m = int(math.exp(rng.uniform(math.log(2.0e4), math.log(top))))
    c = {"op": op, "graph": graph, "n": max(int(m / math.exp(rng.uniform(math.log(5.0), math.log(30.0)))), 400), "m": m,
         "L": rng.randint(3, 8), "k": 3 if op in ("dir", "et") or (op in ("full", "count") and rng.random() < 0.2) else 4}
    if graph == "sbm":
        c["L"] = rng.randint(2, 6)
    if graph == "cl":
        c["gamma"] = round(rng.uniform(2.1, 2.5), 2)
        c["wmax"] = round(min(5.0e4 * (m / 2.0e7) ** 0.62 * rng.uniform(0.5, 1.0), c["n"] / 8), 1)
        c["zipf"] = rng.choice([0.0, 1.2])
        c["shuffle"] = rng.random() < 0.5
    if op == "batch":
        c.update(n=0, m_min=100, graphs=rng.randint(16, 300))
    if op == "et":
        c["X"] = rng.randint(1, 4)
    return c


# ---------------------------------------------------------------- inputs

def _blocks(case):
    """(nodes, edges) of every graph of the case."""
    if case["op"] != "batch":
        return [(case["n"], case["m"])]
    lo, hi, c = case["m_min"], case["m"], case["graphs"]
    ms = [int(lo * (hi / lo) ** ((g + 0.5) / c)) for g in range(c)]
    return [(max(m // 16, int(4 * math.sqrt(m))), m) for m in ms]


def _weights(n, m, gamma, wmax):
    """Chung-Lu weights (i + i0)^-a scaled to sum 2m, i0 such that the largest is about wmax."""
    a = 1.0 / (gamma - 1.0)
    i = np.arange(n, dtype=np.float64)
    lo, hi = 1e-3, float(max(n, 2))
    for _ in range(40):
        i0 = math.sqrt(lo * hi)
        w = (i + i0) ** -a
        if w[0] * 2 * m / w.sum() > wmax:
            lo = i0
        else:
            hi = i0
    return (i + i0) ** -a


def _edges(case, gen):
    """Distinct undirected edges u < v as sorted keys u * n + v, the node types and the graphs' node offsets."""
    blocks, kind, L = _blocks(case), case["graph"], case["L"]
    off = np.concatenate([[0], np.cumsum([b[0] for b in blocks])])
    n, m = int(off[-1]), sum(b[1] for b in blocks)
    rand = lambda k: torch.rand(k, generator=gen, device="cuda", dtype=torch.float64)  # noqa: E731
    if kind == "sbm":
        share = np.array([1.0 / (1 << min(b, 4)) for b in range(L)])
        cut = torch.as_tensor(np.round(np.cumsum(share / share.sum()) * n)[:-1], dtype=torch.int64, device="cuda")
        types = torch.searchsorted(cut, torch.arange(n, device="cuda"), right=True).to(torch.uint8)
    else:
        z = np.arange(1, L + 1, dtype=np.float64) ** -case.get("zipf", 0.0)
        cut = torch.as_tensor(np.cumsum(z / z.sum())[:-1], device="cuda")
        types = torch.searchsorted(cut, rand(n), right=True).to(torch.uint8)
    offs, want = torch.as_tensor(off, device="cuda"), torch.as_tensor([b[1] for b in blocks], device="cuda")
    if kind == "cl":
        # graph g takes its endpoints from the g-th unit of the concatenated distribution
        cdf = []
        for g, (nb, mb) in enumerate(blocks):
            w = np.cumsum(_weights(nb, mb, case["gamma"], min(case["wmax"], nb / 4)))
            cdf.append(g + w / w[-1])
        cdf = torch.as_tensor(np.concatenate(cdf), device="cuda")
        which = torch.repeat_interleave(torch.arange(len(blocks), device="cuda"), want).double()
        of_node = torch.searchsorted(offs, torch.arange(n, device="cuda"), right=True)
        perm = torch.argsort(rand(n) + of_node) if case["shuffle"] else torch.arange(n, device="cuda")
    keys = torch.empty(0, dtype=torch.int64, device="cuda")
    for _ in range(24):
        if kind == "cl":
            u, v = (perm[torch.searchsorted(cdf, rand(m) * (1 - 1e-12) + which, right=True).clamp_(max=n - 1)]
                    for _ in range(2))
        else:
            u, v = (torch.randint(0, n, (m,), generator=gen, device="cuda") for _ in range(2))
            if kind == "sbm":
                ok = (types[u] != types[v]) | (rand(m) < 0.05)
                u, v = u[ok], v[ok]
        new = (torch.minimum(u, v) * n + torch.maximum(u, v))[u != v]
        keys = torch.unique(torch.cat([keys, new]))
        have = torch.diff(torch.searchsorted(keys, offs * n))        # keys of graph g lie in its nodes' range
        if bool((have >= want).all()):
            break
    # exactly m_g edges of every graph, at random
    of_key = torch.repeat_interleave(torch.arange(len(blocks), device="cuda"), have)
    order = torch.argsort(rand(keys.numel()) + of_key)               # grouped by graph
    place = torch.arange(keys.numel(), device="cuda") - (torch.cumsum(have, 0) - have)[of_key]
    keys = torch.sort(keys[order[place < want[of_key]]])[0]
    return keys, n, types, off


def _csr(src, dst, n, extra=None):
    key, at = torch.sort(src * n + dst)
    rp = torch.searchsorted(key, torch.arange(n + 1, device="cuda") * n)
    return rp, (key % n).to(torch.int32), None if extra is None else extra[at].contiguous()


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    keys, n, types, off = _edges(case, gen)
    u, v = keys // n, keys % n
    m, L, k, op = keys.numel(), case["L"], case["k"], case["op"]
    s = {"op": op, "L": L, "k": k, "X": case.get("X", 0), "types": types}
    graphs = len(off) - 1
    if op == "dir":
        flip = torch.rand(m, generator=gen, device="cuda") < 0.5
        s["rp"], s["col"], _ = _csr(torch.where(flip, v, u), torch.where(flip, u, v), n)
        lay = tg.tg_directed_layout(L)
    else:
        xi = torch.randint(0, case["X"], (m,), generator=gen, device="cuda", dtype=torch.uint8) if op == "et" else None
        s["rp"], s["col"], s["xi"] = _csr(torch.cat([u, v]), torch.cat([v, u]), n,
                                          None if xi is None else torch.cat([xi, xi]))
        lay = (tg.tg_edge_typed_layout(L, case["X"]) if op == "et" else tg.tg_pa_layout(L) if op == "pa"
               else tg.tg_layout(L, k))
    where = {"device": "cuda"}
    if op == "host":
        for name in ("rp", "col", "types"):
            s[name] = s[name].cpu().pin_memory()
        where = {"pin_memory": True}
    s["rows"] = torch.empty((m, lay["per_edge_slots"]), dtype=torch.int32, **where)
    s["totals"] = torch.empty((graphs, lay["global_slots"]), dtype=torch.int64, **where)
    if op in ("count", "pa"):
        s["handle"] = tg.tg_build(s["rp"], s["col"], types, L)
    if op == "batch":
        s["stream"] = torch.cuda.Stream()                            # a capture needs a stream of its own
        s["stream"].wait_stream(torch.cuda.current_stream())
        s["handle"] = tg.tg_build_batch(off, s["rp"], s["col"], types, L, stream=s["stream"])
    return s


def run(s):
    op, rows, totals = s["op"], s["rows"], s["totals"]
    if op == "count":
        tg.tg_count(s["handle"], s["k"], rows, totals)
    elif op == "pa":
        tg.tg_count_position_aware(s["handle"], rows, totals)
    elif op == "batch":
        tg.tg_count_batch(s["handle"], s["k"], rows, totals, stream=s["stream"])
        torch.cuda.current_stream().wait_stream(s["stream"])
    else:
        if op == "dir":
            h = tg.tg_build_directed(s["rp"], s["col"], s["types"], s["L"])
            tg.tg_count_directed3(h, rows, totals)
        elif op == "et":
            h = tg.tg_build_edge_typed(s["rp"], s["col"], s["types"], s["xi"], s["L"], s["X"])
            tg.tg_count_edge_typed3(h, rows, totals)
        else:
            h = tg.tg_build(s["rp"], s["col"], s["types"], s["L"])
            tg.tg_count(h, s["k"], rows, totals)
        h.free()
    return {"rows": rows, "totals": totals}


def work(case):
    """The CSR and the types read once, every row and total written once (a kept handle: its CSR)."""
    blocks, op, L, k = _blocks(case), case["op"], case["L"], case["k"]
    n, m = sum(b[0] for b in blocks), sum(b[1] for b in blocks)
    lay = (tg.tg_directed_layout(L) if op == "dir" else tg.tg_edge_typed_layout(L, case["X"]) if op == "et"
           else tg.tg_pa_layout(L) if op == "pa" else tg.tg_layout(L, k))
    entries = m if op == "dir" else 2 * m
    return {"bytes": 8 * (n + 1) + n + (5 if op == "et" else 4) * entries + 4 * m * lay["per_edge_slots"]
            + 8 * len(blocks) * lay["global_slots"], "flops": 0}


# ---------------------------------------------------------------- the counts from their definitions

def exact(case, seed):
    """Rows and totals by dense 64-bit products of the indicator matrices of the sets T, S_i, S_j and I of every edge
    (undirected counts of graphs of up to 3,000 nodes)."""
    if case["op"] not in ("full", "count", "host") or case["n"] > 3000 or case["n"] * case["m"] > 4.0e7:
        return None
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    keys, n, types, _ = _edges(case, gen)
    i, j, L, m = keys // n, keys % n, case["L"], keys.numel()
    A = torch.zeros((n, n), dtype=torch.float64, device="cuda")
    A[i, j] = A[j, i] = 1.0
    ends = torch.zeros((m, n), dtype=torch.float64, device="cuda")
    ends[torch.arange(m, device="cuda"), i] = ends[torch.arange(m, device="cuda"), j] = 1.0
    gi, gj = A[i] * (1 - ends), A[j] * (1 - ends)
    T, Si, Sj, I = gi * gj, gi * (1 - gj), gj * (1 - gi), (1 - gi) * (1 - gj) * (1 - ends)
    onehot = torch.nn.functional.one_hot(types.long(), L).double()   # n x L

    def pairs(X, Y):
        """[e, t, t']: all pairs of X^t and Y^t', and the adjacent ones."""
        adj = torch.stack([(X * ((Y * onehot[:, q]) @ A)) @ onehot for q in range(L)], dim=2)
        return (X @ onehot)[:, :, None] * (Y @ onehot)[:, None, :], adj

    def inside(X):
        """The same of distinct nodes of one set, either order."""
        every, adj = pairs(X, X)
        return every - torch.diag_embed(X @ onehot), adj

    def both(M):                                                     # two different sets, either order
        return M + M.transpose(1, 2)

    rows = [Si @ onehot + Sj @ onehot, T @ onehot]
    if case["k"] == 4:
        (ii, iia), (jj, jja), (tt, tta) = inside(Si), inside(Sj), inside(T)
        ij, ija = pairs(Si, Sj)
        ts, tsa = (x + y for x, y in zip(pairs(T, Si), pairs(T, Sj)))
        orbits = [both(pairs(Si, I)[1] + pairs(Sj, I)[1]), both(ij - ija), ii - iia + jj - jja, both(ija), iia + jja,
                  both(pairs(T, I)[1]), both(ts - tsa), both(tsa), tt - tta, tta]
        a, b = torch.triu_indices(L, L, device="cuda")
        rows += [M[:, a, b] * torch.where(a == b, 0.5, 1.0) for M in orbits]
    p, q, third = types[i].long(), types[j].long(), torch.arange(L, device="cuda")
    totals = [_by_types(L, [p, q], torch.ones(m, dtype=torch.float64, device="cuda"))]
    totals += [_by_types(L, [p[:, None], q[:, None], third], rows[o]) / e for o, e in ((0, 2), (1, 3))]
    if case["k"] == 4:
        for of, e in (((2, 3), 3), ((4,), 3), ((5,), 4), ((6, 7, 8), 4), ((9, 10), 5), ((11,), 6)):
            totals.append(_by_types(L, [p[:, None], q[:, None], a, b], sum(rows[o] for o in of)) / e)
    return {"rows": torch.cat(rows, dim=1).round().to(torch.int32),
            "totals": torch.cat(totals).round().to(torch.int64)[None]}


def _by_types(L, types, values):
    """`values` summed by the multiset of their nodes' types, in lexicographic order."""
    sets = list(itertools.combinations_with_replacement(range(L), len(types)))
    rank = torch.zeros(L ** len(types), dtype=torch.int64)
    for r, x in enumerate(sets):
        for y in itertools.permutations(x):
            rank[sum(t * L ** at for at, t in enumerate(y))] = r
    code = sum(t * L ** at for at, t in enumerate(types)).expand(values.shape)
    return torch.bincount(rank.cuda()[code.reshape(-1)], weights=values.reshape(-1), minlength=len(sets))
