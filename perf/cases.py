"""What is measured: calls that a user of this framework makes, through its
public entry points, over the sizes they are made at.

A case is a dict of plain values; ``listed()`` names the fixed ones, ``draw``
makes more of the same ranges, ``prepare`` makes the inputs and the handle a
program holds, ``run`` is one call.  Every output is a whole number (counts,
randomised targets) or a Z-score.
"""
import math

import numpy as np
import torch

import paper_1203_3415_gb300 as acc

DEV = "cuda:0"
MODES = {"count": acc.ACC_MODE_COUNT, "auto": acc.ACC_MODE_AUTO}
RANDOMISE = {"swap": acc.ACC_RAND_SWAP, "mutual": acc.ACC_RAND_MUTUAL}


def listed():
    return [
        # the smallest use: the motifs of a small random graph, one call after
        # another (launches and latency)
        {"name": "k3_er_1000", "kind": "count", "graph": "er", "n": 1000, "m": 5000, "cap": 0, "k": 3,
         "mode": "auto", "call": "enqueue"},
        # k = 3 on a large scale-free graph with hubs, default mode
        {"name": "k3_chung_lu_50000", "kind": "count", "graph": "chung_lu", "n": 50000, "m": 250000, "cap": 500,
         "k": 3, "mode": "count", "call": "enqueue"},
        # the plainest call on a small graph: counts returned, errors raised, the call waits
        {"name": "k4_call_400", "kind": "count", "graph": "chung_lu", "n": 400, "m": 1600, "cap": 60, "k": 4,
         "mode": "count", "call": "wait"},
        # the headline: k = 4 on a scale-free graph of 20000 vertices
        {"name": "k4_chung_lu_20000", "kind": "count", "graph": "chung_lu", "n": 20000, "m": 100000, "cap": 500,
         "k": 4, "mode": "auto", "call": "enqueue"},
        # a graph held in host memory, copied in and counts copied out by the call
        {"name": "k4_host_5000", "kind": "count", "graph": "chung_lu", "n": 5000, "m": 20000, "cap": 200, "k": 4,
         "mode": "auto", "call": "host"},
        # a graph above the dense adjacency limit: sorted raw rows and hashed adjacency
        {"name": "k4_chung_lu_1000000", "kind": "count", "graph": "chung_lu", "n": 1000000, "m": 3000000,
         "cap": 500, "k": 4, "mode": "count", "call": "enqueue"},
        # k = 5 on a sparse regulatory network (out-hubs)
        {"name": "k5_regulatory_5000", "kind": "count", "graph": "regulatory", "n": 5000, "m": 15000, "cap": 200,
         "k": 5, "mode": "auto", "call": "enqueue"},
        # k = 5 on a small dense graph (the shape of the paper's Facebook row)
        {"name": "k5_chung_lu_1899", "kind": "count", "graph": "chung_lu", "n": 1899, "m": 20296, "cap": 200,
         "k": 5, "mode": "auto", "call": "enqueue"},
        # k = 5 on a graph large enough for the hashed adjacency
        {"name": "k5_chung_lu_60000", "kind": "count", "graph": "chung_lu", "n": 60000, "m": 180000, "cap": 60,
         "k": 5, "mode": "count", "call": "enqueue"},
        # the batch of a significance study: 8 graphs and 500 copies of each, prepared once
        {"name": "batch_k4_4008", "kind": "batch", "k": 4, "graphs": 8, "copies": 500, "n_lo": 500, "n_hi": 5000,
         "degree": 4},
        # one whole significance step: randomise (mutual arcs kept), count, Z-scores
        {"name": "significance_k4_404", "kind": "significance", "k": 4, "graphs": 4, "copies": 100, "n_lo": 500,
         "n_hi": 2000, "degree": 4, "randomise": "mutual"},
        # requests of mixed k on resident graphs, all queued at once and served
        {"name": "serve_64", "kind": "serve", "graphs": 24, "requests": 64, "n_lo": 100, "n_hi": 20000, "slots": 8},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["count3", "count4", "count4", "count5", "count5", "batch", "significance", "serve"])
    if kind == "count3":
        n = _log_int(rng, 50, 1000000)
        if 131072 <= n <= 524288:  # (a dense adjacency block of n^2 / 4 bytes: three states would not fit the card)
            n //= 4
        return {"kind": "count", "graph": rng.choice(["er", "chung_lu", "regulatory"]), "n": n,
                "m": int(n * rng.uniform(1.5, 6.0)), "cap": _log_int(rng, 20, 500), "k": 3,
                "mode": rng.choice(["count", "auto"]), "call": rng.choice(["enqueue", "wait", "host"])}
    if kind == "count4":
        n = _log_int(rng, 100, 1000000)
        if 131072 <= n <= 524288:
            n //= 4
        return {"kind": "count", "graph": rng.choice(["er", "chung_lu", "chung_lu", "regulatory"]), "n": n,
                "m": int(n * rng.uniform(1.5, 3.0 if n > 100000 else 6.0)), "cap": _log_int(rng, 20, 500), "k": 4,
                "mode": rng.choice(["count", "auto"]), "call": rng.choice(["enqueue", "wait", "host"])}
    if kind == "count5":
        n = _log_int(rng, 100, 60000)
        return {"kind": "count", "graph": rng.choice(["er", "chung_lu", "regulatory"]), "n": n,
                "m": int(n * rng.uniform(1.5, 3.0 if n > 10000 else 6.0)),
                "cap": _log_int(rng, 20, 60 if n > 10000 else 200), "k": 5,
                "mode": rng.choice(["count", "auto"]), "call": rng.choice(["enqueue", "wait", "host"])}
    if kind == "batch":
        return {"kind": "batch", "k": rng.choice([3, 4, 4]), "graphs": rng.randint(1, 8),
                "copies": _log_int(rng, 10, 400), "n_lo": rng.randint(60, 700), "n_hi": rng.randint(701, 5000),
                "degree": rng.randint(2, 5)}
    if kind == "significance":
        return {"kind": "significance", "k": rng.choice([3, 4]), "graphs": rng.randint(1, 4),
                "copies": _log_int(rng, 10, 200), "n_lo": rng.randint(60, 500), "n_hi": rng.randint(501, 2500),
                "degree": rng.randint(2, 5), "randomise": rng.choice(["swap", "mutual"])}
    return {"kind": "serve", "graphs": rng.randint(4, 24), "requests": rng.randint(8, 64), "n_lo": 100,
            "n_hi": _log_int(rng, 1000, 20000), "slots": rng.choice([4, 8])}


# --------------------------------------------------------------------------
# inputs: simple directed graphs (numpy, from the seed alone)
# --------------------------------------------------------------------------

def _pareto_weights(rng, n, alpha, cap, total):
    """Pareto weights scaled so that min(c w, cap) sums to about total."""
    w = rng.pareto(alpha, n) + 1.0
    lo, hi = 0.0, float(total)
    for _ in range(60):
        c = 0.5 * (lo + hi)
        if np.minimum(c * w, cap).sum() < total:
            lo = c
        else:
            hi = c
    return np.minimum(hi * w, cap)


def _distinct_pairs(n, need, sample):
    """`need` arcs (src, dst) with distinct unordered pairs, in the order drawn."""
    src, dst = np.zeros(0, np.int64), np.zeros(0, np.int64)
    for attempt in range(200):
        s, d = sample(int((need - len(src)) * 1.3) + 64, attempt)
        keep = s != d
        src, dst = np.concatenate([src, s[keep]]), np.concatenate([dst, d[keep]])
        key = np.minimum(src, dst) * n + np.maximum(src, dst)
        first = np.unique(key, return_index=True)[1]
        first.sort()
        src, dst = src[first], dst[first]
        if len(src) >= need:
            return src[:need], dst[:need]
    raise RuntimeError("graph too dense for its size")


def make_graph(kind, n, m, cap, rng):
    """(rowptr int64[n+1], col int32[m], n) of a simple directed graph: single
    arcs of distinct pairs, then about 10% (regulatory 3%) of the arcs in
    reciprocal pairs.  Rows sorted."""
    m = min(m, n * (n - 1) // 3)
    recip = int(round((0.03 if kind == "regulatory" else 0.10) * m / 2))
    single = m - recip

    def uniform(count):
        return rng.integers(0, n, count), rng.integers(0, n, count)

    if kind == "er":
        def sample(count, attempt):
            return uniform(count)
    elif kind == "chung_lu":
        cap_ = min(cap, max(4, n // 2))
        out = np.cumsum(_pareto_weights(rng, n, 1.2, cap_, m))
        inn = np.cumsum(_pareto_weights(rng, n, 1.2, cap_, m))

        def sample(count, attempt):
            if attempt > 100:  # weights exhausted on a tiny dense graph
                return uniform(count)
            return (np.minimum(np.searchsorted(out, rng.random(count) * out[-1]), n - 1),
                    np.minimum(np.searchsorted(inn, rng.random(count) * inn[-1]), n - 1))
    else:  # regulatory: 5% hubs regulate uniformly drawn targets
        hubs = rng.permutation(n)[:max(1, n // 20)]
        cw = np.cumsum(_pareto_weights(rng, len(hubs), 1.0, cap, m))

        def sample(count, attempt):
            if attempt > 100:
                return uniform(count)
            return hubs[np.minimum(np.searchsorted(cw, rng.random(count) * cw[-1]), len(hubs) - 1)], \
                rng.integers(0, n, count)
    src, dst = _distinct_pairs(n, single, sample)
    back = rng.permutation(single)[:recip]
    src, dst = np.concatenate([src, dst[back]]), np.concatenate([dst, src[back]])
    order = np.argsort(src * n + dst, kind="stable")
    rowptr = np.zeros(n + 1, np.int64)
    np.cumsum(np.bincount(src, minlength=n), out=rowptr[1:])
    return rowptr, dst[order].astype(np.int32), n


def _to_device(g):
    return torch.from_numpy(g[0]).to(DEV), torch.from_numpy(g[1]).to(DEV), g[2]


def _sizes(case):
    """Vertex counts of a case's graphs: log-spaced over [n_lo, n_hi]."""
    g, lo, hi = case["graphs"], case["n_lo"], case["n_hi"]
    return [int(round(math.exp(math.log(lo) + (math.log(hi) - math.log(lo)) * (i + 0.5) / g))) for i in range(g)]


def _base_graphs(case, rng):
    return [make_graph("chung_lu", n, case["degree"] * n, min(500, n // 2), rng) for n in _sizes(case)]


def _serve_specs(case):
    """(n, m) per resident graph and (graph, k) per request; fixed by the case."""
    sizes = [(n, 4 * n + (n * (i % 7)) // 2) for i, n in enumerate(_sizes(case))]
    ks = [3, 3, 4, 3, 5, 4, 3, 4, 3, 3, 4, 3, 3, 4, 5, 4, 3, 4, 3, 3]  # 50% k=3, 35-40% k=4, 10-15% k=5
    return sizes, [((5 * r + 3 * (r // 7)) % len(sizes), ks[r % len(ks)]) for r in range(case["requests"])]


# --------------------------------------------------------------------------
# one case: state, pass, work
# --------------------------------------------------------------------------

def prepare(case, seed):
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    if kind == "count":
        g = make_graph(case["graph"], case["n"], case["m"], case["cap"], rng)
        c = acc.Counter(0)
        c.set_mode(MODES[case["mode"]])
        c.prepare(case["k"])
        st = {"case": case, "counter": c}
        if case["call"] == "host":
            # (pinned arrays, as the header recommends)
            st["graph"] = (torch.from_numpy(g[0]).pin_memory(), torch.from_numpy(g[1]).pin_memory(), g[2])
            st["counts"] = np.zeros(acc.NUM_CLASSES[case["k"]], np.int64)
        else:
            st["graph"] = _to_device(g)
            if case["call"] == "enqueue":
                st["counts"] = torch.zeros(acc.NUM_CLASSES[case["k"]], dtype=torch.int64, device=DEV)
                st["status"] = torch.zeros(1, dtype=torch.int32, device=DEV)
        return st
    if kind == "serve":
        sizes, requests = _serve_specs(case)
        srv = acc.Server(0, case["slots"])
        ids = []
        for n, m in sizes:
            r, c, n = _to_device(make_graph("chung_lu", n, m, 200, rng))
            ids.append(srv.add_graph(r, c, n))
        srv.reserve()
        return {"case": case, "server": srv, "requests": [(ids[g], k) for g, k in requests]}
    bases = [_to_device(g) for g in _base_graphs(case, rng)]
    c = acc.Counter(0)
    c.prepare(case["k"])
    st = {"case": case, "counter": c, "bases": bases, "seeds": [seed * 1000003 + 10 ** 6 * b for b in range(len(bases))]}
    if kind == "batch":
        out, _ = c.randomise(bases, case["copies"], st["seeds"])
        members = []
        for g, copies in zip(bases, acc.Counter.copies(bases, case["copies"], out)):
            members.append(g)
            members.extend(copies)
        st["members"] = members
        c.prepare_batch(members, case["k"])
        st["counts"] = torch.zeros((len(members), acc.NUM_CLASSES[case["k"]]), dtype=torch.int64, device=DEV)
        st["status"] = torch.zeros(1, dtype=torch.int32, device=DEV)
    return st


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "count":
        rowptr, col, n = state["graph"]
        c, k = state["counter"], case["k"]
        if case["call"] == "host":
            return c.count_host(rowptr, col, n, k, counts=state["counts"])
        if case["call"] == "wait":
            return c.count(rowptr, col, n, k)
        c.count(rowptr, col, n, k, counts=state["counts"], status=state["status"])
        return [state["counts"], state["status"]]
    if kind == "batch":
        c = state["counter"]
        c.run_batch(counts=state["counts"], status=state["status"])
        z = c.zscores(state["counts"], case["graphs"], case["copies"] + 1, case["k"])
        return [state["counts"], state["status"], z]
    if kind == "significance":
        return list(state["counter"].significance(state["bases"], case["k"], case["copies"], state["seeds"],
                                                  mode=RANDOMISE[case["randomise"]]))
    srv = state["server"]
    rids = [srv.submit(g, k) for g, k in state["requests"]]
    srv.drain()
    return [srv.poll(rid)[1] for rid in rids]


def work(case):
    """Bytes of one pass: each graph read once (8-byte row offsets, 4-byte
    targets), each output written once.  The operations that the counting
    itself cannot do without depend on the graph and are whole-number ones:
    one look at each end of each arc is what any method needs."""
    kind = case["kind"]
    if kind == "count":
        return {"bytes": 8 * (case["n"] + 1) + 4 * case["m"] + 8 * acc.NUM_CLASSES[case["k"]],
                "flops": 2 * case["m"]}
    if kind == "serve":
        sizes, requests = _serve_specs(case)
        return {"bytes": sum(8 * (sizes[g][0] + 1) + 4 * sizes[g][1] + 8 * acc.NUM_CLASSES[k] for g, k in requests),
                "flops": sum(2 * sizes[g][1] for g, _ in requests)}
    n, members = sum(_sizes(case)), case["copies"] + 1
    m = case["degree"] * n
    out = case["graphs"] * members * 8 * acc.NUM_CLASSES[case["k"]]
    if kind == "batch":
        return {"bytes": (8 * n + 4 * m) * members + out, "flops": 2 * m * members}
    # the copies are written once and read once; three swap attempts an arc
    return {"bytes": 8 * n + 4 * m + 2 * 4 * m * case["copies"] + out, "flops": (2 + 3) * m * members}


# --------------------------------------------------------------------------
# plain values
# --------------------------------------------------------------------------

MAX_SETS = 2000000


def _class_of_codes(k):
    """code -> class (rank of the smallest relabelled code among the weakly
    connected ones), -1 for the others; bit i (k - 1) + j - [j > i] of a code
    is the arc from vertex i to vertex j."""
    from itertools import permutations
    bits = [(i, j) for i in range(k) for j in range(k) if i != j]
    at = {b: x for x, b in enumerate(bits)}
    codes = np.arange(1 << len(bits), dtype=np.int64)
    canon = codes.copy()
    for p in permutations(range(k)):
        moved = np.zeros_like(codes)
        for (i, j), x in at.items():
            moved |= ((codes >> x) & 1) << at[(p[i], p[j])]
        canon = np.minimum(canon, moved)
    reach = np.ones_like(codes)  # vertices reached from vertex 0, as a bit set
    for _ in range(k):
        for (i, j), x in at.items():
            arc = (codes >> x) & 1
            reach |= arc * ((((reach >> i) & 1) << j) | (((reach >> j) & 1) << i))
    connected = reach == (1 << k) - 1
    cls = np.full(len(codes), -1, np.int64)
    cls[connected] = np.unique(canon[connected], return_inverse=True)[1]
    return cls


def _plain_counts(rowptr, col, n, k):
    """Every connected k-set grown from the connected (k-1)-sets by one
    neighbour, each kept once, and classified; None above MAX_SETS."""
    src = np.repeat(np.arange(n, dtype=np.int64), np.diff(rowptr))
    arcs = np.unique(src * n + col)
    und = np.unique(np.concatenate([arcs, (arcs % n) * n + arcs // n]))
    ptr = np.searchsorted(und // n, np.arange(n + 1))
    nbr, deg = und % n, np.diff(ptr)
    sets = np.arange(n, dtype=np.int64)[:, None]
    for size in range(2, k + 1):
        grown = []
        if int(deg[sets].sum()) > 6 * MAX_SETS:
            return None
        for i in range(size - 1):
            d = deg[sets[:, i]]
            rows = np.repeat(np.arange(len(sets)), d)
            pos = np.arange(d.sum()) - np.repeat(np.cumsum(d) - d, d) + np.repeat(ptr[sets[:, i]], d)
            new = nbr[pos]
            ok = (sets[rows] != new[:, None]).all(1)
            grown.append(np.concatenate([sets[rows[ok]], new[ok, None]], 1))
        sets = np.sort(np.concatenate(grown), 1)
        order = np.lexsort(sets.T[::-1])
        sets = sets[order]
        keep = np.ones(len(sets), bool)
        keep[1:] = (sets[1:] != sets[:-1]).any(1)
        sets = sets[keep]
        if len(sets) > MAX_SETS:
            return None
    code = np.zeros(len(sets), np.int64)
    x = 0
    for i in range(k):
        for j in range(k):
            if i != j:
                key = sets[:, i] * n + sets[:, j]
                at = np.minimum(np.searchsorted(arcs, key), max(0, len(arcs) - 1))
                code |= (arcs[at] == key).astype(np.int64) << x
                x += 1
    return np.bincount(_class_of_codes(k)[code], minlength=acc.NUM_CLASSES[k]).astype(np.int64)


def exact(case, seed):
    # counts are whole numbers; given where a plain walk over the subsets is
    # short, None elsewhere (a batch or a large graph has 10^8 and more)
    if case["kind"] != "count" or case["n"] > 20000:
        return None
    g = make_graph(case["graph"], case["n"], case["m"], case["cap"], np.random.default_rng(seed))
    counts = _plain_counts(*g, case["k"])
    if counts is None:
        return None
    return [counts, np.zeros(1, np.int32)] if case["call"] == "enqueue" else counts
