"""The calls of this library whose time matters, from the smallest to the largest.

Each case is one use of the public entry points (paper_1804_08487_gb300.cb):
a resident chain that is stepped and read, a graph randomised from its CSR to
its edge list, an ensemble of chains in one handle, the serving loop, uniform
single trades, the paper's two measurements, and the permutation alone.  Sizes
and degree laws are those of the paper's experiments as this repository runs
them (PLD([a,b), gamma) degrees, n from 2^10 to 2^25).

Every output is a whole number (node ids, counts), so all of them are exact.
"""
import functools
import math
import random

import numpy as np
import torch

from paper_1804_08487_gb300 import cb, synth

# Above this size input graphs come from a random pairing built on the GPU:
# Havel-Hakimi on the host takes seconds per graph there.
HOST_GRAPH_NODES = 1 << 20


# ------------------------------------------------------------------- the cases

def listed():
    return [
        # one super step's permutation for a host framework that owns every
        # allocation: the smallest call, a handful of launches
        {"name": "permutation n=4096", "kind": "permutation", "n": 4096},
        # a small resident graph, ten super steps, its edges read: launch-bound
        {"name": "chain n=4096", "kind": "chain", "n": 4096, "a": 10, "b": 100, "gamma": 2.0, "steps": 10,
         "relaxed": False, "cuda_graph": False},
        # the ordinary null-model sample: a graph of a million nodes, twenty
        # super steps, its edges read
        {"name": "chain n=2^20", "kind": "chain", "n": 1 << 20, "a": 10, "b": 1000, "gamma": 2.0, "steps": 20,
         "relaxed": False, "cuda_graph": False},
        # hubs of n/20 neighbours (the swap experiment's law), odd n, relaxed
        # permutations, replayed as a CUDA graph
        {"name": "chain hubs n=300007", "kind": "chain", "n": 300007, "a": 10, "b": 300007 // 20, "gamma": 2.0,
         "steps": 5, "relaxed": True, "cuda_graph": True},
        # a graph that a program holds in host memory, randomised whole:
        # import, validation, super steps, canonical edges back in host memory
        {"name": "randomise host n=2^17", "kind": "randomise", "n": 1 << 17, "a": 10, "b": 1000, "gamma": 2.0,
         "steps": 10, "host": True},
        # the largest graph (about 1.1e9 edges) from a device CSR to its
        # randomised edge list
        {"name": "randomise n=2^25", "kind": "randomise", "n": 1 << 25, "a": 10, "b": 10000, "gamma": 2.0,
         "steps": 5, "host": False},
        # an ensemble of uneven graphs in one handle, one graph launch per step
        {"name": "ensemble 256", "kind": "ensemble", "count": 256, "n_min": 1 << 10, "n_max": 1 << 16,
         "steps": 50},
        # a burst of requests of different sizes through the serving loop
        {"name": "serving 24", "kind": "serving", "count": 24, "n_min": 1 << 12, "n_max": 1 << 18},
        # as many uniform single trades as one global trade has
        {"name": "uniform n=2^20", "kind": "uniform", "n": 1 << 20, "a": 10, "b": 1000, "gamma": 2.0},
        # the swap-fraction experiment on a regular graph: one global trade
        # and n/2 uniform trades, both counted
        {"name": "swaps 10-regular n=2^16", "kind": "swaps", "n": 1 << 16, "degree": 10},
        # the mixing experiment: eight recorded chains, then the autocorrelation
        {"name": "autocorrelation 8 x 2000", "kind": "autocorr", "count": 8, "n": 2000, "a": 5, "b": 25,
         "steps": 300, "kmax": 32},
    ]


def _log_uniform(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["permutation", "chain", "chain", "chain", "randomise", "randomise", "ensemble", "serving",
                       "uniform", "swaps", "autocorr"])
    if kind == "permutation":
        return {"kind": kind, "n": _log_uniform(rng, 2, 1 << 20)}
    if kind in ("chain", "randomise", "uniform"):
        host = rng.random() < 0.5
        top = {"chain": 1 << 20, "randomise": 1 << 20 if host else 1 << 24, "uniform": 1 << 19}[kind]
        n = _log_uniform(rng, 1 << 10, top)
        a = rng.choice([4, 5, 10])
        # the paper's laws: a fixed largest degree, or one that grows with n
        b = max(a + 2, min(n // 4, rng.choice([100, 1000, n // 16 + 1, n // 20]), 20000))
        case = {"kind": kind, "n": n, "a": a, "b": b, "gamma": round(rng.uniform(2.0, 3.0), 2)}
        if kind == "chain":
            case.update(steps=rng.randint(1, 20), relaxed=rng.random() < 0.25, cuda_graph=rng.random() < 0.5)
        elif kind == "randomise":
            case.update(steps=rng.randint(1, 10), host=host)
        return case
    if kind == "ensemble":
        return {"kind": kind, "count": _log_uniform(rng, 2, 256), "n_min": 1 << rng.randint(8, 10),
                "n_max": _log_uniform(rng, 1 << 11, 1 << 16), "steps": rng.randint(5, 50)}
    if kind == "serving":
        return {"kind": kind, "count": rng.randint(2, 24), "n_min": 1 << 12,
                "n_max": _log_uniform(rng, 1 << 13, 1 << 18)}
    if kind == "swaps":
        return {"kind": kind, "n": 2 * _log_uniform(rng, 1 << 9, 1 << 16), "degree": rng.choice([4, 10, 16])}
    n = rng.randint(200, 2000)
    return {"kind": kind, "count": rng.randint(1, 8), "n": n, "a": 5, "b": rng.choice([25, n // 4]),
            "steps": rng.randint(20, 300), "kmax": rng.choice([8, 32])}


# ------------------------------------------------------------------- the inputs

def _pairing_graph(n, a, b, gamma, seed):
    """(row_ptr, col) on the GPU: endpoints drawn in proportion to PLD([a,b),
    gamma) weights, loops and repeated edges dropped, 9/10 of the weights'
    edges kept; rows ascending."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    k = torch.arange(a, b, dtype=torch.float64, device="cuda")
    cdf = torch.cumsum(k ** -gamma, 0)
    u = (torch.randperm(n, device="cuda", generator=gen).double() + 0.5) / n * cdf[-1]
    ends = torch.cumsum(a + torch.searchsorted(cdf, u, right=True).clamp_(max=b - a - 1), 0)
    total = int(ends[-1])
    m = int(0.45 * total)
    del u
    key = torch.empty(0, dtype=torch.int64, device="cuda")
    want = total // 2
    while key.numel() < m:
        parts = [key]
        for lo in range(0, want, 1 << 28):
            c = min(1 << 28, want - lo)
            x = torch.searchsorted(ends, torch.randint(total, (c,), device="cuda", generator=gen), right=True)
            y = torch.searchsorted(ends, torch.randint(total, (c,), device="cuda", generator=gen), right=True)
            pair = torch.minimum(x, y) * n + torch.maximum(x, y)
            parts.append(pair[x != y])
        key = torch.unique_consecutive(torch.sort(torch.cat(parts)).values)
        want = total // 16
    del parts, pair, x, y, ends
    spare = key.numel() - m   # dropped at even distances
    if spare:
        keep = torch.ones(key.numel(), dtype=torch.bool, device="cuda")
        keep[torch.arange(spare, device="cuda") * key.numel() // spare] = False
        key = key[keep]
        del keep
    up_row, up_col = key // n, (key % n).to(torch.int32)
    up_deg = torch.bincount(up_row, minlength=n)
    key = torch.sort(key % n * n + up_row).values
    low_row, low_col = key // n, (key % n).to(torch.int32)
    del key
    low_deg = torch.bincount(low_row, minlength=n)
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(up_deg + low_deg, 0, out=row_ptr[1:])
    up0, low0 = torch.cumsum(up_deg, 0) - up_deg, torch.cumsum(low_deg, 0) - low_deg
    col = torch.empty(2 * m, dtype=torch.int32, device="cuda")
    # every row holds its entries below the diagonal, then those above; filled
    # in row ranges of about 2^29 entries
    cuts = torch.searchsorted(row_ptr, torch.arange(0, 2 * m + (1 << 29), 1 << 29, device="cuda")).clamp_(max=n)
    cuts = sorted(set([0] + cuts.tolist() + [n]))
    for r0, r1 in zip(cuts, cuts[1:]):
        e0, e1 = int(row_ptr[r0]), int(row_ptr[r1])
        view = col[e0:e1]
        for row, val, first, skip in ((low_row, low_col, low0, None), (up_row, up_col, up0, low_deg)):
            i0 = int(first[r0])
            i1 = int(first[r1]) if r1 < n else m
            r = row[i0:i1]
            at = torch.arange(i0, i1, device="cuda") - first[r] + row_ptr[r] - e0
            if skip is not None:
                at += skip[r]
            view[at] = val[i0:i1]
    del up_row, up_col, low_row, low_col, r, at
    torch.cuda.empty_cache()   # the library allocates from a pool of its own
    return row_ptr, col


@functools.lru_cache(maxsize=300)
def _havel_hakimi(n, a, b, gamma, degree_seed):
    g = synth.powerlaw_graph(n, a, b, gamma, degree_seed)
    return torch.from_numpy(g.row_ptr), torch.from_numpy(g.col)


def _relabelled_graph(n, a, b, gamma, seed, degree_seed=1):
    """(row_ptr, col) on the GPU: a Havel-Hakimi realisation of PLD([a,b),
    gamma) degrees under node labels drawn from the seed; rows ascending."""
    row_ptr, col = (t.cuda() for t in _havel_hakimi(n, a, b, gamma, degree_seed))
    gen = torch.Generator(device="cuda").manual_seed(seed)
    label = torch.randperm(n, device="cuda", generator=gen)
    deg = row_ptr[1:] - row_ptr[:-1]
    row = torch.repeat_interleave(label, deg, output_size=col.numel())
    key = torch.sort(row * n + label[col.long()]).values
    new_deg = torch.empty_like(deg)
    new_deg[label] = deg
    new_ptr = torch.zeros_like(row_ptr)
    torch.cumsum(new_deg, 0, out=new_ptr[1:])
    return new_ptr, (key % n).to(torch.int32)


def _graph(law, seed, host, degree_seed=1):
    """A graph of the law (n, a, b, gamma) as CSR, in host memory (numpy) or on the GPU (torch)."""
    if law[0] > HOST_GRAPH_NODES:
        row_ptr, col = _pairing_graph(*law, seed)
    else:
        row_ptr, col = _relabelled_graph(*law, seed, degree_seed)
    return (row_ptr.cpu().numpy(), col.cpu().numpy()) if host else (row_ptr, col)


def _members(case):
    """(law, steps, degree seed) of every member of an ensemble or a burst of
    requests: PLD([4, n/16), gamma in [2, 3]), as the case has it for any seed."""
    rng = random.Random(case["count"])
    for i in range(case["count"]):
        n = _log_uniform(rng, case["n_min"], case["n_max"])
        yield (n, 4, max(n // 16, 6), rng.uniform(2.0, 3.0)), rng.randint(5, 20), 1000 + i


def _law(case):
    return case["n"], case["a"], case["b"], case.get("gamma", 2.0)


def prepare(case, seed):
    kind = case["kind"]
    state = dict(case, seed=seed)
    if kind == "permutation":
        state["order"] = torch.empty(case["n"], dtype=torch.int32, device="cuda")
    elif kind == "randomise":
        state["graph"] = _graph(_law(case), seed, case["host"])
        m = len(state["graph"][1]) // 2
        state["edges"] = (np.empty((m, 2), dtype=np.int32) if case["host"]
                          else torch.empty((m, 2), dtype=torch.int32, device="cuda"))
    elif kind == "serving":
        state["requests"] = [_graph(law, seed + i, True, ds) + (seed + i, steps)
                             for i, (law, steps, ds) in enumerate(_members(case))]
        state["server"] = cb.Server(120 * 10**9, max_active=64, depth=2)
    else:
        if kind == "ensemble":
            graphs = [_graph(law, seed + i, True, ds) for i, (law, _, ds) in enumerate(_members(case))]
            chain = cb.Ensemble(graphs, [seed + i for i in range(len(graphs))])
            chain.set_option("cuda_graph", 1)
        elif kind == "autocorr":
            graphs = [_graph(_law(case), seed + i, True) for i in range(case["count"])]
            chain = cb.Ensemble(graphs, [seed + i for i in range(len(graphs))])
        elif kind == "swaps":
            graphs = [_graph((case["n"], case["degree"], case["degree"] + 1, 2.0), seed, True)]
            chain = cb.Curveball(*graphs[0], seed=seed)
            chain.global_trades(10)   # away from the structured start, as the experiment does
            chain.set_option("swap_stats", 1)
        else:
            graphs = [_graph(_law(case), seed, True)]
            chain = cb.Curveball(*graphs[0], seed=seed)
            if case.get("relaxed"):
                chain.set_option("relaxed", 1)
            if case.get("cuda_graph"):
                chain.set_option("cuda_graph", 1)
        state["chain"] = chain
        m = sum(len(col) for _, col in graphs) // 2
        state["edges"] = torch.empty((m, 2), dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    return state


# --------------------------------------------------------------------- one pass

def run(state):
    kind = state["kind"]
    if kind == "permutation":
        cb.cb_permutation_static(state["n"], state["seed"], 0, state["order"])
        return state["order"]
    if kind == "randomise":
        row_ptr, col = state["graph"]
        chain = cb.Curveball(row_ptr, col, state["seed"])
        chain.global_trades(state["steps"])
        chain.edges(state["edges"])
        chain.close()
        return state["edges"]
    if kind == "serving":
        server = state["server"]
        ids = [server.submit(*request) for request in state["requests"]]
        results = {}
        while len(results) < len(ids):
            for done in server.poll(timeout_ms=1000):
                results[done] = server.result(done)[0]
        return [results[i] for i in ids]
    chain = state["chain"]
    if kind == "uniform":
        chain.uniform_trades(state["n"] // 2)
        return chain.edges(state["edges"])
    if kind == "swaps":
        chain.global_trades(1)
        after_global = chain.swap_counts()
        chain.uniform_trades(state["n"] // 2)
        return [after_global, chain.swap_counts(), chain.edges(state["edges"])]
    if kind == "autocorr":
        chain.set_option("presence", state["steps"])
        chain.global_trades(state["steps"])
        correlated, near_ties, occurring, states = chain.autocorr(state["kmax"])
        return [np.array(correlated), np.array(near_ties), occurring, states, chain.edges(state["edges"])]
    chain.global_trades(state["steps"])
    return chain.edges(state["edges"])


# --------------------------------------------------------------- what it cannot do without

def _mean_degree(a, b, gamma):
    k = np.arange(a, b, dtype=np.float64)
    w = k ** -gamma
    return float((k * w).sum() / w.sum())


def _step_bytes(n, m):
    """One super step: every directed entry read and written once, the nodes'
    keys, order and positions (24 bytes a node)."""
    return 16 * m + 24 * n


def work(case):
    kind = case["kind"]
    if kind == "permutation":
        total = 4 * case["n"]
    elif kind in ("ensemble", "serving"):
        # expected over the members: n log-uniform, gamma uniform in [2, 3]
        lo, hi = math.log(case["n_min"]), math.log(case["n_max"])
        total = 0.0
        for i in range(16):
            n = math.exp(lo + (hi - lo) * (i + 0.5) / 16)
            m = n * sum(_mean_degree(4, max(int(n) // 16, 6), g) for g in (2.125, 2.375, 2.625, 2.875)) / 8
            steps = case.get("steps", 12.5)
            total += case["count"] / 16 * (steps * _step_bytes(n, m) + 8 * m)
            if kind == "serving":   # the request's graph comes in
                total += case["count"] / 16 * (8 * m + 8 * n)
    elif kind == "swaps":
        n, m = case["n"], case["n"] * case["degree"] / 2
        total = 2 * _step_bytes(n, m) + 8 * m
    elif kind == "autocorr":
        n, m = case["n"], case["n"] * _mean_degree(case["a"], case["b"], 2.0) / 2
        pairs = n * (n - 1) / 2
        total = case["count"] * (case["steps"] * _step_bytes(n, m) + pairs * case["steps"] / 8 + 8 * m)
    else:
        n, m = case["n"], case["n"] * _mean_degree(case["a"], case["b"], case["gamma"]) / 2
        total = case.get("steps", 1) * _step_bytes(n, m) + 8 * m
        if kind == "randomise":   # the graph comes in
            total += 8 * m + 8 * n
    return {"bytes": float(total), "flops": 0.0}


# ------------------------------------------------------------------------ exact

def _permutation(n, seed, g):
    """Nodes in order of (key, node), the key being the first 64 bits of
    Philox4x32-10 on counter (node, 0, g, 0)."""
    mask = np.uint64(0xFFFFFFFF)
    c = [np.arange(n, dtype=np.uint64), np.zeros(n, np.uint64), np.full(n, g, np.uint64), np.zeros(n, np.uint64)]
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    for _ in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & mask,
             (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), p0 & mask]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return np.argsort((c[0] << np.uint64(32)) | c[1], kind="stable").astype(np.int32)


def exact(case, seed):
    """The permutation as numpy sorts it.  The other cases' outputs are node
    ids and counts, with no value in floating point to be near to."""
    if case["kind"] == "permutation":
        return _permutation(case["n"], seed, 0)
    return None
