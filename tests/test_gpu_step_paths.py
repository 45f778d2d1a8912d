"""The super step at the edges of its launch rules: the permutation's rescan
and scatter forms, its slow bucket paths, the row offsets that both write, and
the passes over deferred trades for small and large handles.  Whole numbers:
equal to the oracle element by element."""
import numpy as np
import pytest

from oracle import Oracle
from paper_1804_08487_gb300 import synth
from paper_1804_08487_gb300.cb import CB_EINVAL, CbError, Curveball, Ensemble

pytestmark = pytest.mark.gpu


# 2^15 nodes in 64 buckets are the most keys a rescan computes; one more node
# (and every larger size) goes through the scatter.  1024 and 1025: one and two
# buckets.  bucket_cap 2 and 600: buckets above shared memory, in both forms.
@pytest.mark.parametrize("n,options", [
    (2, {}), (511, {}), (1023, {}), (1024, {}), (1025, {}), (32767, {}), (32768, {}), (32769, {}), (65535, {}),
    (65536, {}), (2047, {"bucket_cap": 2}), (40000, {"bucket_cap": 600}), (20000, {"bucket_cap": 600}),
])
def test_permutation_and_rows(n, options):
    g = synth.powerlaw_graph(n, 1, max(2, min(n - 1, 6)), 2.5, n)
    c = Curveball(g.row_ptr, g.col, n)
    o = Oracle(g.row_ptr, g.col, n)
    for k, v in options.items():
        c.set_option(k, v)
    for step in (0, 1, 7):
        assert np.array_equal(c.permutation(step), o.permutation(step).astype(np.int32))
    for _ in range(2):
        c.global_trades(1)
        o.superstep(1)
        assert np.array_equal(c.edges(), o.edges())
    c.close()


@pytest.mark.parametrize("sizes", [(3, 1, 0, 2), (1023, 1024, 1025, 9), (9000, 12001, 700), (40001, 30, 20000)])
@pytest.mark.parametrize("graph", [0, 1])
def test_batches_of_both_permutation_forms(sizes, graph):
    graphs, seeds = [], []
    for i, n in enumerate(sizes):
        if n < 4:
            graphs.append((np.zeros(n + 1, np.int64), np.zeros(0, np.int32)))
        else:
            g = synth.powerlaw_graph(n, 2, min(n // 2, 60), 2.0, n)
            graphs.append((g.row_ptr, g.col))
        seeds.append(50 + i)
    e = Ensemble(graphs, seeds)
    e.set_option("cuda_graph", graph)
    e.global_trades(3)
    for i, (rp, col) in enumerate(graphs):
        o = Oracle(rp, col, seeds[i])
        o.superstep(3)
        assert np.array_equal(e.graph_edges(i), o.edges())
    e.close()


# 2^21 nodes are 2^20 trades: the first size with retry passes; dense cores
# of a few hundred nodes make hundreds of deferred trades.
@pytest.mark.parametrize("n,b", [((1 << 21) - 2, 900), (1 << 21, 900)])
@pytest.mark.parametrize("retry", [0, 2])
def test_deferred_trades_around_the_retry_rule(n, b, retry):
    g = synth.powerlaw_graph(n, 1, b, 2.2, 3)
    c = Curveball(g.row_ptr, g.col, 11)
    c.set_option("retry_passes", retry)
    o = Oracle(g.row_ptr, g.col, 11)
    c.global_trades(1)
    o.superstep(1)
    st = c.stats()
    assert st["deferred"] > 0 and st["inorder_trades"] <= st["deferred"]
    assert np.array_equal(c.edges(), o.edges())
    c.close()


@pytest.mark.parametrize("n,b,options", [
    (400, 200, {}), (3000, 1500, {}), (3000, 1500, {"inorder_threads": 256}), (9000, 4000, {}),
    (9000, 4000, {"inorder_threads": 256, "block_max": 128}), (9000, 4000, {"smem_max": 64}),
])
def test_dense_cores_through_the_in_order_pass(n, b, options):
    g = synth.powerlaw_graph(n, 8, b, 2.0, 17)
    c = Curveball(g.row_ptr, g.col, 5)
    for k, v in options.items():
        c.set_option(k, v)
    o = Oracle(g.row_ptr, g.col, 5)
    for _ in range(3):
        c.global_trades(1)
        o.superstep(1)
        assert np.array_equal(c.edges(), o.edges())
    assert c.stats()["deferred"] > 0
    c.close()


# rows of 32, 33, 256, 257, 1024, 1025 and more entries above the diagonal
# (a warp on its tile, a warp on a listed row, 128 to 1024 threads, a global slice), a star
# whose hub is the first or the last node, and an output buffer that is only
# 4-byte aligned.
@pytest.mark.parametrize("d", [1, 2, 31, 32, 33, 64, 65, 128, 129, 255, 256, 257, 511, 512, 513, 1023, 1024, 1025, 2047, 2048,
                               2049, 4097, 8192, 8193, 16384, 16385, 20000])
@pytest.mark.parametrize("hub_last", [False, True])
def test_export_of_long_rows(d, hub_last):
    import torch
    n = d + 40
    rng = np.random.default_rng(d)
    hub = n - 1 if hub_last else 0
    leaves = np.setdiff1d(rng.permutation(n)[:d + 1], [hub])[:d]
    extra = rng.integers(0, n, (30, 2))
    e = {(min(hub, x), max(hub, x)) for x in leaves.tolist()} | {(min(a, b), max(a, b)) for a, b in extra.tolist() if a != b}
    e = np.array(sorted(e), dtype=np.int64)
    both = np.concatenate([e, e[:, ::-1]])
    both = both[np.lexsort((both[:, 1], both[:, 0]))]
    rp = np.concatenate([[0], np.cumsum(np.bincount(both[:, 0], minlength=n))]).astype(np.int64)
    c = Curveball(rp, both[:, 1].astype(np.int32), 3)
    assert np.array_equal(c.edges(), e)
    c.global_trades(1)
    o = Oracle(rp, both[:, 1].astype(np.int32), 3)
    o.superstep(1)
    buf = torch.zeros(2 * len(e) + 1, dtype=torch.int32, device="cuda")
    c.edges(buf[1:])
    assert np.array_equal(buf[1:].cpu().numpy().reshape(-1, 2), o.edges())
    assert np.array_equal(c.edges(), o.edges())
    c.close()


# one wrong entry in an otherwise symmetric graph of many tiles and buckets:
# an entry moved, repeated, out of range, a self loop, a missing mirror
@pytest.mark.parametrize("n", [40, 5000, 70000])
@pytest.mark.parametrize("what", ["moved", "repeated", "range", "negative", "loop", "mirror"])
@pytest.mark.parametrize("shuffled", [False, True])
def test_malformed_graphs_are_refused(n, what, shuffled):
    g = synth.powerlaw_graph(n, 3, min(n // 3, 200), 2.0, 5)
    rp, col = g.row_ptr, g.col.copy()
    rng = np.random.default_rng(n)
    if shuffled:
        for x in range(0, n, 7):
            rng.shuffle(col[rp[x]:rp[x + 1]])
    x = int(rng.integers(n // 2, n))
    i = int(rp[x]) + 1
    row = set(col[rp[x]:rp[x + 1]].tolist())
    if what == "moved" or what == "mirror":
        y = next(v for v in range(n) if v not in row and v != x)
        col[i] = y
    elif what == "repeated":
        col[i] = col[i - 1]
    elif what == "range":
        col[int(rp[x + 1]) - 1] = n
    elif what == "negative":
        col[int(rp[x])] = -1
    else:
        col[i] = x
    with pytest.raises(CbError) as err:
        Curveball(rp, col, 1)
    assert err.value.code == CB_EINVAL


# Trades of 4097 to 8192 entries run with eight entries per thread; above, or
# above smem_max, they keep their hash in shared memory up to 26214
# entries, with key prefixes and flags beside it up to about 18000 (16384 in the first
# pass's kernel); above, all of it is in global memory.  Hubs on both sides of
# these limits, adjacent to each other so that their trades depend on one
# another; smem_max 64 sends every trade above 64 entries the same way.
@pytest.mark.parametrize("options", [{}, {"inorder_threads": 256}, {"smem_max": 64}, {"smem_max": 2000, "cta_paths": 0}])
def test_trades_of_the_largest_class(options):
    n = 40000
    rng = np.random.default_rng(5)
    g = synth.powerlaw_graph(n, 2, 30, 2.0, 12)
    rows = np.repeat(np.arange(n, dtype=np.int64), np.diff(g.row_ptr))
    pairs = [np.stack([rows, g.col.astype(np.int64)], 1)]
    for hub, d in enumerate([4085, 4200, 8185, 8300, 12000, 15990, 16400, 17700, 20000, 26190, 26240, 30000]):
        pairs.append(np.stack([np.full(d, hub), rng.permutation(n)[:d]], 1))
    e = np.concatenate(pairs)
    e = e[e[:, 0] != e[:, 1]]
    e = np.unique(np.sort(e, axis=1), axis=0)
    both = np.concatenate([e, e[:, ::-1]])
    both = both[np.lexsort((both[:, 1], both[:, 0]))]
    rp = np.concatenate([[0], np.cumsum(np.bincount(both[:, 0], minlength=n))]).astype(np.int64)
    col = both[:, 1].astype(np.int32)
    c, o = Curveball(rp, col, 3), Oracle(rp, col, 3)
    for k, v in options.items():
        c.set_option(k, v)
    for _ in range(4):
        c.global_trades(1)
        o.superstep(1)
        assert np.array_equal(c.edges(), o.edges())
    assert c.stats()["global_ws_trades"] > 0
    c.close()


# Steps of one call compute the next permutation (of larger handles the first
# of its kernels) beside the in-order pass, in a third set of arrays: calls of different lengths, single
# steps, recorded steps and other uses of the handle between them.
@pytest.mark.parametrize("n,b", [(9, 5), (1025, 60), (4096, 200), (5001, 2000), (32769, 30), (65534, 12), (150001, 9)])
def test_calls_of_several_steps(n, b):
    g = synth.powerlaw_graph(n, 1, max(2, b), 2.0, 23)
    c, o = Curveball(g.row_ptr, g.col, 7), Oracle(g.row_ptr, g.col, 7)
    for i, k in enumerate([1, 2, 3, 1, 4, 5, 6, 2, 2, 7]):
        if i == 4:
            c.set_option("cuda_graph", 1)
        if i == 6:
            c.set_option("cuda_graph", 0)
        if i == 8:
            c.set_option("relaxed", 1)
            o.set_relaxed(True)
        if i == 9:
            c.set_option("relaxed", 0)
            o.set_relaxed(False)
        c.global_trades(k)
        o.superstep(k)
        assert np.array_equal(c.edges(), o.edges()), f"after call {i} of {k} steps"
        if i % 3 == 0 and n > 1:
            c.uniform_trades(n)
            o.uniform_trades(n)
        if i == 5:
            c.set_option("cuda_graph", 1)
            c.global_trades(1)
            o.superstep(1)
            c.set_option("cuda_graph", 0)
            c.global_trades(4)
            o.superstep(4)
            c.set_option("cuda_graph", 1)
            c.global_trades(3)
            o.superstep(3)
            assert np.array_equal(c.edges(), o.edges())
    c.close()


@pytest.mark.parametrize("sizes", [(3, 1, 0, 2), (1023, 1024, 1025, 9), (9000, 12001, 700), (40001, 30, 90000)])
def test_batch_calls_of_several_steps(sizes):
    graphs = []
    for n in sizes:
        g = synth.powerlaw_graph(n, 2, min(n // 2, 60), 2.0, n) if n >= 4 else None
        graphs.append((g.row_ptr, g.col) if g else (np.zeros(n + 1, np.int64), np.zeros(0, np.int32)))
    seeds = [5 + i for i in range(len(graphs))]
    e = Ensemble(graphs, seeds)
    oracles = [Oracle(rp, col, s) for (rp, col), s in zip(graphs, seeds)]
    for k in (2, 3, 1, 5):
        e.global_trades(k)
        for i, o in enumerate(oracles):
            o.superstep(k)
            assert np.array_equal(e.graph_edges(i), o.edges())
    e.close()
