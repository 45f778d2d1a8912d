"""The super step at the edges of its launch rules: the permutation's rescan
and scatter forms, its slow bucket paths, the row offsets that both write, and
the passes over deferred trades for small and large handles.  Whole numbers:
equal to the oracle element by element."""
import numpy as np
import pytest

from oracle import Oracle
from paper_1804_08487_gb300 import synth
from paper_1804_08487_gb300.cb import Curveball, Ensemble

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
