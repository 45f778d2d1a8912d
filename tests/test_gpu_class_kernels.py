"""The kernels of large graphs on small ones.  "fuse_max" 0 gives every size
class its own first-pass kernel (eight entries per thread above 256 entries,
two hash slots per entry), "retry_min" 0 makes retry passes run: both with the
options that force their rarer branches, on handles of one graph and of
several.  Whole numbers: equal to the oracle."""
import numpy as np
import pytest

from oracle import Oracle
from paper_1804_08487_gb300 import synth
from paper_1804_08487_gb300.cb import CB_EINVAL, TRADE_CLASSES, CbError, Curveball, Ensemble

pytestmark = pytest.mark.gpu

# n, smallest and largest degree: small trades only; every class up to 2048
# entries; hubs up to the largest class; a dense core of dependent trades
GRAPHS = {"small": (3001, 2, 40), "middle": (3000, 4, 1500), "hubs": (12000, 8, 6000), "dense": (400, 60, 300)}


def _graph(name):
    n, a, b = GRAPHS[name]
    return synth.powerlaw_graph(n, a, b, 2.0, 13)


@pytest.mark.parametrize("name", GRAPHS)
@pytest.mark.parametrize("options", [
    {}, {"cand_max": 1}, {"wide_pack": 1}, {"lane_teams": 0}, {"lane_teams": 0, "cand_max": 1}, {"tile_max": 0}, {"tile_max": 48},
    {"tile_paths": 0}, {"block_max": 128}, {"block_max": 300}, {"block_max": 2048}, {"smem_max": 64}, {"smem_max": 600},
    {"smem_max": 3000}, {"smem_max": 5000}, {"cta_paths": 0}, {"inorder_threads": 256}, {"fix_passes": 3},
])
def test_a_kernel_per_class(name, options):
    g = _graph(name)
    c, o = Curveball(g.row_ptr, g.col, 5), Oracle(g.row_ptr, g.col, 5)
    c.set_option("fuse_max", 0)
    for k, v in options.items():
        c.set_option(k, v)
    for steps in (1, 2):
        c.global_trades(steps)
        o.superstep(steps)
        assert np.array_equal(c.edges(), o.edges())
    st = c.stats()
    assert sum(st[f"class{k}_trades"] for k in range(TRADE_CLASSES)) == (g.n + 1) // 2
    c.close()


def test_every_class_has_trades():
    st = []
    for name in GRAPHS:
        g = _graph(name)
        c = Curveball(g.row_ptr, g.col, 5)
        c.set_option("fuse_max", 0)
        c.global_trades(1)
        st.append(c.stats())
        c.close()
    for k in range(TRADE_CLASSES):
        assert sum(s[f"class{k}_trades"] for s in st) > 0, k


@pytest.mark.parametrize("fuse_max", [0, 1 << 17])
@pytest.mark.parametrize("retry", [0, 1, 2, 3, 4])
@pytest.mark.parametrize("name,options", [
    ("small", {}), ("middle", {}), ("middle", {"cand_max": 1, "inorder_threads": 256}), ("hubs", {}),
    ("hubs", {"smem_max": 2000}), ("dense", {}), ("dense", {"block_max": 0, "tile_max": 0}),
])
def test_retry_passes(name, options, retry, fuse_max):
    g = _graph(name)
    c, o = Curveball(g.row_ptr, g.col, 9), Oracle(g.row_ptr, g.col, 9)
    for k, v in {"retry_min": 0, "retry_passes": retry, "fuse_max": fuse_max, **options}.items():
        c.set_option(k, v)
    launches = []
    for steps in (1, 1, 3):   # the last call computes its permutations ahead
        c.global_trades(steps)
        o.superstep(steps)
        st = c.stats()
        launches.append(st["launches"])
        assert 1 <= st["passes"] <= 2 + retry and 0 <= st["inorder_trades"] <= st["deferred"]
        assert np.array_equal(c.edges(), o.edges())
    c.set_option("retry_passes", 0)
    c.global_trades(1)
    # a retry pass is up to three kernels: trades up to 128, up to 1024, larger
    kernels = 1 + (2 * int(np.diff(g.row_ptr).max()) > 128) + (2 * int(np.diff(g.row_ptr).max()) > 1024)
    assert launches[1] - c.stats()["launches"] == retry * kernels
    c.close()


@pytest.mark.parametrize("options", [{}, {"cand_max": 1}, {"wide_pack": 1}, {"lane_teams": 0}, {"cta_paths": 0}])
@pytest.mark.parametrize("retry", [0, 3])
def test_batch(options, retry):
    graphs = [_graph(name) for name in GRAPHS]
    e = Ensemble([(g.row_ptr, g.col) for g in graphs], [1, 2, 3, 4])
    oracles = [Oracle(g.row_ptr, g.col, i + 1) for i, g in enumerate(graphs)]
    for k, v in {"fuse_max": 0, "retry_min": 0, "retry_passes": retry, **options}.items():
        e.set_option(k, v)
    for steps in (1, 2):
        e.global_trades(steps)
        for i, o in enumerate(oracles):
            o.superstep(steps)
            assert np.array_equal(e.graph_edges(i), o.edges())
    e.close()


@pytest.mark.parametrize("key", ["fuse_max", "retry_min"])
def test_option_range(key):
    g = _graph("small")
    c = Curveball(g.row_ptr, g.col, 1)
    for bad in (-1, (1 << 31) + 1):
        with pytest.raises(CbError) as e:
            c.set_option(key, bad)
        assert e.value.code == CB_EINVAL
    c.close()
