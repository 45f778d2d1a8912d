"""cb_autotune spends its super steps on settings that change what a call
launches: below 2^20 trades no retry pass runs, so retry_passes is neither
tried nor changed, and the other six candidates and the current settings share
the steps.  A trial of several steps is launched like a call of several, with
the next permutation computed beside the in-order pass: the chain stays equal
to the oracle's."""
import numpy as np
import pytest

from oracle import Oracle
from paper_1804_08487_gb300 import synth
from paper_1804_08487_gb300.cb import Curveball, Ensemble

pytestmark = pytest.mark.gpu


# one step to load the kernels, then (steps - 1) // 7 for each of six candidates
# and the rest for the current settings
@pytest.mark.parametrize("steps", [0, 1, 2, 7, 8, 15, 24])
@pytest.mark.parametrize("retry", [0, 4])
def test_steps_and_chain(steps, retry):
    g = synth.powerlaw_graph(5000, 4, 1500, 2.0, 13)
    c, o = Curveball(g.row_ptr, g.col, 6), Oracle(g.row_ptr, g.col, 6)
    c.set_option("retry_passes", retry)
    got = c.autotune(steps)
    assert got["steps"] == steps == c.step
    assert got["retry_passes"] == retry
    o.superstep(steps)
    assert np.array_equal(c.edges(), o.edges())
    for graph in (0, 1):
        c.set_option("cuda_graph", graph)
        c.global_trades(3)
        o.superstep(3)
        assert np.array_equal(c.edges(), o.edges())
    c.close()


def test_batch():
    graphs = [synth.powerlaw_graph(n, 2, 60, 2.0, n) for n in (500, 1501, 4000)]
    e = Ensemble([(g.row_ptr, g.col) for g in graphs], [1, 2, 3])
    got = e.autotune(22)
    assert got["steps"] == 22 == e.step and got["retry_passes"] == 2
    for i, g in enumerate(graphs):
        o = Oracle(g.row_ptr, g.col, i + 1)
        o.superstep(22)
        assert np.array_equal(e.graph_edges(i), o.edges())
    e.close()
