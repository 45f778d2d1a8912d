"""Uniform single trades at the sizes where the executor changes hands: one
warp up to 64 entries (128 in calls of more than 65536 trades), a team of the
CTA above, its entries in shared memory
up to 2048 (CTAs of 256 and 512 threads) or 4096 entries (1024), in global
memory above.  Whole numbers: equal to the oracle edge for edge."""
import numpy as np
import pytest

from oracle import Oracle
from paper_1804_08487_gb300 import synth
from paper_1804_08487_gb300.cb import Curveball

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,a,b,trades", [
    (500, 1, 3, 4000),          # a few entries: most lanes idle
    (900, 14, 19, 3000),        # around one entry per lane
    (1200, 29, 36, 4000),       # around 64
    (1200, 60, 69, 4000),       # around 128: warps and teams feed each other
    (140, 120, 138, 700),       # dense: nearly every neighbour common
    (1400, 1020, 1029, 300),    # around 2048
    (2400, 2044, 2053, 120),    # around 4096
])
@pytest.mark.parametrize("threads", [256, 512, 1024])
def test_trades_around_the_size_limits(n, a, b, trades, threads):
    g = synth.powerlaw_graph(n, a, b, 1.5, n)
    c = Curveball(g.row_ptr, g.col, n)
    o = Oracle(g.row_ptr, g.col, n)
    c.set_option("uniform_threads", threads)
    for count in (trades, 1, trades // 3):
        c.uniform_trades(count)
        o.uniform_trades(count)
        assert np.array_equal(c.edges(), o.edges())
    c.close()


@pytest.mark.parametrize("a,b", [(2, 5), (29, 36), (60, 69)])
def test_calls_on_both_sides_of_the_short_call_rule(a, b):
    g = synth.powerlaw_graph(131074, a, b, 1.5, 3)   # a chunk of the sequence is at most n/2 trades
    c = Curveball(g.row_ptr, g.col, 5)
    o = Oracle(g.row_ptr, g.col, 5)
    for count in (65536, 65537):
        c.uniform_trades(count)
        o.uniform_trades(count)
        assert np.array_equal(c.edges(), o.edges())
    c.close()
