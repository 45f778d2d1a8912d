"""Edge autocorrelation of long records, on both sides of the rule that picks
the classifier: up to 8192 states in a record of at most 8192 the counts and a
fixed-point table, above (or in a longer record, however little of it is used)
the FP64 formula.  A small graph, thinnings up to 64; the reference is
oracle/autocorr.py (counts are whole numbers, equal up to decisions within
1e-9 of the BIC boundary)."""
import pytest

from oracle import Oracle
from oracle import autocorr as ac
from paper_1804_08487_gb300 import synth
from paper_1804_08487_gb300.cb import Curveball

pytestmark = pytest.mark.gpu


# a record of 8191 steps has 8192 states in 256 words, one of 8192 has 257 words
@pytest.mark.parametrize("record,steps", [(8191, 8191), (8191, 100), (8192, 8191), (8192, 8192), (8192, 100), (9000, 1)])
@pytest.mark.parametrize("kmax", [1, 64])
def test_counts_on_both_sides_of_the_rule(record, steps, kmax):
    n = 20
    g = synth.powerlaw_graph(n, 3, 9, 2.0, 5)
    c, o = Curveball(g.row_ptr, g.col, 77), Oracle(g.row_ptr, g.col, 77)
    c.set_option("presence", record)
    c.global_trades(steps)
    corr, near, occ, states = c.autocorr(kmax)
    lists = [o.edges()]
    for _ in range(steps):
        o.superstep(1)
        lists.append(o.edges())
    want, occ_w, near_w = ac.fraction_correlated(lists, n, kmax)
    assert (occ, states) == (occ_w, steps + 1)
    for k in range(kmax):
        assert abs(corr[k] - want[k]) <= near_w[k], (k + 1, corr[k], want[k])
    c.close()
