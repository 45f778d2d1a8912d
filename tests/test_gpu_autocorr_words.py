"""Edge autocorrelation at the edges of the record's 32-bit words: thinnings
up to 64 shift the series by zero, one and two words, and the number of
states ends before, at and after a word (oracle/autocorr.py as the reference;
counts are whole numbers, equal up to decisions within 1e-9 of the BIC
boundary)."""
import pytest

from oracle import Oracle
from oracle import autocorr as ac
from paper_1804_08487_gb300 import synth
from paper_1804_08487_gb300.cb import Curveball

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("steps", [1, 2, 30, 31, 32, 63, 64, 95, 127, 128, 200])
def test_counts_at_word_edges(steps):
    n, kmax = 61, 64
    g = synth.powerlaw_graph(n, 3, 20, 2.0, 5)
    c = Curveball(g.row_ptr, g.col, 77)
    c.set_option("presence", steps)
    c.global_trades(steps)
    corr, near, occ, states = c.autocorr(kmax)
    o = Oracle(g.row_ptr, g.col, 77)
    lists = [o.edges()]
    for _ in range(steps):
        o.superstep(1)
        lists.append(o.edges())
    want, occ_w, near_w = ac.fraction_correlated(lists, n, kmax)
    assert (occ, states) == (occ_w, steps + 1)
    for k in range(kmax):
        assert abs(corr[k] - want[k]) <= near_w[k], (k + 1, corr[k], want[k])
    c.close()
