"""The in-order pass completes on any part of its grid.  Other streams' kernels
may keep some of its CTAs from starting, so no chunk of deferred trades may
belong to a CTA by its index; "inorder_ctas" lets only the first CTAs take
part, the others leave at once.  Whole numbers: equal to the oracle."""
import numpy as np
import pytest

from oracle import Oracle
from paper_1804_08487_gb300 import synth
from paper_1804_08487_gb300.cb import CB_EINVAL, CbError, Curveball

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ctas", [1, 3, 100])
@pytest.mark.parametrize("threads", [256, 1024])
def test_part_of_the_grid(ctas, threads):
    # a dense core: deferred trades of every kind
    g = synth.powerlaw_graph(9000, 8, 4000, 2.0, 17)
    c, o = Curveball(g.row_ptr, g.col, 5), Oracle(g.row_ptr, g.col, 5)
    c.set_option("inorder_threads", threads)
    c.set_option("inorder_ctas", ctas)
    for steps in (1, 2):
        c.global_trades(steps)
        o.superstep(steps)
        assert np.array_equal(c.edges(), o.edges())
    assert c.stats()["deferred"] > 4
    c.close()


def test_option_range():
    g = synth.powerlaw_graph(100, 2, 10, 2.0, 1)
    c = Curveball(g.row_ptr, g.col, 1)
    for bad in (-1, 65536):
        with pytest.raises(CbError) as e:
            c.set_option("inorder_ctas", bad)
        assert e.value.code == CB_EINVAL
    c.close()
