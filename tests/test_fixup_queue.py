"""The rebuild's queue of prefix ties.  Every warp of a CTA has to take the same
decision to empty it, so the decision travels with the barrier: the queue's
length, which a faster warp may already be changing, is read only while the
queue is emptied (no GPU: the source is read).  With few CTAs the queue fills
many times over; equal to the oracle."""
import os
import re

import numpy as np
import pytest

from paper_1804_08487_gb300 import synth

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1804_08487_gb300", "csrc")


def test_the_barrier_carries_the_decision():
    with open(os.path.join(CSRC, "trade.cu")) as f:
        code = re.sub(r"//[^\n]*", "", f.read())
    body = code[code.index("k_fixup(StepCtx c"):]
    body = body[:body.index("\n}\n")]
    flush = body[body.index("auto flush"):]
    flush = flush[:flush.index("};") + 2]
    outside = re.sub(r"atomicAdd\(&qn, 1\)", "", body.replace(flush, ""))
    reads = [line.strip() for line in outside.splitlines() if re.search(r"\bqn\b", line)]
    assert reads == ["__shared__ int qn;", "if (threadIdx.x == 0) qn = 0;"]
    assert "__syncthreads_or(full)" in outside


# about 3 million entries: 1 in 256 of them ties, a CTA's queue holds 4096
@pytest.mark.gpu
@pytest.mark.parametrize("ctas", [1, 2, 3])
@pytest.mark.parametrize("options", [{}, {"fix_passes": 3}, {"wide_pack": 1}])
def test_queue_that_fills(ctas, options):
    from oracle import Oracle
    from paper_1804_08487_gb300.cb import Curveball
    g = synth.powerlaw_graph(60000, 20, 400, 2.0, 3)
    c, o = Curveball(g.row_ptr, g.col, 8), Oracle(g.row_ptr, g.col, 8)
    c.set_option("fix_ctas", ctas)
    for k, v in options.items():
        c.set_option(k, v)
    c.global_trades(2)
    o.superstep(2)
    assert np.array_equal(c.edges(), o.edges())
    c.close()
