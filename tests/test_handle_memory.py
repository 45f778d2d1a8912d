"""Device memory of a handle beside its adjacency, and the lists that share an
array.  The class lists and the deferred trades' lists hold every trade once,
so two lists share an array of as many places as there are trades: one from the
front, one from the back (csrc/pair_lists.cuh, compiled as plain C++ here)."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_1804_08487_gb300 import synth
from paper_1804_08487_gb300.cb import Curveball, cb_device_bytes, cb_estimate_bytes

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1804_08487_gb300", "csrc")


# offsets, orders, positions (three sets where steps run ahead, below 2^20
# trades), lists, thresholds, records, permutation scratch
@pytest.mark.parametrize("n,limit", [(1 << 15, 90), (1 << 15 | 2, 97), (1 << 20, 97), ((1 << 21) - 2, 97), (1 << 21, 82),
                                     (1 << 25, 82), (1 << 28, 82), ((1 << 31) - 2, 87)])
def test_bytes_per_node(n, limit):
    fixed = 16 << 20   # slack of the estimate
    assert (cb_estimate_bytes(n, 2, 1) - fixed) / (1 + 1 / 64) <= limit * n


_PROG = r"""
#define __host__
#define __device__
#include <cstdio>
#include "pair_lists.cuh"
int main() {
  long long list, i, cap;
  while (std::scanf("%lld %lld %lld", &list, &i, &cap) == 3)
    std::printf("%lld\n", static_cast<long long>(cb::pair_place(static_cast<int>(list), i, cap)));
  return 0;
}
"""


@pytest.mark.parametrize("lengths", [[5], [0, 5], [3, 2], [1, 0, 2, 2], [0, 0, 0, 0, 0, 0, 0, 5, 0], [1, 1, 1, 1, 1, 0, 0, 0, 0],
                                     [0, 4, 1], [1 << 10, 7, 0, 1]])
def test_paired_lists_do_not_meet(tmp_path, lengths):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("g++ not available")
    src, exe = tmp_path / "lists.cpp", tmp_path / "lists"
    src.write_text(_PROG)
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    cap = sum(lengths)
    text = "".join(f"{k} {i} {cap}\n" for k, length in enumerate(lengths) for i in range(length))
    out = subprocess.run([str(exe)], input=text, capture_output=True, text=True, check=True).stdout
    places = [int(v) for v in out.split()]
    assert len(places) == len(set(places)) == cap
    assert min(places) >= 0 and max(places) < (len(lengths) + 1) // 2 * cap


@pytest.mark.gpu
@pytest.mark.parametrize("n", [4096, 32768, 40000])
def test_wide_records_and_relaxed_steps_within_the_estimate(n):
    from oracle import Oracle
    g = synth.powerlaw_graph(n, 2, 40, 2.0, 4)
    c, o = Curveball(g.row_ptr, g.col, 9), Oracle(g.row_ptr, g.col, 9)
    before = cb_device_bytes(c.h)[0]
    assert before <= cb_estimate_bytes(g.n, len(g.col), int(np.diff(g.row_ptr).max()))
    c.set_option("wide_pack", 1)
    c.set_option("wide_pack", 1)
    assert cb_device_bytes(c.h)[0] == before + 16 * (n // 2)
    c.global_trades(2)
    c.set_option("wide_pack", 0)
    assert cb_device_bytes(c.h)[0] == before
    c.global_trades(2)
    o.superstep(4)
    assert np.array_equal(c.edges(), o.edges())
    c.set_option("relaxed", 1)
    o.set_relaxed(True)
    c.global_trades(3)
    o.superstep(3)
    assert np.array_equal(c.edges(), o.edges())
    c.close()
