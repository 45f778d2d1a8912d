"""The uniform executor's two run queues in one array (no GPU): csrc/run_queues.cuh
compiled as plain C++.  Their places are disjoint and fill the array, and a
place past a queue's own length, which would be the other queue's, is refused."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1804_08487_gb300", "csrc")

_PROG = r"""
#define __host__
#define __device__
#include <cstdio>
#include "run_queues.cuh"
int main() {
  long long trades, large;
  while (std::scanf("%lld %lld", &trades, &large) == 2) {
    const cb::RunQueues rq{trades, large};
    for (int big = 0; big < 2; ++big)
      for (long long q = 0; q < trades + 2; ++q)
        std::printf("%d %lld %d %lld\n", big, q, rq.holds(big, q) ? 1 : 0, static_cast<long long>(rq.place(big, q)));
  }
  return 0;
}
"""


@pytest.mark.parametrize("trades,large", [(1, 0), (1, 1), (7, 0), (7, 3), (7, 7), (100, 1), (100, 99)])
def test_places(tmp_path, trades, large):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("g++ not available")
    src, exe = tmp_path / "queues.cpp", tmp_path / "queues"
    src.write_text(_PROG)
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], input=f"{trades} {large}\n", capture_output=True, text=True, check=True).stdout
    places = []
    for line in out.splitlines():
        big, q, holds, place = (int(v) for v in line.split())
        assert holds == (q < (large if big else trades - large))
        if holds:
            places.append(place)
    assert sorted(places) == list(range(trades))


def test_the_executor_uses_them():
    """A push checks its own queue, the final check both."""
    with open(os.path.join(CSRC, "uniform.cu")) as f:
        code = f.read()
    push = code[code.index("void push(const UniCtx& c"):]
    push = push[:push.index("\n}\n")]
    assert "if (!rq.holds(big, q))" in push and push.index("rq.holds") < push.index("c.queue + rq.place")
    check = code[code.index("void k_uni_check("):]
    check = check[:check.index("\n}\n")]
    assert "rq.length(big)" in check and "kTail" in check and "kHead" in check
