"""Kernels that may be resident while the kernel before them still runs (no GPU:
the sources are read).  A kernel that calls after_previous() must not promise
the compiler that its inputs never change while it lives: no __restrict__
parameter, and __ldg only for what the creation of a handle fixed."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1804_08487_gb300", "csrc")

# what __ldg may read in the files of such kernels: members of the segment
# table and arrays that only the creation of a handle writes
FIXED = re.compile(r"__ldg\((&S->(seed|off|n|span|bucket_base|slot_base|B|cap)|&ks\.segs\[mid\]\.bucket_base|"
                   r"ks\.seg_of \+ x|deg \+ x)\)")


def _code(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def _body(text, start):
    """The braces that open at or after `start`."""
    i = text.index("{", start)
    depth = 0
    for j in range(i, len(text)):
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        if depth == 0:
            return text[i:j + 1]
    raise AssertionError("unbalanced braces")


def _kernels(text):
    for m in re.finditer(r"__global__[^;{]*?\b(k_\w+)\s*\(([^{;]*)\)\s*\{", text):
        yield m.group(1), m.group(2), _body(text, m.end() - 1)


def test_overlapped_kernels_take_plain_pointers():
    seen = []
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith(".cu"):
            continue
        for kernel, params, body in _kernels(_code(name)):
            if "after_previous()" in body:
                seen.append(kernel)
                assert "__restrict__" not in params, f"{name}: {kernel}"
                assert "__restrict__" not in body, f"{name}: {kernel}"
    assert {"k_phase_a_class", "k_phase_a_small", "k_phase_a_large", "k_phase_a_huge", "k_phase_a_block", "k_def_list",
            "k_resolve", "k_fixup", "k_perm_rescan", "k_perm_scatter", "k_bucket_sort"} <= set(seen)


@pytest.mark.parametrize("name", ["trade.cu", "permute.cu", "classes.cuh", "team.cuh", "philox.cuh"])
def test_read_only_loads_are_of_fixed_data(name):
    code = _code(name)
    assert len(re.findall(r"__ldg\(", code)) == len(FIXED.findall(code)), name
