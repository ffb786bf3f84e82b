"""Shared memory of the small FP64 steps (no GPU: reads the sources).

Asking for more shared memory than a kernel uses, to hold its blocks one or two
to an SM, also keeps other solvers' blocks off the SM: eight FP64 solvers of
64 x 64 sites on their own streams then took 83 us per step of all instead of 58.
"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_1804_02418_gb300", "csrc")


@pytest.mark.parametrize("name,kernel,after", [
    # launch_chained(kernel, grid, block, smem, ..) and launch_chained(stream, kernel, grid, block, smem, ..)
    ("prec_impl.cuh", "k_step_split<", 2), ("massive.cu", "k_mstep", 2)])
def test_no_shared_memory_is_requested_for_room(name, kernel, after):
    code = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    calls = re.findall(r"launch_chained\(((?:[^()]|\([^()]*\))*)\);", code)
    calls = [c for c in calls if kernel in c]
    assert calls
    for c in calls:
        flat, depth, args = "", 0, []
        for ch in c:
            depth += ch in "(<"
            depth -= ch in ")>"
            if ch == "," and depth == 0:
                args.append(flat.strip())
                flat = ""
            else:
                flat += ch
        at = next(i for i, a in enumerate(args) if kernel in a)
        assert args[at + after + 1] == "0", c
