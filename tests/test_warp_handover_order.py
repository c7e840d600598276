"""Counters that one lane acquires on behalf of its warp (no GPU needed: read from the source).

Warp reductions, votes and shuffles hand a value to the other lanes without ordering memory
among them.  A function that acquires a counter in one lane and passes the value on by such an
intrinsic has to end the hand-over with __syncwarp(), or the other lanes' reads of what the
counter guards race with the writes it was released after."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1104_2499_gb300", "csrc")
CROSS_LANE = re.compile(r"__(?:reduce_\w+|shfl\w*|ballot|any|all|match\w*)_sync\s*\(")


def functions():
    """(name, body) of every function at namespace scope that reads a counter with acquire semantics."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"^__device__[^;{]*?\b(\w+)\([^;{]*\)\s*\{(.*?)^\}", src, flags=re.S | re.M):
            if "ld_acquire" in m.group(2):
                yield m.group(1), m.group(2)


def test_the_consumers_counters_are_found():
    assert {"ws_filled", "ws_wait"} <= {name for name, _ in functions()}


@pytest.mark.parametrize("name,body", list(functions()), ids=lambda v: v if len(v) < 40 else "")
def test_values_acquired_by_one_lane_are_handed_over_with_a_warp_barrier(name, body):
    for m in CROSS_LANE.finditer(body):
        assert "__syncwarp()" in body[m.end():], name
