"""Every bounded wait of the device code gives its warp one answer.

A bounded wait decides per lane.  A lane whose wait expired leaves the pipeline for
the block barrier, while one that saw the phase complete goes on to an instruction
that the whole warp executes together (mma.sync, tcgen05 loads and stores,
__syncwarp): if the lanes of one warp took different answers, neither group would
ever finish.  So a per-lane wait may be called only where a single lane runs, or
inside a warp-wide vote.  Read from the sources, no GPU."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2410_06270_gb300", "csrc")
LANE_WAITS = ("g_wait", "wait_or_abort", "mbar_wait")  # the bounded waits that answer per lane
# single-lane code: under a test of the lane, or in a function that only such code calls
ONE_LANE = re.compile(r"lane == 0|\bif \(producer\)|\bpp_produce\(")
DEFINES = re.compile(r"__forceinline__ bool (%s)\(" % "|".join(LANE_WAITS))


def _code(path):
    return re.sub(r"//[^\n]*", "", open(path).read())


def _headers(src, at):
    """Texts before the '{' of every block that encloses position `at`, innermost first."""
    out, depth, i = [], 0, at
    while i > 0:
        i -= 1
        if src[i] == "}":
            depth += 1
        elif src[i] == "{":
            if depth:
                depth -= 1
                continue
            start = max(src.rfind(c, 0, i) for c in ";{}")
            out.append(src[start + 1:i])
    return out


def per_lane_answers(src):
    """Calls of a per-lane wait whose answer a whole warp would act on lane by lane."""
    bad = []
    for m in re.finditer(r"\b(%s)\(" % "|".join(LANE_WAITS), src):
        heads = _headers(src, m.start())
        statement = src[max(src.rfind(c, 0, m.start()) for c in ";{}") + 1:m.start()]
        if DEFINES.search(statement + m.group(0)) or any(DEFINES.search(h) for h in heads):
            continue  # the definition itself, or its overload
        if statement.rstrip().endswith("__all_sync(0xffffffffu,") or any(ONE_LANE.search(h) for h in heads):
            continue
        bad.append(src[:m.start()].count("\n") + 1)
    return bad


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(CSRC, "*.cu"))), ids=os.path.basename)
def test_warps_take_one_answer_from_a_bounded_wait(path):
    assert per_lane_answers(_code(path)) == []


def test_a_per_lane_answer_is_found():
    ok = "__global__ void k() { if (lane == 0) { if (!g_wait(b, 0)) return; } x = __all_sync(0xffffffffu, g_wait(b, 0)); }"
    assert per_lane_answers(ok) == []
    assert per_lane_answers("__global__ void k() { while (true) { if (!g_wait(b, 0)) break; mma(); } }") == [1]
