"""Bounded waits in front of warp-wide operations, read from the source: a wait that runs out may answer differently from
lane to lane, and tensor-memory loads and stores need the whole warp.  Every branch on such an answer has to be taken once
per warp (mbar_wait_warp, or a vote); single threads may branch on their own."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_10918_b200", "csrc")
FILES = sorted(glob.glob(os.path.join(CSRC, "*_tc.cu")))
SINGLE = ("if (elect_one()) {", "if (lane == 0) {", "if (threadIdx.x == 0) {")


def _without_single_thread_blocks(src):
    src = re.sub(r"//[^\n]*", "", src)
    for head in SINGLE:
        while head in src:
            start = src.index(head)
            depth, i = 1, start + len(head)
            while depth:
                depth += {"{": 1, "}": -1}.get(src[i], 0)
                i += 1
            src = src[:start] + src[i:]
    return src


def _lane_branches(src):
    for m in re.finditer(r"\bmbar_wait(_cluster)?\(", src):
        line = src[src.rfind("\n", 0, m.start()) + 1: src.find("\n", m.start())]
        before = line[: line.find("mbar_wait")]
        if "__all_sync" in before or not re.search(r"\bif \(|=|&&", before):
            continue  # voted, or the answer is not looked at
        if re.search(r"\b(row|cl|t|threadIdx\.x) == 0 &&", before):
            continue  # a single thread's
        if re.search(r"\bok = (ok && )?$", before) and "__all_sync(0xffffffffu, ok)" in src:
            continue  # kept by the lane, voted on where it counts
        if re.search(r"const bool go =|&& *$|^\s*\(n == 0", before) and "__all_sync(0xffffffffu, go)" in src:
            continue
        yield line.strip()


@pytest.mark.parametrize("path", FILES, ids=[os.path.basename(f) for f in FILES])
def test_branches_on_waits_are_taken_once_per_warp(path):
    assert list(_lane_branches(_without_single_thread_blocks(open(path).read()))) == []
