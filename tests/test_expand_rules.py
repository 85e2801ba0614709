"""The rule by which the workers of the forward / dX kernel share the last output (csrc/expand_rules.h),
against the pipeline played through step by step.  Host code only: no GPU is needed."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2210_03858_b200", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "expand_rules.h"
int main() {
    std::printf("%d %d\n", bcq::kPfGroups, bcq::kPfWeightSlots);
    for (int full = 1; full <= 40; ++full)
        for (int kb = 1; kb <= 12; ++kb)
            for (int parts = 0; parts < 2; ++parts)
                std::printf("%d %d %d %d\n", full, kb, parts, (int)bcq::helpers_may_share(full, parts, 8, kb));
}
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    src, exe = d / "rules.cpp", d / "rules"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    lines = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.splitlines()
    groups, slots = map(int, lines[0].split())
    return groups, slots, {tuple(map(int, l.split()[:3])): l.split()[3] == "1" for l in lines[1:]}


def worst_case_is_safe(groups, slots, segments, kb):
    """Whether every group, as far ahead as its waits allow, finds the accumulator's use before last
    complete when it starts to wait for the last one.  (A part in front is counted as long as a tile: what
    comes before the last two segments does not matter.)"""
    total = segments * kb
    if segments < 3:
        return True
    use_before_last = (segments - 2) * kb - 1       # last stage of the segment two back
    for g in range(groups):
        stages = range(g, total, groups)
        if not stages:
            return False
        retired = stages[-1] - slots                # the newest stage this group knows to be retired
        # the accumulator is signalled behind that stage's own signal: a later stage has to be retired
        if retired <= use_before_last:
            return False
    return True


def test_workers_share_the_last_output_only_where_the_parity_is_unambiguous(rule):
    groups, slots, allowed = rule
    for (full, kb, parts), ok in allowed.items():
        # 8 pairs; a pair walks full / 8 tiles, rounded up or down, after perhaps one part of a shared tile
        for tiles in {full // 8, -(-full // 8)}:
            if ok:
                assert worst_case_is_safe(groups, slots, tiles + parts, kb), (full, kb, parts)
    # ... and wherever there is no earlier use, or the K loop is not short, they do
    assert all(ok for (full, kb, parts), ok in allowed.items()
               if -(-full // 8) + parts <= 2 or 2 * kb >= groups + slots)
