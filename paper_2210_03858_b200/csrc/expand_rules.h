// Pipeline geometry of the forward / dX kernel (expand.cu) and the rule that depends on it.  Plain C++,
// so that the rule can be checked without a GPU.
#pragma once

namespace bcq {

constexpr int kPfGroups = 4;       // worker groups; group g expands the stages whose running index is g mod 4
constexpr int kPfWeightSlots = 6;  // ring of expanded weight tiles

// Whether the worker warps may share the output of a CTA's last segment.  They find its accumulator by the
// parity of a barrier alone, and that parity is ambiguous until the accumulator's previous use, two
// segments back, is complete.  All a worker knows is what it waited for: a group's last stage may be
// kPfGroups stages before the end, and to write it the group waited for the UMMAs of the stage
// kPfWeightSlots before that one.  So a stage after the segment two back (its accumulator is signalled
// behind its last stage) has to be that old: the last two segments need
// kPfWeightSlots + kPfGroups stages between them.  Where there are three segments or more the last
// two are whole tiles (a part of a shared tile comes first); with at most two there is no previous use.
// parts: whether pairs have a part of a shared tile to do.  (256 -> 4096 at 2048 tokens, two tiles of four
// stages a pair, 18.1 us with the workers' help and 20.3 without.)
inline bool helpers_may_share(int full_tiles, bool parts, int pairs, int num_kb) {
    const int segments = (full_tiles + pairs - 1) / pairs + (parts ? 1 : 0);
    return segments <= 2 || 2 * num_kb >= kPfWeightSlots + kPfGroups;
}

}  // namespace bcq
