// Depth of the matrix-free product's stage ring and the generator groups that share it
// (gemm_mf.cuh).  Plain C++.
#pragma once

namespace wfq {
namespace tc {

constexpr int MF_GROUPS = 4;

struct MfPlan {
    int stages, groups;
};

// `fit`: stages that shared memory holds, or the autotuner's shallower choice (>= 2).  Groups
// take the stages in turn and wait only for their own, by a barrier's one-bit phase parity: right
// only if a waiter has seen the slot's previous phase complete.  The bulk copies of two stages may
// land in either order, so a group must itself have waited for each earlier use of its slots: the
// depth is a multiple of the groups (7, 6 and 5 stages, of blocks of 96 to 192 real columns, are cut
// to 4).  With fewer than MF_GROUPS stages one group generates every stage.
inline MfPlan mf_plan(int fit) {
    if (fit >= MF_GROUPS) return {fit / MF_GROUPS * MF_GROUPS, MF_GROUPS};
    return {fit, 1};
}

}  // namespace tc
}  // namespace wfq
