// Split-axis passes (ksplit.cuh) of the grid sides 72, 80, 90, 96, 100, 108.
#include "ksplit.cuh"

namespace pat {

const SplitOps* split_ops_small(int ng) {
    switch (ng) {
        case 72: { static const SplitOps o = SplitImpl<8, 9, 4, 4>::ops(); return &o; }
        case 80: { static const SplitOps o = SplitImpl<8, 10, 4, 4>::ops(); return &o; }
        case 90: { static const SplitOps o = SplitImpl<9, 10, 4, 4>::ops(); return &o; }
        case 96: { static const SplitOps o = SplitImpl<8, 12, 4, 4>::ops(); return &o; }
        case 100: { static const SplitOps o = SplitImpl<10, 10, 4, 4>::ops(); return &o; }
        case 108: { static const SplitOps o = SplitImpl<9, 12, 4, 4>::ops(); return &o; }
        default: return nullptr;
    }
}

}  // namespace pat
