// Split-axis passes (ksplit.cuh) of the grid sides 180, 192, 200, 216, 240.
#include "ksplit.cuh"

namespace pat {

const SplitOps* split_ops_large(int ng) {
    switch (ng) {
        case 180: { static const SplitOps o = SplitImpl<12, 15, 4, 4>::ops(); return &o; }
        case 192: { static const SplitOps o = SplitImpl<12, 16, 4, 4>::ops(); return &o; }
        case 200: { static const SplitOps o = SplitImpl<10, 20, 4, 4>::ops(); return &o; }
        case 216: { static const SplitOps o = SplitImpl<12, 18, 4, 4>::ops(); return &o; }
        case 240: { static const SplitOps o = SplitImpl<12, 20, 4, 4>::ops(); return &o; }
        default: return nullptr;
    }
}

}  // namespace pat
