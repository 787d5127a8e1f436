// Split-axis passes (ksplit.cuh) of the grid sides 120, 128, 144, 150, 160.
#include "ksplit.cuh"

namespace pat {

const SplitOps* split_ops_mid(int ng) {
    switch (ng) {
        case 120: { static const SplitOps o = SplitImpl<10, 12, 4, 4>::ops(); return &o; }
        case 128: { static const SplitOps o = SplitImpl<8, 16, 4, 4>::ops(); return &o; }
        case 144: { static const SplitOps o = SplitImpl<12, 12, 4, 4>::ops(); return &o; }
        case 150: { static const SplitOps o = SplitImpl<10, 15, 4, 4>::ops(); return &o; }
        case 160: { static const SplitOps o = SplitImpl<10, 16, 4, 4>::ops(); return &o; }
        default: return nullptr;
    }
}

}  // namespace pat
