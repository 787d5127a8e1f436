// Split-axis passes (ksplit.cuh) of the grid sides 360, 384, 400.
#include "ksplit.cuh"

namespace pat {

const SplitOps* split_ops_huge(int ng) {
    switch (ng) {
        case 360: { static const SplitOps o = SplitImpl<18, 20, 4, 4>::ops(); return &o; }
        case 384: { static const SplitOps o = SplitImpl<16, 24, 4, 4>::ops(); return &o; }
        case 400: { static const SplitOps o = SplitImpl<20, 20, 4, 4>::ops(); return &o; }
        default: return nullptr;
    }
}

}  // namespace pat
