// Split-axis passes (ksplit.cuh) of the grid sides 256, 270, 288, 300.
#include "ksplit.cuh"

namespace pat {

const SplitOps* split_ops_xl(int ng) {
    switch (ng) {
        case 256: { static const SplitOps o = SplitImpl<16, 16, 4, 4>::ops(); return &o; }
        case 270: { static const SplitOps o = SplitImpl<15, 18, 4, 4>::ops(); return &o; }
        case 288: { static const SplitOps o = SplitImpl<16, 18, 4, 4>::ops(); return &o; }
        case 300: { static const SplitOps o = SplitImpl<15, 20, 4, 4>::ops(); return &o; }
        default: return nullptr;
    }
}

}  // namespace pat
