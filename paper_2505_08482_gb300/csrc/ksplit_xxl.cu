// Split-axis passes (ksplit.cuh) of the grid sides 250, 320, 324.
#include "ksplit.cuh"

namespace pat {

const SplitOps* split_ops_xxl(int ng) {
    switch (ng) {
        case 250: { static const SplitOps o = SplitImpl<10, 25, 4, 4>::ops(); return &o; }
        case 320: { static const SplitOps o = SplitImpl<16, 20, 4, 4>::ops(); return &o; }
        case 324: { static const SplitOps o = SplitImpl<18, 18, 4, 4>::ops(); return &o; }
        default: return nullptr;
    }
}

}  // namespace pat
