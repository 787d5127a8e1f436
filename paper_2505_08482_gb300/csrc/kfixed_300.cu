// Fixed-size passes of the four-pass step for the grid side Ng = 300 = 20 x 15 (variant 0 of the plan is
// the split-axis step, ksplit.cuh; entry 0 here is the plan's last variant and serves workspaces too small for
// the split-axis step).  Entries, the plan's variants from 1 on: 0 column and velocity
// passes on the 20 x 15 factorisation, density passes on 15 x 20 (fewer registers where the
// state is preloaded), and 8-column tiles for the column passes of the forward sweep, which
// runs alone on the GPU; 1 all 20 x 15, 4 rows / 4 columns per CTA; 2 the same with 8 rows /
// 2 columns; 3 state staged in shared memory by TMA bulk copies; 4 all 15 x 20; 5 as 0 with 8 rows per CTA in the row passes; 6 as 0 with the segment recompute's row passes staged by TMA (fewer registers beside the adjoint); 7 as 5 with the column
// passes on the three-level 5 x 10 x 6 transform (60 threads per column: 4 columns per CTA,
// 8 in the forward sweep); 8 the same with 2 and 4 columns per CTA; 9 as 5 with 4-column tiles
// for the column passes of the forward sweep too (more CTAs per SM when a launch has many waves);
// 10 as 5 with column passes that form their multipliers where they use them (less shared memory:
// faster for launches of many waves, slower in a chain of one-wave launches).
#include "kfixed.cuh"

namespace pat {

namespace {
using A4 = FixedImpl<20, 15, 4, 4, false>;
using A8 = FixedImpl<20, 15, 8, 2, false>;
using S4 = FixedImpl<20, 15, 4, 4, true>;
using B4 = FixedImpl<15, 20, 4, 4, false>;
using C8 = FixedImpl<20, 15, 4, 8, false>;
using B8 = FixedImpl<15, 20, 8, 2, false>;   // density rows, 8 rows per CTA
using SB = FixedImpl<15, 20, 4, 4, true>;    // density rows staged by TMA (segment recompute)
using PA = FixedImpl<20, 15, 8, 4, false>;   // persistent sweep: columns and velocity rows
using PB = FixedImpl<15, 20, 8, 4, false>;   // persistent sweep: density rows
using T4 = Col3Impl<5, 10, 6, 4>;            // three-level column passes
using T8 = Col3Impl<5, 10, 6, 8>;
using T2 = Col3Impl<5, 10, 6, 2>;
using L4 = ColLeanImpl<20, 15, 4>;           // column passes, multipliers formed where used
using L8 = ColLeanImpl<20, 15, 8>;
}  // namespace

const FixedOps* fixed_ops_300(int v) {
    static const FixedOps ops[] = {MixedImpl<A4, A4, B4, B4, C8>::ops(), A4::ops(), A8::ops(), S4::ops(), B4::ops(),
                                   MixedImpl<A4, A8, B8, B8, C8>::ops(),
                                   MixedImpl<A4, A4, B4, B4, C8, S4, SB>::ops(),
                                   MixedImpl<T4, A8, B8, B8, T8>::ops(), MixedImpl<T2, A8, B8, B8, T4>::ops(),
                                   MixedImpl<A4, A8, B8, B8, A4>::ops(), MixedImpl<L4, A8, B8, B8, L8>::ops()};
    return (v >= 0 && v < int(sizeof(ops) / sizeof(ops[0]))) ? &ops[v] : nullptr;
}

const SweepOps* sweep_ops_300() {
    static const SweepOps ops = SweepImpl<PersistentImpl<PA, PA, PB>>::ops();
    return &ops;
}

}  // namespace pat
