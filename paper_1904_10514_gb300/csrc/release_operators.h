// Gives back the per-order operators of a plan that runs the sweeps instead, and sets
// the plan to that path.  The row offsets and the tile list stay where the synthesis
// operators S_{m,c} do: they have the operators' rows, and the kernels that apply
// S_{m,c} and its transpose walk them by the same list.
#pragma once
#include "plan.h"

namespace hpx {

template <class F>
void release_operators(hpx_plan_s* P, F release) {
    auto give = [&](auto*& q) {
        if (q) release((void*)q);
        q = nullptr;
    };
    give(P->fusedM);
    if (!P->synM) {
        give(P->fusedOff);
        give(P->fusedTiles);
    }
    give(P->tcOff);
    give(P->tcFirst);
    give(P->tcRinv);
    give(P->bscale);
    give(P->bpk);
    P->bytes -= P->fused_bytes;
    P->fused_bytes = 0;
    P->use_tc = false;
    P->flags |= HPX_FLAG_SWEEPS;
}

}  // namespace hpx
