// ac_mixed_host.h -- host-side choices of the mixed form's pressure reference and level
// (shared by the single-tank and batched contexts).
#pragma once

#include "../../include/ac.h"

namespace acgb {

inline bool is_wall_side(int b) { return b == AC_BC_WALL_SLIP || b == AC_BC_WALL_NOSLIP; }

// The hydrostatic reference applies when both y sides are walls and the
// pressure gradient comes from the rearranged momentum equation.
inline bool mixed_uses_reference(const ac_bc &bc, int gradp) {
    return is_wall_side(bc.ylo) && is_wall_side(bc.yhi) && gradp == AC_GRADP_NEW;
}

// The pressure is carried as an FP32 increment over an FP64 level when the
// pressure gradient comes from the rearranged momentum equation; a limited
// pressure gradient needs pressure differences, so there the FP32 record
// holds p itself.
inline bool mixed_uses_level(int gradp) { return gradp == AC_GRADP_NEW; }

}  // namespace acgb
