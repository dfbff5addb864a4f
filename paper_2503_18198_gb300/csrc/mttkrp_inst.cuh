// mttkrp_inst.cuh -- kernel selection for one factor storage type and a set
// of input-mode counts.  Included by several translation units so that the
// instantiations compile in parallel.
#pragma once

#include "mttkrp_kernel.cuh"

namespace spm {

using MttkrpKernelFn = void (*)(const MttkrpArgs);

#ifndef SPM_MT_NARROW
#define SPM_MT_NARROW 0
#endif

// Ranks between the fast shapes: VEC ranks per lane (a divisor of R that keeps
// every lane's load aligned), the lanes padded to a power of two and masked, so
// that a warp step still holds 32 / LPN nonzeros.  Odd ranks take one rank per
// lane.  (2M nonzeros, R = 24, FP32, three modes: 652 us with one nonzero per
// step and eight chunks of 32 ranks, 158 us so; R = 10, 48, 100 with 3 modes: 253,
// 280, 335 us per mode against 43, 72, 112.)  Lean plans take the same shapes, so
// that their sums are the full plan's bit for bit (same 2M nonzeros, R = 24, all modes: 619 -> 170 us).
template <typename FT, int NIN, bool LEAN = false>
MttkrpKernelFn pick_mttkrp_between_t(int R) {
  constexpr int RI = record_int4s(NIN + 1);
  if constexpr (sizeof(FT) == 2) {
    if (R % 8 == 0 && R > 32) {
      if (R <= 64) return &mttkrp_kernel<RI, NIN, FT, 8, 8, 1, LEAN, false, true>;
      if (R <= 128) return &mttkrp_kernel<RI, NIN, FT, 8, 16, 1, LEAN, false, true>;
      return &mttkrp_kernel<RI, NIN, FT, 8, 32, 1, LEAN, false, true>;
    }
  }
  if (R % 4 == 0 && R <= 128) {
    if (R <= 32) return &mttkrp_kernel<RI, NIN, FT, 4, 8, 1, LEAN, false, true>;
    if (R <= 64) return &mttkrp_kernel<RI, NIN, FT, 4, 16, 1, LEAN, false, true>;
    return &mttkrp_kernel<RI, NIN, FT, 4, 32, 1, LEAN, false, true>;
  }
  if (R % 2 == 0 && R <= 64) {
    if (R <= 16) return &mttkrp_kernel<RI, NIN, FT, 2, 8, 1, LEAN, false, true>;
    if (R <= 32) return &mttkrp_kernel<RI, NIN, FT, 2, 16, 1, LEAN, false, true>;
    return &mttkrp_kernel<RI, NIN, FT, 2, 32, 1, LEAN, false, true>;
  }
  if (R <= 16) return &mttkrp_kernel<RI, NIN, FT, 1, 16, 1, LEAN>;
  if (R <= 32) return &mttkrp_kernel<RI, NIN, FT, 1, 32, 1, LEAN>;
  if (R <= 64) return &mttkrp_kernel<RI, NIN, FT, 1, 32, 2, LEAN>;
  return nullptr;
}

// Fast shapes: the rank is VEC * LPN * CPL with one 16-byte load per lane
// and chunk.  Anything else uses the scalar variant (one nonzero per step)
// unless pick_mttkrp_between_t has a shape for it.
template <typename FT, int NIN, bool LEAN = false, bool PLAN = false>
MttkrpKernelFn pick_mttkrp_t(int R) {
  constexpr int RI = record_int4s(NIN > 0 ? NIN + 1 : SPM_MAX_MODES);
  constexpr int VEC = 16 / (int)sizeof(FT);
  if constexpr (sizeof(FT) == 2 && NIN == 2) {  // 3-mode BF16 with R <= 32: 8-byte lane loads
    if (R % 4 == 0 && R <= 32) {
      switch (R / 4) {
        case 1: return &mttkrp_kernel<RI, NIN, FT, 4, 1, 1, LEAN, PLAN>;
        case 2: return &mttkrp_kernel<RI, NIN, FT, 4, 2, 1, LEAN, PLAN>;
        case 4: return &mttkrp_kernel<RI, NIN, FT, 4, 4, 1, LEAN, PLAN>;
        case 8: return &mttkrp_kernel<RI, NIN, FT, 4, 8, 1, LEAN, PLAN>;
        default: break;
      }
    }
  }
#if SPM_MT_NARROW
  // FP32 rows of 32 or 64 ranks on half as many lanes, two 16-byte chunks
  // per lane: twice the nonzeros per warp step
  if constexpr (sizeof(FT) == 4 && NIN > 0) {
    if (R == 8 * VEC) return &mttkrp_kernel<RI, NIN, FT, VEC, 4, 2, LEAN, PLAN>;
    if (R == 16 * VEC) return &mttkrp_kernel<RI, NIN, FT, VEC, 8, 2, LEAN, PLAN>;
  }
#endif
  if (R % VEC == 0) {
    switch (R / VEC) {
      case 1: return &mttkrp_kernel<RI, NIN, FT, VEC, 1, 1, LEAN, PLAN>;
      case 2: return &mttkrp_kernel<RI, NIN, FT, VEC, 2, 1, LEAN, PLAN>;
      case 4: return &mttkrp_kernel<RI, NIN, FT, VEC, 4, 1, LEAN, PLAN>;
      case 8: return &mttkrp_kernel<RI, NIN, FT, VEC, 8, 1, LEAN, PLAN>;
      case 16:
        if constexpr (!PLAN || 16 * VEC <= 64) return &mttkrp_kernel<RI, NIN, FT, VEC, 16, 1, LEAN, PLAN>;
        break;
      default: break;
    }
    if constexpr (!PLAN) {  // plan order serves CP-ALS: R <= 64
      switch (R / VEC) {
        case 32: return &mttkrp_kernel<RI, NIN, FT, VEC, 32, 1, LEAN>;
        case 64: return &mttkrp_kernel<RI, NIN, FT, VEC, 32, 2, LEAN>;
        default: break;
      }
    }
  }
  // Plan order at other ranks: the scalar variant's order (one nonzero per warp
  // step, which the masked shapes would change) with the chunks that R fills
  if constexpr (PLAN) {
    if (R <= 32) return &mttkrp_kernel<RI, NIN, FT, 1, 32, 1, LEAN, PLAN>;
    return &mttkrp_kernel<RI, NIN, FT, 1, 32, 2, LEAN, PLAN>;
  }
  return &mttkrp_kernel<RI, NIN, FT, 1, 32, 8, LEAN, PLAN>;
}

// The generic-N variant (six or more modes) only has the scalar shape.
template <typename FT, bool PLAN = false>
MttkrpKernelFn pick_mttkrp_generic_t(int) {
  return &mttkrp_kernel<2, 0, FT, 1, 32, 8, false, PLAN>;
}

}  // namespace spm
