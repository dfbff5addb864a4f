// BF16-factor MTTKRP instantiations in plan order (CP-ALS), 4 and more modes.
#include "mttkrp_inst.cuh"

namespace spm {
MttkrpKernelFn pick_mttkrp_bf16_plan_b(int nin, int R) {
  switch (nin) {
    case 3: return pick_mttkrp_t<__nv_bfloat16, 3, false, true>(R);
    case 4: return pick_mttkrp_t<__nv_bfloat16, 4, false, true>(R);
    default: return pick_mttkrp_generic_t<__nv_bfloat16, true>(R);
  }
}
}  // namespace spm
