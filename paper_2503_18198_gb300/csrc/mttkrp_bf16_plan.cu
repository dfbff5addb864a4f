// BF16-factor MTTKRP instantiations in plan order (CP-ALS), 2 and 3 modes.
#include "mttkrp_inst.cuh"

namespace spm {
MttkrpKernelFn pick_mttkrp_bf16_plan_a(int nin, int R) {
  return nin == 1 ? pick_mttkrp_t<__nv_bfloat16, 1, false, true>(R)
                  : pick_mttkrp_t<__nv_bfloat16, 2, false, true>(R);
}
}  // namespace spm
