// BF16-factor MTTKRP instantiations for ranks between the fast shapes, 5 modes.
#include "mttkrp_inst.cuh"

namespace spm {
MttkrpKernelFn pick_mttkrp_bf16_between5(int R) { return pick_mttkrp_between_t<__nv_bfloat16, 4>(R); }
}  // namespace spm
