// BF16-factor MTTKRP instantiations of memory-lean copies for ranks between the
// fast shapes, 4 modes.
#include "mttkrp_inst.cuh"

namespace spm {
MttkrpKernelFn pick_mttkrp_bf16_lean_between4(int R) { return pick_mttkrp_between_t<__nv_bfloat16, 3, true>(R); }
}  // namespace spm
