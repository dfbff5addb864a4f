// BF16-factor MTTKRP instantiations of memory-lean copies for ranks between the
// fast shapes, 5 modes.
#include "mttkrp_inst.cuh"

namespace spm {
MttkrpKernelFn pick_mttkrp_bf16_lean_between5(int R) { return pick_mttkrp_between_t<__nv_bfloat16, 4, true>(R); }
}  // namespace spm
