// F32-factor MTTKRP instantiations of memory-lean copies for ranks between the
// fast shapes, 3 modes.
#include "mttkrp_inst.cuh"

namespace spm {
MttkrpKernelFn pick_mttkrp_f32_lean_between3(int R) { return pick_mttkrp_between_t<float, 2, true>(R); }
}  // namespace spm
