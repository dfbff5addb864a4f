// F32-factor MTTKRP instantiations for ranks between the fast shapes, 3 modes.
#include "mttkrp_inst.cuh"

namespace spm {
MttkrpKernelFn pick_mttkrp_f32_between3(int R) { return pick_mttkrp_between_t<float, 2>(R); }
}  // namespace spm
