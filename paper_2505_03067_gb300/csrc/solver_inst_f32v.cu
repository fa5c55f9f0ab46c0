// solver_inst_f32v.cu -- instances of the persistent GMRES and whole-step kernels
// (solver_kernels.cuh) for systems with a per-voxel diffusivity.
#include "solver_kernels.cuh"

namespace mpm {
Variant inst_f32_8_var() { return var_of<float, 8, 1, 1, 512, true>(); }
Variant inst_f32_16_var() { return var_of<float, 16, 1, 1, 512, true>(); }
}  // namespace mpm
