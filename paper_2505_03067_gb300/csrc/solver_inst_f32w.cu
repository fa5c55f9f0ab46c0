// solver_inst_f32w.cu -- instances of the persistent GMRES and whole-step kernels
// (solver_kernels.cuh) for systems with a per-voxel diffusivity.
#include "solver_kernels.cuh"

namespace mpm {
Variant inst_f32_32_var() { return var_of<float, 32, 1, 1, 512, true>(); }
}  // namespace mpm
