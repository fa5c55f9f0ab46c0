// solver_inst_f64v.cu -- instances of the persistent GMRES and whole-step kernels
// (solver_kernels.cuh) for systems with a per-voxel diffusivity.
#include "solver_kernels.cuh"

namespace mpm {
Variant inst_f64_8_var() { return var_of<double, 8, 2, 1, 512, true>(); }
Variant inst_f64_16_var() { return var_of<double, 16, 1, 1, 512, true>(); }
}  // namespace mpm
