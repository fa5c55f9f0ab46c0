// solver_inst_f64w.cu -- instances of the persistent GMRES and whole-step kernels
// (solver_kernels.cuh) for systems with a per-voxel diffusivity.
#include "solver_kernels.cuh"

namespace mpm {
Variant inst_f64_32_var() { return var_of<double, 32, 1, 1, 512, true>(); }
}  // namespace mpm
