// Reverse-mode step (FP64).
#include "adjoint_binned.cuh"

namespace rsol {

cudaError_t adjoint_step_f64(const AdjDesc &d, cudaStream_t s) { return adjoint_dispatch<double>(d, s); }

} // namespace rsol
