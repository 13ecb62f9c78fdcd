// adjoint_k0.cu -- the adjoint kernels of kind 0 (adjoint_kernel.cuh).
#include "adjoint_kernel.cuh"

namespace rubix {
AdjointFn adjoint_fn_k0(int R, bool mean) { return adjoint_fn<0>(R, mean); }
}  // namespace rubix
