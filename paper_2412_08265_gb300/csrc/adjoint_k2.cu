// adjoint_k2.cu -- the adjoint kernels of kind 2 (adjoint_kernel.cuh).
#include "adjoint_kernel.cuh"

namespace rubix {
AdjointFn adjoint_fn_k2(int R, bool mean) { return adjoint_fn<2>(R, mean); }
}  // namespace rubix
