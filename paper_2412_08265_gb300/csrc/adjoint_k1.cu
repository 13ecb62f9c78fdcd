// adjoint_k1.cu -- the adjoint kernels of kind 1 (adjoint_kernel.cuh).
#include "adjoint_kernel.cuh"

namespace rubix {
AdjointFn adjoint_fn_k1(int R, bool mean) { return adjoint_fn<1>(R, mean); }
}  // namespace rubix
