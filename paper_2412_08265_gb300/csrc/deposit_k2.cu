// deposit_k2.cu -- the deposit kernels of kind 2 (deposit_kernel.cuh).
#include "deposit_kernel.cuh"

namespace rubix {
DepositFn deposit_fn_k2(int R, bool means) { return deposit_fn<2>(R, means); }
}  // namespace rubix
