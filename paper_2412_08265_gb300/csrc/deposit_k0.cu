// deposit_k0.cu -- the deposit kernels of kind 0 (deposit_kernel.cuh).
#include "deposit_kernel.cuh"

namespace rubix {
DepositFn deposit_fn_k0(int R, bool means) { return deposit_fn<0>(R, means); }
}  // namespace rubix
