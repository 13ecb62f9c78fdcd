// deposit_k1.cu -- the deposit kernels of kind 1 (deposit_kernel.cuh).
#include "deposit_kernel.cuh"

namespace rubix {
DepositFn deposit_fn_k1(int R, bool means) { return deposit_fn<1>(R, means); }
}  // namespace rubix
