// deposit.cu -- launch of the deposit (deposit_kernel.cuh) over one or more
// galaxies that share the SSP grid and the output wavelength grid.
#include "deposit_kernel.cuh"

namespace rubix {

size_t deposit_smem_bytes(int pitch, int slab_w) { return kDepHeader + (size_t)pitch * slab_w * sizeof(float2); }

int launch_deposit(const DepositParams& P, int n_ctas, int threads, size_t smem, cudaStream_t st) {
    if (P.n_jobs < 1 || P.n_jobs > kMaxJobs) return -1;
    const int B = kind_bins(P.kind);
    if (P.tile_w % B != 0) return -1;
    bool means = false;
    for (int j = 0; j < P.n_jobs; ++j) means = means || P.jobs[j].resample;
    const int R = P.tile_w / B;
    const DepositFn fn = P.kind == 0 ? deposit_fn_k0(R, means)
                                     : (P.kind == 1 ? deposit_fn_k1(R, means) : deposit_fn_k2(R, means));
    if (!fn) return -1;
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return -1;
    fn<<<n_ctas, threads, smem, st>>>(P);
    return 1;
}

}  // namespace rubix
