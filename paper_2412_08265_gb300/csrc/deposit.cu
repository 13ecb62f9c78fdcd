// deposit.cu -- launch of the deposit (deposit_kernel.cuh) over one or more
// galaxies that share the SSP grid and the output wavelength grid.
#include "deposit_kernel.cuh"

namespace rubix {

size_t deposit_smem_bytes(int pitch, int slab_w) { return kDepHeader + (size_t)pitch * slab_w * sizeof(float2); }

// Per-tile cost of each job (in-field particles + cost_c0 per work item) and
// its exclusive prefix, read from the device-side counts of every job.
__global__ void k_job_cost(const DepositParams P, long long* job_cost) {
    if (blockIdx.x != 0 || threadIdx.x != 0) return;
    long long acc = 0;
    for (int j = 0; j < P.n_jobs; ++j) {
        const DepJob& J = P.jobs[j];
        job_cost[j] = acc;
        const long long n_in = J.seg_off[(long long)J.n_s * P.n_bands];
        const long long n_items = J.item_off[J.n_s];
        acc += n_in + (long long)P.cost_c0 * n_items;
    }
    job_cost[P.n_jobs] = acc;
}

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
    k_job_cost<<<1, 32, 0, st>>>(P, P.job_cost);
    fn<<<n_ctas, threads, smem, st>>>(P);
    return 2;  // job-cost prep + deposit
}

}  // namespace rubix
