// cg_pr_kernel_pair.cu -- launches of the persistent parallel-rejection kernel
// (cg_pr_lattice.cuh) with two-electron hops on the L x L square lattice,
// L known at run time (a power of two or any even L), deterministic clock
// (the stochastic-clock instances are in cg_pr_kernel_pair_time.cu).
#include "cg_pr_lattice.cuh"

namespace cg {

template <typename Real, int kThreads>
static cudaError_t launch_pair_t(const DevReplica *d_reps, const int *d_index, int n_ctas,
                                 int smem_bytes, const RunArgs &args, cudaStream_t st, int L)
{
    if (args.time_mode)
        return launch_pr_persistent_pair_time(sizeof(Real) == 8 ? CG_FP64 : CG_FP32, d_reps,
                                              d_index, n_ctas, kThreads, smem_bytes, args, st, L);
    if (L == 64)
        pr_lattice<Real, kThreads, 6, false, 2, true>
            <<<n_ctas, kThreads, smem_bytes, st>>>(d_reps, d_index, args);
    else if ((L & (L - 1)) == 0)
        pr_lattice<Real, kThreads, 0, false, 2, true>
            <<<n_ctas, kThreads, smem_bytes, st>>>(d_reps, d_index, args);
    else
        pr_lattice<Real, kThreads, -1, false, 2, true>
            <<<n_ctas, kThreads, smem_bytes, st>>>(d_reps, d_index, args);
    return cudaGetLastError();
}

template <typename Real, int kThreads>
static cudaError_t set_pair_one(int bytes)
{
    const void *k[3] = {(const void *)pr_lattice<Real, kThreads, 6, false, 2, true>,(const void *)pr_lattice<Real, kThreads, 0, false, 2, true>,
                        (const void *)pr_lattice<Real, kThreads, -1, false, 2, true>};
    for (const void *f : k) {
        const cudaError_t e =
            cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        if (e) return e;
    }
    return cudaSuccess;
}

cudaError_t set_pr_pair_smem_limit(int precision, int bytes)
{
    cudaError_t e = set_pr_pair_time_smem_limit(precision, bytes);
    if (e) return e;
    if (precision == CG_FP64) {
        if ((e = set_pair_one<double, 1024>(bytes)) || (e = set_pair_one<double, 512>(bytes)) ||
            (e = set_pair_one<double, 384>(bytes)) || (e = set_pair_one<double, 256>(bytes)))
            return e;
    } else {
        if ((e = set_pair_one<float, 1024>(bytes)) || (e = set_pair_one<float, 512>(bytes)) ||
            (e = set_pair_one<float, 384>(bytes)) || (e = set_pair_one<float, 256>(bytes)))
            return e;
    }
    return cudaSuccess;
}

cudaError_t launch_pr_persistent_pair(int precision, const DevReplica *d_reps,
                                      const int *d_index, int n_ctas, int threads,
                                      int smem_bytes, const RunArgs &args, cudaStream_t st,
                                      int L)
{
    if (precision == CG_FP64) {
        switch (threads) {
        case 1024: return launch_pair_t<double, 1024>(d_reps, d_index, n_ctas, smem_bytes, args, st, L);
        case 512: return launch_pair_t<double, 512>(d_reps, d_index, n_ctas, smem_bytes, args, st, L);
        case 384: return launch_pair_t<double, 384>(d_reps, d_index, n_ctas, smem_bytes, args, st, L);
        case 256: return launch_pair_t<double, 256>(d_reps, d_index, n_ctas, smem_bytes, args, st, L);
        }
    } else {
        switch (threads) {
        case 1024: return launch_pair_t<float, 1024>(d_reps, d_index, n_ctas, smem_bytes, args, st, L);
        case 512: return launch_pair_t<float, 512>(d_reps, d_index, n_ctas, smem_bytes, args, st, L);
        case 384: return launch_pair_t<float, 384>(d_reps, d_index, n_ctas, smem_bytes, args, st, L);
        case 256: return launch_pair_t<float, 256>(d_reps, d_index, n_ctas, smem_bytes, args, st, L);
        }
    }
    return cudaErrorInvalidValue;
}

}  // namespace cg
