// cg_pr_kernel_pair.cu -- launches of the persistent parallel-rejection kernel
// (cg_pr_lattice.cuh) with two-electron hops on the square lattice,
// deterministic clock (the stochastic-clock instances are in
// cg_pr_kernel_pair_time.cu).
#include "cg_pr_lattice.cuh"

namespace cg {

cudaError_t set_pr_pair_smem_limit(int precision, int bytes)
{
    const cudaError_t e = set_pr_pair_time_smem_limit(precision, bytes);
    return e ? e : set_lattice_limit<false, 2, true>(precision, bytes);
}

cudaError_t launch_pr_persistent_pair(int precision, const DevReplica *d_reps,
                                      const int *d_index, int n_ctas, int threads,
                                      int smem_bytes, const RunArgs &args, cudaStream_t st,
                                      int L)
{
    if (args.time_mode)
        return launch_pr_persistent_pair_time(precision, d_reps, d_index, n_ctas, threads,
                                              smem_bytes, args, st, L);
    return launch_lattice<false, 2, true>(precision, d_reps, d_index, n_ctas, threads, smem_bytes,
                                          args, st, L);
}

}  // namespace cg
