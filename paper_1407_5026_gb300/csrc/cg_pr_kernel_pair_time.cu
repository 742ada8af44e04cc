// cg_pr_kernel_pair_time.cu -- the two-electron-hop instances of the
// persistent parallel-rejection kernel (cg_pr_lattice.cuh) with the
// stochastic clock of step 3c (CG_TIME_GAUSSIAN), square lattice.
#include "cg_pr_lattice.cuh"

namespace cg {

cudaError_t set_pr_pair_time_smem_limit(int precision, int bytes)
{
    return set_lattice_limit<true, 2, true>(precision, bytes);
}

cudaError_t launch_pr_persistent_pair_time(int precision, const DevReplica *d_reps,
                                           const int *d_index, int n_ctas, int threads,
                                           int smem_bytes, const RunArgs &args, cudaStream_t st,
                                           int L)
{
    return launch_lattice<true, 2, true>(precision, d_reps, d_index, n_ctas, threads, smem_bytes,
                                         args, st, L);
}

}  // namespace cg
