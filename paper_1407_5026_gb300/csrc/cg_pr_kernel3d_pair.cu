// cg_pr_kernel3d_pair.cu -- launches of the persistent parallel-rejection
// kernel (cg_pr_lattice.cuh) with two-electron hops on the L x L x L cubic
// lattice, both clocks.
#include "cg_pr_lattice.cuh"

namespace cg {

cudaError_t set_pr3_pair_smem_limit(int precision, int bytes)
{
    const cudaError_t e = set_lattice_limit<false, 3, true>(precision, bytes);
    return e ? e : set_lattice_limit<true, 3, true>(precision, bytes);
}

cudaError_t launch_pr_persistent3_pair(int precision, const DevReplica *d_reps,
                                       const int *d_index, int n_ctas, int threads,
                                       int smem_bytes, const RunArgs &args, cudaStream_t st,
                                       int L)
{
    return args.time_mode
               ? launch_lattice<true, 3, true>(precision, d_reps, d_index, n_ctas, threads,
                                               smem_bytes, args, st, L)
               : launch_lattice<false, 3, true>(precision, d_reps, d_index, n_ctas, threads,
                                                smem_bytes, args, st, L);
}

}  // namespace cg
