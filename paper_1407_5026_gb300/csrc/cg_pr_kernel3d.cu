// cg_pr_kernel3d.cu -- launches of the persistent parallel-rejection kernel
// (cg_pr_lattice.cuh) on the L x L x L cubic lattice, single hops, both clocks
// (two-electron hops: cg_pr_kernel3d_pair.cu).
#include "cg_pr_lattice.cuh"

namespace cg {

cudaError_t set_pr3_smem_limit(int precision, int bytes, bool pair)
{
    if (pair) return set_pr3_pair_smem_limit(precision, bytes);
    const cudaError_t e = set_lattice_limit<false, 3, false>(precision, bytes);
    return e ? e : set_lattice_limit<true, 3, false>(precision, bytes);
}

cudaError_t launch_pr_persistent3(int precision, const DevReplica *d_reps, const int *d_index,
                                  int n_ctas, int threads, int smem_bytes, const RunArgs &args,
                                  cudaStream_t st, int L)
{
    if (args.pair)
        return launch_pr_persistent3_pair(precision, d_reps, d_index, n_ctas, threads, smem_bytes,
                                          args, st, L);
    return args.time_mode
               ? launch_lattice<true, 3, false>(precision, d_reps, d_index, n_ctas, threads,
                                                smem_bytes, args, st, L)
               : launch_lattice<false, 3, false>(precision, d_reps, d_index, n_ctas, threads,
                                                 smem_bytes, args, st, L);
}

}  // namespace cg
