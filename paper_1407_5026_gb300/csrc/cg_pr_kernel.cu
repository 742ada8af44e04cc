// cg_pr_kernel.cu -- launches of the persistent parallel-rejection kernel
// (cg_pr_lattice.cuh) on the square lattice, single hops, both clocks; cubic
// lattices go to cg_pr_kernel3d.cu, two-electron hops to cg_pr_kernel_pair.cu.
#include "cg_pr_lattice.cuh"

namespace cg {

cudaError_t set_pr_smem_limit(int precision, int bytes, bool pair)
{
    cudaError_t e = set_pr3_smem_limit(precision, bytes, pair);
    if (e) return e;
    if (pair) return set_pr_pair_smem_limit(precision, bytes);
    e = set_lattice_limit<false, 2, false>(precision, bytes);
    return e ? e : set_lattice_limit<true, 2, false>(precision, bytes);
}

cudaError_t launch_pr_persistent(int precision, const DevReplica *d_reps, const int *d_index,
                                 int n_ctas, int threads, int smem_bytes, const RunArgs &args,
                                 cudaStream_t st, int L, int dim)
{
    // the square lattice's update needs L/2 columns, the cubic one's L
    if (threads < L / 2 || (dim == 3 && threads < L)) return cudaErrorInvalidValue;
    if (dim == 3)
        return launch_pr_persistent3(precision, d_reps, d_index, n_ctas, threads, smem_bytes,
                                     args, st, L);
    if (args.pair)
        return launch_pr_persistent_pair(precision, d_reps, d_index, n_ctas, threads, smem_bytes,
                                         args, st, L);
    return args.time_mode
               ? launch_lattice<true, 2, false>(precision, d_reps, d_index, n_ctas, threads,
                                                smem_bytes, args, st, L)
               : launch_lattice<false, 2, false>(precision, d_reps, d_index, n_ctas, threads,
                                                 smem_bytes, args, st, L);
}

}  // namespace cg
