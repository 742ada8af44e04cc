// cg_internal.h -- structures shared by the host side of libcg and its
// kernels.  Not part of the public ABI (include/cg.h is).
#pragma once

#include <cstddef>
#include <cstdint>

#include <cuda_runtime.h>

#include "../../include/cg.h"

namespace cg {

// Device-resident counters of one replica (written back at the end of every
// persistent launch; read by cg_read_state / cg_observables).
struct alignas(16) DevCounters {
    unsigned long long rounds;
    unsigned long long hops;
    unsigned long long attempts;
    unsigned long long evaluated;
    long long P;
    double energy;
    unsigned long long cycles_reject;
    unsigned long long cycles_update;
    unsigned long long refreshes;
    unsigned long long max_err_bits;   // max |eps - eps_ref| of the last refresh (binary64 bits)
    int status;                        // CG_OK, CG_ESTUCK or CG_ETIMEOUT
    float m_ema;                       // running mean of attempts per hop (chunk sizing)
    int trace_count;                   // points recorded
    int trace_cap;                     // trace capacity (0: no trace)
    double trace_next;                 // attempt count of the next trace point
    double trace_ratio;                // ratio between consecutive trace points
    double time;                       // stochastic time (CG_TIME_GAUSSIAN), else 0
    float rate;                        // attempts per hop of the last launch (0: none yet)
};

// Guide table of the tower: bucket b = x1 >> (32 - kGuideBits) holds the
// smallest vector index whose threshold is >= the bucket's first value (14
// bits), bit 15 set when a threshold falls strictly inside the bucket (one
// compare decides between that vector and the next) and bit 14 when two or
// more do (a scan finds the exact vector); see tower_lookup.
constexpr int kGuideBits = 12;
constexpr int kGuide = 1 << kGuideBits;

// Guide table of the lattice kernels but for two-electron hops on clusters
// (cg_pr_lattice.cuh): bucket
// b = x1 >> (32 - kLatGuideBits) holds v - lat_guide_base(V) when every x1 of
// the bucket selects the same vector v and that difference is in [0, 254],
// else 255 (the kernel then searches the thresholds between the bounds of
// x1's top kLatHintBits bits).  The vectors are ordered dy outer, dx inner, so
// the probable ones lie in the middle of the list: the base centres the 255
// representable ones there.
constexpr int kLatGuideBits = 14;
constexpr int kLatHintBits = 7;
__host__ __device__ inline int lat_guide_base(int V) { return V <= 255 ? 0 : (V - 255) / 2; }

// Everything one CTA needs to run one replica.
struct alignas(16) DevReplica {
    int L, N, H1, V;          // side, sites, folded extent L/2+1, hop vectors
    int words;                // occupation bitmask words, ceil(N/32)
    unsigned int magicL;      // y = umulhi(s, magicL) == s / L for s < N
    unsigned int key0, key1;  // Philox key (seed lo, seed hi)
    unsigned int replica;     // Philox counter word 3
    int dim;                  // 2 (square lattice) or 3 (cubic lattice)
    unsigned int pair_T;      // two-electron hops: a label pairs iff its word x3 < pair_T
    int pair_R;               // their offset bound |e| <= pair_R
    double nu, T, E;
    double negC0nu;           // -nu * sum_{t != s} 1/r_st (same for every s)
    double C0;                // sum_{t != s} 1/r_st
    double Gamma;             // N * Z (/ (1 - pair_T 2^-32)), the total proposal rate
    // tables (device)
    const double *tinv64;     // H1*H1, [fy*H1 + fx] = 1/sqrt(fx^2+fy^2), 0 at origin
    const float *tinv32;      // the same rounded to binary32
    const unsigned int *thr;  // V tower thresholds C_k - 1
    const int *disp;          // V packed hop vectors: (dx & 0xffff) | (dy << 16)
    const double *tinvd;      // V: 1/r of each hop vector (binary64)
    const double *tinv_r2_64; // cubic lattice: 1/r by r^2 = fx^2+fy^2+fz^2, 3 (L/2)^2 + 1
    const float *tinv_r2_32;  // entries (the folded table's values); null on the square one
    const unsigned short *guide; // kGuide entries
    const unsigned char *guide8; // 2^kLatGuideBits entries
    // state (device)
    void *eps;                // N binary64 (CG_FP64) or binary32 (CG_FP32)
    unsigned int *occ;        // occupation bitmask, bit s%32 of word s/32
    const double *phi;        // N site energies
    DevCounters *ctr;
    cg_hop *log;              // NULL, or n_hops entries for this replica
    cg_trace_point *trace;    // NULL, or ctr->trace_cap points
    // random-site geometry (CG_SITES_RANDOM; null otherwise)
    const double *G;          // N x N minimum-image 1/r, 0 on the diagonal
    const int *rguide;        // 16 ints per site: kRandomGuide layout
    const uint32_t *rw;       // per pair: C - 1
    const uint32_t *rj;       // per pair: random_partner_word
    const double2 *rgx;       // per pair: 1/r, E dx (minimum-image dx, binary64)
    int rguide_small;         // 1: every partner list holds at most 255 pairs
};

// Thread 0 at commit: record trace points whose attempt threshold the
// replica's attempt count has reached (several if one hop spans them).
__device__ __forceinline__ void trace_hop(const DevReplica &Rg, unsigned long long attempts,
                                          unsigned long long hops, long long P, double energy,
                                          int time_mode, double time)
{
    DevCounters *c = Rg.ctr;
    if (!Rg.trace || c->trace_count >= c->trace_cap || (double)attempts < c->trace_next) return;
    cg_trace_point pt;
    pt.attempts = attempts;
    pt.hops = hops;
    pt.P = P;
    pt.energy = energy;
    pt.time = time_mode ? time : __ddiv_rn((double)attempts, Rg.Gamma);
    Rg.trace[c->trace_count++] = pt;
    double next = c->trace_next;
    while (next <= (double)attempts) next = next * c->trace_ratio > next + 1.0 ? next * c->trace_ratio : next + 1.0;
    c->trace_next = next;
}

struct RunArgs {
    unsigned long long n_hops;     // hops every replica executes in this launch
    unsigned long long max_rounds; // rounds per hop before CG_ESTUCK
    unsigned long long log_offset; // index of this launch's first hop in each log
    unsigned long long hop_timeout_ns; // wall-clock limit of one hop
    unsigned long long hop_timeout_cyc; // the same in SM cycles at the peak clock
    unsigned int M;                // labels per round
    int toy;                       // constant-acceptance test mode
    int time_mode;                 // CG_TIME_DETERMINISTIC or CG_TIME_GAUSSIAN
    int pair;                      // 1: two-electron hops (the kPair instances)
    int smem_guide;                // random sites, one CTA: guide records in shared memory
    int *sched;                    // single hops, several CTAs per SM: the claim table of
                                   // launch_pr_schedule, or null (CTA b runs replica b)
    int n_sms;                     // SMs of the device (with sched)
    int guide_bits;                // log2 of the guide table's entries (LatLayout)
    int cluster_r2;                // cubic clusters: the update reads 1/r by r^2
    double toy_A0;
};

// Shared-memory carve-up of the persistent kernel (bytes, 16-aligned).
struct SmemLayout {
    int off_eps, off_tinv, off_occ, off_guide, off_thr, off_disp;
    int off_vr64, off_edx64, off_cv32, total;
};

__host__ __device__ inline int cg_align16(int x) { return (x + 15) & ~15; }

// tab_entries: (L/2+1)^dim entries of the folded 1/r table
__host__ __device__ inline SmemLayout smem_layout(int N, int tab_entries, int V, int words,
                                                  int real_bytes)
{
    SmemLayout s;
    int o = 0;
    s.off_eps = o;   o = cg_align16(o + N * real_bytes);
    s.off_tinv = o;  o = cg_align16(o + tab_entries * real_bytes);
    s.off_occ = o;   o = cg_align16(o + words * 4);
    s.off_guide = o; o = cg_align16(o + kGuide * 2);
    s.off_thr = o;   o = cg_align16(o + V * 4);
    s.off_disp = o;  o = cg_align16(o + V * 4);
    s.off_vr64 = o;  o = cg_align16(o + V * 8);
    s.off_edx64 = o; o = cg_align16(o + V * 8);
    s.off_cv32 = o;  o = cg_align16(o + V * 4);
    s.total = o;
    return s;
}

// Shared-memory carve-up of the lattice kernels but for two-electron hops on
// clusters (cg_pr_lattice.cuh), with a guide table of 2^gbits entries.
struct LatLayout {
    int off_eps, off_tinv, off_occ, off_guide, off_hint, off_thr, off_rec;
    int off_vr64, off_edx64, total;
};

__host__ __device__ inline LatLayout lat_layout(int N, int tab_entries, int V, int words,
                                                int real_bytes, int gbits)
{
    LatLayout s;
    int o = 0;
    s.off_eps = o;   o = cg_align16(o + N * real_bytes);
    s.off_tinv = o;  o = cg_align16(o + tab_entries * real_bytes);
    s.off_occ = o;   o = cg_align16(o + words * 4);
    s.off_guide = o; o = cg_align16(o + (1 << gbits));
    s.off_hint = o;  o = cg_align16(o + ((1 << kLatHintBits) + 1) * 2);
    s.off_thr = o;   o = cg_align16(o + V * 4);
    s.off_rec = o;   o = cg_align16(o + V * 8);
    s.off_vr64 = o;  o = cg_align16(o + V * 8);
    s.off_edx64 = o; o = cg_align16(o + V * 8);
    s.total = o;
    return s;
}

// Shared memory a kernel may not take dynamically: its static part (the
// cluster kernel's exchange slots take it past 2 KiB with two-electron hops).
inline int lat_static_bytes(bool pair) { return pair ? 3072 : 2048; }

// Guide bits of that kernel: a finer table sends fewer labels to the search
// (about 0.5% of x1's range at 14 bits, 1% at 13 for r_max = 8), so the
// largest of 14, 13 and 12 that costs no CTA per SM (228 KiB of shared memory,
// at most four CTAs of 256 threads by registers) and fits `most` bytes, the
// room the lattice is admitted by.  12 bits take less than smem_layout, so a
// lattice that fits that layout fits this one.
constexpr int kSmemPerCta = 227 * 1024;
inline int lat_guide_bits(int N, int tab_entries, int V, int words, int real_bytes, int most)
{
    auto total = [&](int b) { return lat_layout(N, tab_entries, V, words, real_bytes, b).total; };
    auto ctas = [&](int b) {
        const int c = (228 * 1024) / (total(b) + 3072);
        return c < 4 ? c : 4;
    };
    for (int b = kLatGuideBits; b > 12; --b)
        if (total(b) <= most && ctas(b) == ctas(12)) return b;
    return 12;
}

// Random sites (cg_pr_random.cu): the coupling matrix from the positions,
// eps from its definition, and the persistent binary64 PR kernel.
cudaError_t launch_g_build(const double *px, const double *py, int L, int N, double *G,
                           cudaStream_t st);
cudaError_t launch_eps_init_random(const DevReplica *d_rep, int N, cudaStream_t st);
cudaError_t launch_pr_random(const DevReplica *d_reps, const int *d_index, int n_ctas,
                             int threads, int smem_bytes, const RunArgs &args, cudaStream_t st);
cudaError_t set_pr_random_smem_limit(int bytes);
// The per-site record of a random-site partner list (16 ints, 64 bytes):
// [0] first pair of the list, [1] one past its last; [2], [3] the list's
// last running weight (lo, hi words); [4 + b/2] holds, in its low (b even)
// or high (b odd) 16 bits, b = 0..15, the offset from [0] of the pair that
// x1 = b 2^28 selects (the smallest m with b 2^28 < C_m; the last pair when
// none); [12..15] unused.  A label with x1 in bucket b = x1 >> 28 finds its
// pair in [start(b), min(start(b + 1), [1] - 1)], start(16) = [1].
// The offsets are 16 bits: the library refuses lists of 2^16 or more pairs.
constexpr int kRandomGuide = 16;
constexpr int kRandomBuckets = 16;
// A pair's partner (17 bits: N <= 131072) and, in the upper 15 bits, sign, exponent
// and six bits of 1/r + E dx, rounded up: the chain's first look at a label needs a
// bound on dH from below only.  Weight and this word take 8 bytes per pair.
constexpr uint32_t kPartnerMask = (1u << 17) - 1;
inline uint32_t random_partner_word(unsigned j, uint32_t cv_bits)
{
    const uint32_t up = cv_bits >> 31 ? cv_bits : cv_bits + kPartnerMask;
    return (up & ~kPartnerMask) | j;
}
// Sites whose eps a CTA of a C-CTA cluster owns: ceil(N / C) rounded up to a
// multiple of 32 (CTA rank owns [rank Nc, min(N, (rank + 1) Nc))).
__host__ __device__ inline int random_cluster_sites(int N, int C)
{
    return C <= 1 ? N : (((N + C - 1) / C + 31) / 32) * 32;
}
// Dynamic shared memory of a random-site CTA: its eps (binary64) and the
// whole occupation bitmask; with guide = true (one CTA per replica, every
// list below 256 pairs) also each site's guide record compacted to 32 bytes
// (kRandomGuideSmem): first pair, the last running weight (33 bits), the
// list's length (16 bits) and the 16 bucket starts as 8-bit offsets.
constexpr int kRandomGuideSmem = 32;
inline int random_smem_bytes(int N, int C = 1, bool guide = false)
{
    return cg_align16(random_cluster_sites(N, C) * 8) + cg_align16(((N + 31) / 32) * 4) +
           (guide ? N * kRandomGuideSmem : 0);
}
// The random-site chain on clusters of `cluster` (2, 4 or 8) CTAs per replica
// (cg_pr_random_cluster.cu); grid = n_reps * cluster CTAs of 256, 512 or 1024
// threads.
cudaError_t launch_pr_random_cluster(const DevReplica *d_reps, const int *d_index, int n_reps,
                                     int cluster, int threads, int smem_bytes,
                                     const RunArgs &args, cudaStream_t st);

// Claim table of a launch whose CTAs share SMs: order[count] (replica positions
// by falling attempts per hop), claimed[count], slots[kSchedSms].
constexpr int kSchedSms = 256;
inline size_t sched_bytes(int count) { return sizeof(int) * (2 * (size_t)count + kSchedSms); }
// Fills it from the counters; one small CTA before the persistent launch.
cudaError_t launch_pr_schedule(const DevReplica *d_reps, const int *d_index, int count,
                               int *sched, cudaStream_t st);

// Launchers (defined in the .cu files).
cudaError_t launch_pr_persistent(int precision, const DevReplica *d_reps,
                                 const int *d_index, int n_ctas, int threads,
                                 int smem_bytes, const RunArgs &args,
                                 cudaStream_t st, int L, int dim);
// The cubic-lattice instances (cg_pr_kernel3d.cu).
cudaError_t launch_pr_persistent3(int precision, const DevReplica *d_reps, const int *d_index,
                                  int n_ctas, int threads, int smem_bytes, const RunArgs &args,
                                  cudaStream_t st, int L);
cudaError_t set_pr3_smem_limit(int precision, int bytes, bool pair);
// The cubic lattice with two-electron hops (cg_pr_kernel3d_pair.cu).
cudaError_t launch_pr_persistent3_pair(int precision, const DevReplica *d_reps,
                                       const int *d_index, int n_ctas, int threads,
                                       int smem_bytes, const RunArgs &args, cudaStream_t st,
                                       int L);
cudaError_t set_pr3_pair_smem_limit(int precision, int bytes);
// The two-electron-hop instances (cg_pr_kernel_pair.cu): square lattice, one
// CTA per replica.
cudaError_t launch_pr_persistent_pair(int precision, const DevReplica *d_reps,
                                      const int *d_index, int n_ctas, int threads,
                                      int smem_bytes, const RunArgs &args, cudaStream_t st,
                                      int L);
cudaError_t set_pr_pair_smem_limit(int precision, int bytes);
// ... and with the stochastic clock (cg_pr_kernel_pair_time.cu).
cudaError_t launch_pr_persistent_pair_time(int precision, const DevReplica *d_reps,
                                           const int *d_index, int n_ctas, int threads,
                                           int smem_bytes, const RunArgs &args, cudaStream_t st,
                                           int L);
cudaError_t set_pr_pair_time_smem_limit(int precision, int bytes);
// The same chain over a thread-block cluster of `cluster` CTAs per replica
// (eps split by rows, or by z-planes on the cubic lattice, dim = 3);
// grid = n_reps * cluster CTAs.
cudaError_t launch_pr_cluster(int precision, const DevReplica *d_reps, const int *d_index,
                              int n_reps, int cluster, int threads, int smem_bytes,
                              const RunArgs &args, cudaStream_t st, int L, int dim);
// Its two-electron-hop instances (cg_pr_cluster_pair.cu).
cudaError_t launch_pr_cluster_pair(int precision, const DevReplica *d_reps, const int *d_index,
                                   int n_reps, int cluster, int threads, int smem_bytes,
                                   const RunArgs &args, cudaStream_t st, int L, int dim);
cudaError_t launch_eps_init(const DevReplica *d_rep, int N, int tab_entries, int words,
                            int precision, cudaStream_t st);
cudaError_t launch_refresh_fp64(const DevReplica *d_reps, const int *d_index, int count, int N,
                                int tab_entries, int words, cudaStream_t st);
cudaError_t launch_debug_philox(const uint32_t *ctr, const uint32_t *key,
                                uint32_t *out, int n, cudaStream_t st);
cudaError_t launch_debug_exp(const double *x, double *out, int n, cudaStream_t st);
cudaError_t launch_debug_gauss(const uint64_t *seed, const uint32_t *rep, const uint64_t *hop,
                               double *z, int n, cudaStream_t st);
cudaError_t launch_debug_tower(const DevReplica *d_rep, const unsigned short *guide,
                               const unsigned *thr, int V, const uint32_t *x1, int *out, int n,
                               cudaStream_t st);
cudaError_t set_pr_smem_limit(int precision, int bytes, bool pair);
int microbench(int kind, int device, double *result);
// Histogram of eps (binary64 or binary32 by precision) of `count` replicas
// starting at d_reps, added to the nbins counters at out.
cudaError_t launch_eps_histogram(const DevReplica *d_reps, int count, int max_N, int precision,
                                 int nbins, double lo, double scale, unsigned long long *out,
                                 cudaStream_t st);
cudaError_t launch_reset_refresh_err(const DevReplica *d_reps, const int *d_index, int R,
                                     cudaStream_t st);
// log2 of the factor applied to 1/r before its binary16 split (cubic lattice)
constexpr int kTcF16Log2Scale = 10;

// Tensor-core refresh of R <= 512 binary32 replicas of one L and dimension
// (dim 2: N = L^2, dim 3: N = L^3; N % 128 == 0).  d_tab: the folded table's
// two-term split (H1^dim entries; BF16 of 1/r for dim 2, binary16 of
// 2^kTcF16Log2Scale / r for dim 3).  d_scratch: refresh_tc_scratch_bytes(N, R)
// bytes (the S image and the K-split partial sums), 256-byte aligned.
cudaError_t launch_refresh_tc(const DevReplica *d_reps, const int *d_index, int R, int L,
                              int dim, const uint32_t *d_tab, unsigned char *d_scratch,
                              int *d_err, cudaStream_t st);
int refresh_tc_smem_bytes(int R_pad, int tab_entries);
// The FFT refresh of R binary32 replicas of one L that refresh_fft_size_ok or
// refresh_fft_plane takes (dim 2 or 3; cg_refresh_fft.cu): d_ghat holds DFT(g)/N (N floats), d_tw the L
// twiddles exp(-2 pi i k / L), d_buf refresh_fft_buffer_bytes.
cudaError_t launch_refresh_fft(const DevReplica *d_reps, const int *d_index, int R, int L,
                               int dim, const float *d_ghat, const float2 *d_tw, float2 *d_buf,
                               cudaStream_t st);
size_t refresh_fft_buffer_bytes(int N, int R);
bool refresh_fft_size_ok(int L);                   // 2^m (4..1024), 3 2^m (6..192)
bool refresh_fft_plane(int L, int dim);            // the per-plane transforms' sides
int refresh_tc_ksplit(int N, int dim);
int refresh_tc_max_replicas(int dim);   // replicas per launch
size_t refresh_tc_scratch_bytes(int N, int dim, int R);

}  // namespace cg
