// cg_pr_lattice.cuh -- the persistent parallel-rejection kernel for single
// hops on one CTA per replica (square lattice: cg_pr_kernel.cu, cubic
// lattice: cg_pr_kernel3d.cu).  Two-electron hops run on cg_pr_persistent.cuh.
//
// One CTA runs one disorder replica for a whole launch.  Its local energies
// eps (N values), the folded minimum-image 1/r table, the occupation bitmask
// and the tower live in shared memory; global memory is touched only to load
// the state at the start and store it at the end.
//
// Per executed hop (mixed PR algorithm, section "Hopping conduction in the
// Coulomb glass", steps 1-3):
//   rounds r = 0, 1, ...: the M labels of a round are evaluated in chunks of
//   C labels in increasing order, dealt to the warps in blocks of 32 or 64.  Label k draws Philox(key = seed, ctr =
//   (k, r lo, r hi, replica)) -> site i from word 0, hop vector from word 1 by
//   tower sampling, acceptance variate from word 2 (step 1 and the three
//   random numbers per label of the GPU paragraph); theta = n_i (1 - n_j) and
//   the Metropolis test on dH = eps_j - eps_i - 1/r_ij - E dx (step 2, Eq. 2).
//   A chunk with no accept costs one block-wide OR barrier; the first chunk
//   with an accept gives the lowest accepting label q, so the hop equals the
//   serial rejection chain's on the same random numbers.
//   Commit (step 3a/3c): flip n_i, n_j, P += dx, attempts += (p-1)M + q.
//   Update (step 3b): eps_l += 1/r_lj - 1/r_li for every l, with the table
//   holding 0 at the origin so l = i and l = j need no special case.
//
// What bounds it (L = 128, T = 0.01, 304 replicas, 512 threads, two CTAs per
// SM): a label costs about 85 warp instructions per 32 labels, 47 of them on
// the integer pipe and 24 on the multiplier, and time goes with their sum
// (Philox alone is 40 of the 71); alone it runs at 266 G labels/s, 470 G being
// the generator by itself.  More warps change nothing.  So the per-label work
// was cut: only a label whose theta holds and whose dH is below the cut (one in
// a few hundred) reaches the exponential, the near-tie test and, in binary64,
// the slow binary64 pipe (its dH is first bounded from the energies' high
// words); the tower is one byte of a 16,384-entry table for 99.5% of the words
// x1; every lane runs the loads without a branch.  A chunk with an accept needs
// no second barrier: the accepting warps write their proposals and lower a
// shared minimum before the one that ends the chunk.
// Measured with the kernel this replaces (ms per run call, same chains):
// L = 128 binary32 12.12 -> 11.10, binary64 (152 replicas) 2.95 -> 2.40;
// L = 32 to 96 mixed 3.16 -> 1.78; 32^3 2.24 -> 2.06.
#pragma once

#include <type_traits>

#include "cg_pr_update.cuh"

namespace cg {

// b of the chunk rule C ~ sqrt(m b)
constexpr float kLatChunkCost = 256.0f;

// Hop vector dx of a packed displacement word (see rec below): with a
// power-of-two L the low field is dx mod L, otherwise dx | dy << 16 (square)
// or 10-bit fields (cubic).
template <bool kPow2, int kDim>
__device__ __forceinline__ void vec_fields(unsigned w, int L, int log2L, int &dx, int &dy)
{
    if (kPow2) {
        dx = (int)(w & (unsigned)(L - 1));
        dx -= (dx >= (L >> 1)) ? L : 0;
        dy = (int)((w >> log2L) & (unsigned)(L - 1));
        dy -= (dy >= (L >> 1)) ? L : 0;
    } else if (kDim == 3) {
        dx = (int)(w << 22) >> 22;
        dy = (int)(w << 12) >> 22;
    } else {
        dx = (int)(short)(w & 0xffffu);
        dy = (int)w >> 16;
    }
}

// The displacement word of a packed hop vector dxy (cg_internal.h).
template <bool kPow2, int kDim>
__device__ __forceinline__ unsigned vec_word(int dxy, int L, int log2L)
{
    if (!kPow2) return (unsigned)dxy;
    const unsigned m = (unsigned)(L - 1);
    if (kDim == 3) {
        const unsigned dx = (unsigned)((dxy << 22) >> 22) & m, dy = (unsigned)((dxy << 12) >> 22) & m,
                       dz = (unsigned)(dxy >> 20) & m;
        return (((dz << log2L) | dy) << log2L) | dx;
    }
    const unsigned dx = (unsigned)(int)(short)(dxy & 0xffff) & m, dy = (unsigned)(dxy >> 16) & m;
    return (dy << log2L) | dx;
}

// Site i displaced by the vector word w.  Power-of-two L: i + w is right in
// the x field, and (i with x cleared) + w in the y field (its x field is dx
// alone and carries nothing), (i with x, y cleared) + w in the z field.
template <bool kPow2, int kDim>
__device__ __forceinline__ unsigned hop_target(unsigned i, unsigned w, int L, int log2L,
                                               unsigned N, unsigned magic)
{
    if (kPow2) {
        const unsigned mx = (unsigned)(L - 1);
        if (kDim == 3) {
            const unsigned my = mx << log2L, mz = my << log2L;
            return ((i + w) & mx) | (((i & ~mx) + w) & my) | (((i & mz) + w) & mz);
        }
        return ((i + w) & mx) | (((i & ~mx) + w) & (N - 1u) & ~mx);
    }
    const unsigned uL = (unsigned)L;
    if (kDim == 3) {
        const unsigned q = __umulhi(i, magic), z = __umulhi(q, magic);
        unsigned xj = i - q * uL + (unsigned)((int)(w << 22) >> 22);
        unsigned yj = q - z * uL + (unsigned)((int)(w << 12) >> 22);
        unsigned zj = z + (unsigned)((int)w >> 20);
        // wrap without a branch: below 0 the unsigned value is huge, at or
        // above L the value less L is the smaller one
        xj = min(min(xj, xj + uL), xj - uL);
        yj = min(min(yj, yj + uL), yj - uL);
        zj = min(min(zj, zj + uL), zj - uL);
        return (zj * uL + yj) * uL + xj;
    }
    const unsigned yi = __umulhi(i, magic);
    unsigned xj = i - yi * uL + (unsigned)(int)(short)(w & 0xffffu);
    unsigned yj = yi + (unsigned)((int)w >> 16);
    xj = min(min(xj, xj + uL), xj - uL);
    yj = min(min(yj, yj + uL), yj - uL);
    return yj * uL + xj;
}

// The arrays of LatLayout in shared memory:
//   occ     occupation bitmask
//   guide   2^gbits bytes: vector index - vbase, 255: search
//   hint    2^kLatHintBits + 1 search bounds (16 bits)
//   thr     thresholds
//   rec     per vector: 1/r_v + E dx_v (binary32 bits), displacement word
//   vr64, edx64   1/r_v and E dx_v (binary64)

// The smallest vector v with x1 <= thr[v], by bisection between the bounds of
// x1's top bits; false for a null proposal (x1 above the last threshold).
__device__ __forceinline__ bool lat_search(const LatLayout &S, uint32_t x1, unsigned thr_last,
                                           int &v)
{
    if (x1 > thr_last) return false;
    const unsigned b = x1 >> (32 - kLatHintBits);
    int lo = sm<unsigned short>(S.off_hint, b), hi = sm<unsigned short>(S.off_hint, b + 1);
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (x1 <= sm<unsigned>(S.off_thr, mid))
            hi = mid;
        else
            lo = mid + 1;
    }
    v = lo;
    return true;
}

// Binary32 value of the high word of a normal binary64 x: truncated to 20
// mantissa bits.  ok is false unless 2^-126 <= |x| < 2^60 (0 included), where
// the word shift does not give x's value.
__device__ __forceinline__ float hi_to_f32(int hi, bool &ok)
{
    ok = ((unsigned)hi << 1) - (897u << 21) < ((1083u - 897u) << 21);
    const unsigned sh = (unsigned)hi * 8u + 0x40000000u;
    return __uint_as_float((sh & 0x7fffffffu) | ((unsigned)hi & 0x80000000u));
}

// What a label's evaluation reads that stays fixed over a launch.
struct LatConst {
    LatLayout S;
    Cand *cand;                // per warp: its lowest accepting label's proposal
    int L, log2L, vbase, vlast, gshift, warp, lane;
    unsigned N, magic, M, thr_last;
    uint32_t key0, key1;
    float cut, invTf;
    double T;
};

// eps_s as binary64.
template <typename Store>
__device__ __forceinline__ double lat_energy(int off_eps, unsigned s)
{
    if constexpr (std::is_same<Store, long long>::value)
        return fix_to_double(sm<long long>(off_eps, s));
    else
        return (double)sm<Store>(off_eps, s);
}

// The warp's block of 32 NL labels from kb on: label kb + 32 n + lane, n < NL.
// Only labels whose theta holds and whose dH is below the cut go through the
// accept test; the lowest accepting lane writes the warp's candidate and
// lowers the CTA's best label.  True when the block holds an accept.
// Store: the type of the energies in shared memory (long long: binary64 in
// fixed point).
template <typename Store, bool kPow2, int kDim, int NL>
__device__ __forceinline__ bool lat_eval(const LatConst &K, unsigned kb, const PhiloxPrefix &PP,
                                         unsigned *best)
{
    constexpr bool kF64 = sizeof(Store) == 8, kFix = std::is_same<Store, long long>::value;
    uint32_t x1[NL], x2[NL];
    unsigned si[NL], sj[NL];
    int v[NL];
    float cv[NL], d[NL];
    bool on[NL], cand[NL];
    bool odd = false;
#pragma unroll
    for (int n = 0; n < NL; ++n) {
        const unsigned k = kb + 32u * (unsigned)n + (unsigned)K.lane;
        uint32_t x[4];
        philox_finish(k, PP, K.key0, K.key1, x);
        x1[n] = x[1];
        x2[n] = x[2];
        si[n] = kPow2 ? (x[0] >> (32 - kDim * K.log2L)) : __umulhi(x[0], K.N);
        const unsigned wi = sm<unsigned>(K.S.off_occ, si[n] >> 5);
        on[n] = ((wi >> (si[n] & 31u)) & 1u) && k < K.M;
        const int g = (int)sm<unsigned char>(K.S.off_guide, x[1] >> K.gshift);
        odd |= on[n] && g == 255;
        v[n] = g + K.vbase;
    }
    // a few buckets leave the vector to a search
    if (odd) {
#pragma unroll
        for (int n = 0; n < NL; ++n)
            if (on[n] && v[n] == 255 + K.vbase) on[n] = lat_search(K.S, x1[n], K.thr_last, v[n]);
    }
    // every lane runs the rest (its addresses are valid whatever theta is):
    // branches around the loads cost more than the loads
#pragma unroll
    for (int n = 0; n < NL; ++n) {
        v[n] = min(v[n], K.vlast);               // 255 of a label that is off
        const uint2 rc = sm<uint2>(K.S.off_rec, v[n]);
        cv[n] = __uint_as_float(rc.x);
        sj[n] = hop_target<kPow2, kDim>(si[n], rc.y, K.L, K.log2L, K.N, K.magic);
        const unsigned wj = sm<unsigned>(K.S.off_occ, sj[n] >> 5);
        const bool theta = on[n] && !((wj >> (sj[n] & 31u)) & 1u);
        if constexpr (kFix) {
            // the high words: units of 2^-28, cut and rounded by at most
            // 2^-28 + 2^-22 each below 4; the cut's slack covers it
            const float fi = __int2float_rn(sm<int>(K.S.off_eps, 2 * si[n] + 1));
            const float fj = __int2float_rn(sm<int>(K.S.off_eps, 2 * sj[n] + 1));
            d[n] = fmaf(fj - fi, 0x1p-28f, -cv[n]);
            cand[n] = theta && d[n] < K.cut;
        } else if constexpr (kF64) {
            bool oi, oj;
            const float fi = hi_to_f32(sm<int>(K.S.off_eps, 2 * si[n] + 1), oi);
            const float fj = hi_to_f32(sm<int>(K.S.off_eps, 2 * sj[n] + 1), oj);
            d[n] = (fj - fi) - cv[n];
            cand[n] = theta &&
                      (fmaf(fabsf(fi) + fabsf(fj), -0x1p-19f, d[n]) < K.cut || !oi || !oj);
        } else {
            d[n] = __fsub_rn(__fsub_rn(sm<float>(K.S.off_eps, sj[n]), sm<float>(K.S.off_eps, si[n])),
                             cv[n]);
            cand[n] = theta && d[n] < K.cut;
        }
    }
    if (!__any_sync(0xffffffffu, cand[0] || cand[NL - 1])) return false;
    // the accept test of the few labels near or below zero
    bool acc[NL];
    double dE[NL];
#pragma unroll
    for (int n = 0; n < NL; ++n) {
        dE[n] = 0.0;
        if constexpr (kF64) {
            acc[n] = cand[n] && metropolis_label<double>(
                                    lat_energy<Store>(K.S.off_eps, si[n]),
                                    lat_energy<Store>(K.S.off_eps, sj[n]),
                                    sm<double>(K.S.off_vr64, v[n]), sm<double>(K.S.off_edx64, v[n]),
                                    cv[n], x2[n], K.T, K.invTf, dE[n]);
        } else {
            acc[n] = cand[n] && metropolis_f32(d[n], x2[n], K.invTf);
            if (cand[n] && fabsf(d[n]) < 1e-5f)      // near tie: decided in binary64
                acc[n] = metropolis_label<float>(
                    sm<float>(K.S.off_eps, si[n]), sm<float>(K.S.off_eps, sj[n]),
                    sm<double>(K.S.off_vr64, v[n]), sm<double>(K.S.off_edx64, v[n]), cv[n], x2[n],
                    K.T, K.invTf, dE[n]);
        }
    }
    // the warp's lowest accepting label: the first of the NL with an accept,
    // then the lowest lane (NL is 1 or 2)
    const unsigned b0 = __ballot_sync(0xffffffffu, acc[0]);
    const unsigned b1 = NL > 1 ? __ballot_sync(0xffffffffu, acc[NL - 1]) : 0u;
    if (!(b0 | b1)) return false;
    if (K.lane == __ffs(b0 ? b0 : b1) - 1) {
        Cand c;
        c.i = b0 ? si[0] : si[NL - 1];
        c.j = b0 ? sj[0] : sj[NL - 1];
        c.dxy = (int)sm<uint2>(K.S.off_rec, b0 ? v[0] : v[NL - 1]).y;
        c.dE = b0 ? dE[0] : dE[NL - 1];
        // binary32: the executed hop's dH is the binary32 one, widened
        if (!kF64 && c.dE == 0.0) c.dE = (double)(b0 ? d[0] : d[NL - 1]);
        K.cand[K.warp] = c;
        atomicMin(best, kb + (b0 ? 0u : 32u * (unsigned)(NL - 1)) + (unsigned)K.lane);
    }
    return true;
}

// Constant-acceptance test mode: label kb + lane accepts iff its variate is
// below A0.
template <bool kPow2, int kDim>
__device__ __forceinline__ bool lat_eval_toy(const LatConst &K, unsigned kb, const PhiloxPrefix &PP,
                                             int V, double A0, unsigned *best)
{
    const unsigned k = kb + (unsigned)K.lane;
    uint32_t x[4];
    philox_finish(k, PP, K.key0, K.key1, x);
    const bool acc = k < K.M && d_mul(d_add((double)x[2], 0.5), 0x1p-32) < A0;
    const unsigned b = __ballot_sync(0xffffffffu, acc);
    if (!b) return false;
    if (K.lane == __ffs(b) - 1) {
        // the proposal, for the log
        int v = V - 1;
        lat_search(K.S, x[1], K.thr_last, v);
        Cand c;
        c.i = kPow2 ? (x[0] >> (32 - kDim * K.log2L)) : __umulhi(x[0], K.N);
        c.dxy = (int)sm<uint2>(K.S.off_rec, v).y;
        c.j = hop_target<kPow2, kDim>(c.i, (unsigned)c.dxy, K.L, K.log2L, K.N, K.magic);
        c.dE = 0.0;
        K.cand[K.warp] = c;
        atomicMin(best, k);
    }
    return true;
}

// The replica position this CTA runs: the first CTA on an SM takes one of the
// heavier half of the order, the second the lighter one that matches it, so the
// SMs' sums of attempts come out close (304 replicas of L = 128 at T = 0.01:
// the largest sum is 1.10 of the mean; 1.32 in replica order, and the launch
// lasts as long as its slowest SM).  The SM only sets the preferred position: a
// taken one passes on to the next, so every position is run exactly once
// wherever the CTAs land.
__device__ __forceinline__ int claim_replica(int *sched, int count, int n_sms)
{
    unsigned sm;
    asm volatile("mov.u32 %0, %%smid;" : "=r"(sm));
    const int *order = sched;
    int *claimed = sched + count, *slots = sched + 2 * count;
    const int r = (int)(sm % (unsigned)n_sms);
    const int slot = atomicAdd(&slots[r], 1);
    const int f = (slot >> 1) * n_sms + r;
    int pos = (slot & 1) ? count - 1 - f : f;
    if (pos < 0 || pos >= count) pos = r % count;
    for (int t = 0; t < count; ++t) {
        if (atomicExch(&claimed[pos], 1) == 0) break;
        pos = pos + 1 < count ? pos + 1 : 0;
    }
    return order[pos];
}

template <typename Real, int kThreads, int kLog2L, bool kTime, int kDim = 2>
__global__ void __launch_bounds__(kThreads, (kThreads >= 1024 ? 1 : 1024 / kThreads))
pr_lattice(const DevReplica *__restrict__ reps, const int *__restrict__ index, RunArgs a)
{
    constexpr bool kPow2 = kLog2L >= 0;
    constexpr bool kF64 = sizeof(Real) == 8;
    // the fixed-point form of binary64 energies (binary32 has none)
    using Fix = typename std::conditional<kF64, long long, Real>::type;
    // L fixed at compile time: 2^kLog2L (kLog2L > 0), or -kLog2L, an even L
    // that is not a power of two (kLog2L < -1); 0 when L is read at run time
    constexpr int kFixL = kLog2L > 0 ? (1 << kLog2L) : (kLog2L < -1 ? -kLog2L : 0);
    // the thread that keeps the books: lane 0 of the last warp, which has no
    // labels of its own when a chunk is smaller than the CTA
    constexpr int kBook = kThreads - 32, kWarps = kThreads / 32;
    __shared__ Cand s_cand[kWarps];
    __shared__ unsigned s_best[2];
    // step-3c deviates of the next hops (CG_TIME_GAUSSIAN): the last warp
    // draws 32 at a time, one per lane
    __shared__ double s_z[kTime ? 32 : 1];
    __shared__ struct {
        unsigned long long hops, attempts, evaluated, cyc_rej, cyc_upd, zbase, hops0, attempts0;
        long long P, t0;
        double energy, time;
        cg_hop *log;
        int tracing;
    } s_c;

    __shared__ int s_pos;
    if (threadIdx.x == 0)
        s_pos = a.sched ? claim_replica(a.sched, (int)gridDim.x, a.n_sms) : (int)blockIdx.x;
    __syncthreads();
    const DevReplica &Rg = reps[index[s_pos]];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int L = kFixL ? kFixL : Rg.L;
    const int N = kDim == 3 ? L * L * L : L * L, H1 = L / 2 + 1, words = (N + 31) / 32;
    const int ntab = kDim == 3 ? H1 * H1 * H1 : H1 * H1;
    const int V = Rg.V;
    // floor(s / L) = umulhi(s, floor(2^32 / L) + 1) for the site indices used;
    // the host computes the same multiplier for run-time L
    const unsigned magic = kPow2  ? 0u
                           : kFixL ? (unsigned)(4294967296ull / (unsigned long long)kFixL + 1ull)
                                   : Rg.magicL;
    const int log2L = kLog2L > 0 ? kLog2L : __ffs(L) - 1;   // used when L is a power of two
    const uint32_t key0 = Rg.key0, key1 = Rg.key1, rep = Rg.replica;
    const double T = Rg.T;
    const float invTf = (float)(1.0 / T);

    const LatLayout lay = lat_layout(N, ntab, V, words, (int)sizeof(Real), a.guide_bits);
    const int vbase = lat_guide_base(V);
    const int gshift = 32 - a.guide_bits;

    // ---- stage the replica into shared memory ----
    {
        const Real *eps_g = reinterpret_cast<const Real *>(Rg.eps);
        for (int l = tid; l < N; l += kThreads) sm<Real>(lay.off_eps, l) = eps_g[l];
        const Real *tab_g = kF64 ? reinterpret_cast<const Real *>(Rg.tinv64)
                                 : reinterpret_cast<const Real *>(Rg.tinv32);
        for (int l = tid; l < ntab; l += kThreads) sm<Real>(lay.off_tinv, l) = tab_g[l];
        for (int l = tid; l < words; l += kThreads) sm<unsigned>(lay.off_occ, l) = Rg.occ[l];
        // the device table has 2^kLatGuideBits entries; a coarser bucket
        // holds its entries' common value, or 255
        const int per = 1 << (kLatGuideBits - a.guide_bits);
        for (int b = tid; b < (1 << a.guide_bits); b += kThreads) {
            unsigned char g = Rg.guide8[b * per];
            for (int e = 1; e < per; ++e)
                if (Rg.guide8[b * per + e] != g) g = 255;
            sm<unsigned char>(lay.off_guide, b) = g;
        }
        for (int l = tid; l < V; l += kThreads) {
            const int dxy = Rg.disp[l];
            // dx of the packed vector (10-bit fields on the cubic lattice)
            const int dx = kDim == 3 ? (dxy << 22) >> 22 : (int)(short)(dxy & 0xffff);
            const double edx = d_mul(Rg.E, (double)dx);   // E * dx, as in the serial chain
            sm<unsigned>(lay.off_thr, l) = Rg.thr[l];
            sm<double>(lay.off_vr64, l) = Rg.tinvd[l];
            sm<double>(lay.off_edx64, l) = edx;
            // one rounding to binary32
            sm<uint2>(lay.off_rec, l) = make_uint2(
                __float_as_uint((float)d_add(Rg.tinvd[l], edx)), vec_word<kPow2, kDim>(dxy, L, log2L));
        }
        // hint[b] = smallest v with thr[v] >= b 2^(32 - kLatHintBits)
        for (int b = tid; b <= (1 << kLatHintBits); b += kThreads) {
            int lo = 0, hi = V - 1;
            const unsigned long long x = (unsigned long long)b << (32 - kLatHintBits);
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (x <= Rg.thr[mid])
                    hi = mid;
                else
                    lo = mid + 1;
            }
            sm<unsigned short>(lay.off_hint, b) = (unsigned short)lo;
        }
    }
    unsigned long long rounds = Rg.ctr->rounds;
    float m_ema = Rg.ctr->m_ema > 0.f ? Rg.ctr->m_ema : 64.0f;
    if (tid == kBook) {
        const DevCounters *cnt = Rg.ctr;
        s_c.log = Rg.log;
        s_c.tracing = Rg.trace != nullptr;
        s_c.hops = cnt->hops;
        s_c.attempts = cnt->attempts;
        s_c.hops0 = cnt->hops;
        s_c.attempts0 = cnt->attempts;
        s_c.evaluated = cnt->evaluated;
        s_c.P = cnt->P;
        s_c.energy = cnt->energy;
        s_c.time = cnt->time;
        s_c.cyc_rej = 0;
        s_c.cyc_upd = 0;
        s_c.zbase = ~0ull;
        s_best[0] = s_best[1] = 0xffffffffu;
    }
    int status = CG_OK;
    __syncthreads();

    const unsigned M = a.M;
    const unsigned thr_last = sm<unsigned>(lay.off_thr, V - 1);
    // dH above which no acceptance variate accepts, with a margin: binary32
    // variates are at least 2^-24 (ln: -16.64), binary64 ones 2^-33, and the
    // binary64 test calls e^y zero below y = -23.  The binary32 form decides
    // |dH| < 1e-5 apart.  The binary64 bound leaves room for cv's rounding.
    const float cut = kF64 ? (float)(23.1 * T + (8.0 + fabs(Rg.E) * (double)(L / 2)) * 0x1p-21)
                           : fmaxf((float)(17.0 * T), 1.1e-5f);

    // binary64: the energies and the table in fixed point where that is exact
    // for every one of them (the configurations' W = 1 and 2 at half filling;
    // a W that is no short binary fraction leaves small energies finer bits)
    bool fixed = false;
    if constexpr (kF64) {
        // from 1024 sites on: below, the update waits for latency, not for the
        // binary64 pipe, and the decoding costs more (L = 24: 3.4 against 3.2 us
        // a hop, L = 32: 2.95 and 2.99, L = 64: 2.9 and 4.2)
        bool ok = N >= 1024;
        for (int l = tid; ok && l < N; l += kThreads) fix_from_double(sm<double>(lay.off_eps, l), ok);
        for (int l = tid; ok && l < ntab; l += kThreads)
            fix_from_double(sm<double>(lay.off_tinv, l), ok);
        fixed = !__syncthreads_or(!ok);
        if (fixed) {
            for (int l = tid; l < N; l += kThreads)
                sm<long long>(lay.off_eps, l) = fix_from_double(sm<double>(lay.off_eps, l), ok);
            for (int l = tid; l < ntab; l += kThreads)
                sm<long long>(lay.off_tinv, l) = fix_from_double(sm<double>(lay.off_tinv, l), ok);
            __syncthreads();
        }
    }

    LatConst K;
    K.S = lay; K.cand = s_cand;
    K.L = L; K.log2L = log2L; K.vbase = vbase; K.vlast = V - 1; K.gshift = gshift;
    K.warp = warp; K.lane = lane;
    K.N = (unsigned)N; K.magic = magic; K.M = M; K.thr_last = thr_last;
    K.key0 = key0; K.key1 = key1;
    K.cut = cut; K.invTf = invTf; K.T = T;

    unsigned par = 0;
    for (unsigned long long h = 0; h < a.n_hops; ++h) {
        if (kTime && warp == kWarps - 1) {
            // the books are this warp's own; its lane 0 has written them
            __syncwarp();
            const unsigned long long hcur = s_c.hops;
            if (hcur < s_c.zbase || hcur - s_c.zbase >= 32ull) {
                s_z[lane] = cg_gauss(key0, key1, rep, hcur + (unsigned long long)lane);
                __syncwarp();
                if (lane == 0) s_c.zbase = hcur;
                __syncwarp();
            }
        }
        if (tid == kBook) s_c.t0 = clock64();
        // labels per chunk ~ sqrt(m b) for m expected labels and a chunk's fixed
        // cost (the barrier and the warps' imbalance before it) worth b/2
        // labels: nb = 2 or 1 blocks of 64 labels per warp when that exceeds
        // blockDim, else one block of 32 for the first nw warps (a power of
        // two, at least 2).  m_ema is the same in every thread, so the choice
        // is uniform.
        const float want = sqrtf(kLatChunkCost * m_ema);
        const bool two = want > (float)kThreads;
        const unsigned nb = want > 2.0f * (float)kThreads ? 2u : 1u;
        unsigned nw = 2;
        while (nw < (unsigned)kWarps && (float)(32u * nw) < want) nw <<= 1;
        if (two || nw > (unsigned)kWarps) nw = kWarps;
        const unsigned step = two ? 64u : 32u;
        const unsigned C = nb * nw * step;
        unsigned long long p = 0;
        unsigned kb_hit = 0;
        bool found = false;
        while (!found) {
            ++p;
            const PhiloxPrefix PP =
                philox_prefix((uint32_t)rounds, (uint32_t)(rounds >> 32), rep, key0, key1);
            for (unsigned kb = 0; kb < M; kb += C) {
                bool hit = false;
                if ((unsigned)warp < nw) {
                    const unsigned k0 = kb + (unsigned)warp * step;
                    if (a.toy) {
                        for (unsigned k = k0; k < kb + C && !hit; k += nw * step)
                            for (unsigned n = 0; n < step && !hit; n += 32u)
                                hit = lat_eval_toy<kPow2, kDim>(K, k + n, PP, V, a.toy_A0,
                                                                      &s_best[par]);
                    } else if (kF64 && fixed) {
                        if (two) {
#pragma unroll 1
                            for (unsigned k = k0; k < kb + C && !hit; k += nw * step)
                                hit = lat_eval<Fix, kPow2, kDim, 2>(K, k, PP, &s_best[par]);
                        } else {
                            hit = lat_eval<Fix, kPow2, kDim, 1>(K, k0, PP, &s_best[par]);
                        }
                    } else if (two) {
#pragma unroll 1
                        for (unsigned k = k0; k < kb + C && !hit; k += nw * step)
                            hit = lat_eval<Real, kPow2, kDim, 2>(K, k, PP, &s_best[par]);
                    } else {
                        hit = lat_eval<Real, kPow2, kDim, 1>(K, k0, PP, &s_best[par]);
                    }
                }
                if (__syncthreads_or(hit)) {
                    kb_hit = kb;
                    found = true;
                    break;
                }
            }
            if (!found) {
                if (tid == kBook) {
                    s_c.attempts += M;
                    s_c.evaluated += M;
                }
                rounds += 1;
                // bounded hop: one thread reads its SM's cycle counter (the
                // limit is in cycles at the peak clock), the block-wide OR
                // makes the decision uniform
                const int late = __syncthreads_or(
                    tid == kBook && (unsigned long long)(clock64() - s_c.t0) > a.hop_timeout_cyc);
                if (late) {
                    status = CG_ETIMEOUT;
                    break;
                }
                if (p >= a.max_rounds) {
                    status = CG_ESTUCK;
                    break;
                }
            }
        }
        if (!found) break;

        // ---- commit (step 3a, 3c) ----
        const unsigned wl = s_best[par];          // the round's lowest accepting label
        const unsigned q = wl + 1;                // 1-based label in the round
        const Cand c = s_cand[(wl - kb_hit) / step % nw];
        const unsigned ci = c.i, cj = c.j;
        const unsigned long long m_hop = (p - 1) * (unsigned long long)M + q;
        m_ema = 0.9f * m_ema + 0.1f * (float)m_hop;
        long long t1 = 0;
        if (tid == kBook) {
            t1 = clock64();
            s_best[par ^ 1u] = 0xffffffffu;       // last read before the previous hop's end
            if (!a.toy) {
                sm<unsigned>(lay.off_occ, ci >> 5) &= ~(1u << (ci & 31));
                sm<unsigned>(lay.off_occ, cj >> 5) |= (1u << (cj & 31));
            }
        }
        __syncwarp();     // or that warp would run the update twice, once for this lane

        // ---- local-energy update (step 3b) ----
        unsigned big = 0;
        if (kF64 && fixed) {
            if (kDim == 3)
                update_cubic<Fix, kThreads, kPow2>(!a.toy, lay.off_eps, lay.off_tinv, ci, cj, L,
                                                   log2L, magic, big);
            else
                update_square<Fix, kThreads, kPow2>(!a.toy, lay.off_eps, lay.off_tinv, ci, cj, L,
                                                    log2L, magic, big);
        } else {
            if (kDim == 3)
                update_cubic<Real, kThreads, kPow2>(!a.toy, lay.off_eps, lay.off_tinv, ci, cj, L,
                                                    log2L, magic, big);
            else
                update_square<Real, kThreads, kPow2>(!a.toy, lay.off_eps, lay.off_tinv, ci, cj, L,
                                                     log2L, magic, big);
        }
        if (kF64 && fixed) {
            // an energy has reached 4 in size: back to binary64 before the
            // next hop could leave the integers' range (one hop moves it by
            // at most 1)
            if (__syncthreads_or((int)(big >> 30) & 1)) {
                for (int l = tid; l < N; l += kThreads)
                    sm<double>(lay.off_eps, l) = fix_to_double(sm<long long>(lay.off_eps, l));
                for (int l = tid; l < ntab; l += kThreads)
                    sm<double>(lay.off_tinv, l) = fix_to_double(sm<long long>(lay.off_tinv, l));
                fixed = false;
                __syncthreads();
            }
        } else {
            __syncthreads();
        }
        // the books of this hop, beside the next hop's first labels
        if (tid == kBook) {
            int cdx, cdy;
            vec_fields<kPow2, kDim>((unsigned)c.dxy, L, log2L, cdx, cdy);
            s_c.cyc_rej += (unsigned long long)(t1 - s_c.t0);
            s_c.cyc_upd += (unsigned long long)(clock64() - t1);
            if (kTime)           // step 3c: Gaussian dt of hop number s_c.hops
                s_c.time = d_add(s_c.time, cg_time_increment(Rg.Gamma, m_hop,
                                                            s_z[s_c.hops - s_c.zbase]));
            s_c.attempts += q;
            // the chunks of the hop's round up to the accepting one
            s_c.evaluated += (kb_hit + C < M) ? (kb_hit + C) : M;
            s_c.hops += 1;
            if (!a.toy) {
                s_c.P += cdx;
                s_c.energy = d_add(s_c.energy, c.dE);
            }
            if (s_c.tracing)
                trace_hop(Rg, s_c.attempts, s_c.hops, s_c.P, s_c.energy, kTime ? 1 : 0, s_c.time);
            if (s_c.log) {
                cg_hop e;
                e.i = ci; e.j = cj; e.q = q; e.p = (uint32_t)p; e.round = rounds;
                e.dx = a.toy ? 0 : cdx; e.dy = a.toy ? 0 : cdy;
                e.dE = a.toy ? 0.0 : c.dE;
                e.k = 0xFFFFFFFFu; e.l = 0xFFFFFFFFu;
                e.dx2 = 0; e.dy2 = 0;
                s_c.log[a.log_offset + h] = e;
            }
        }
        rounds += 1;
        par ^= 1u;
    }

    // ---- store the replica back ----
    {
        Real *eps_g = reinterpret_cast<Real *>(Rg.eps);
        for (int l = tid; l < N; l += kThreads)
            eps_g[l] = kF64 && fixed ? (Real)lat_energy<Fix>(lay.off_eps, l)
                                     : sm<Real>(lay.off_eps, l);
        for (int l = tid; l < words; l += kThreads) Rg.occ[l] = sm<unsigned>(lay.off_occ, l);
    }
    if (tid == kBook) {
        DevCounters *cnt = Rg.ctr;
        cnt->rounds = rounds;
        cnt->hops = s_c.hops;
        cnt->attempts = s_c.attempts;
        cnt->evaluated = s_c.evaluated;
        cnt->P = s_c.P;
        cnt->energy = s_c.energy;
        cnt->time = s_c.time;
        cnt->cycles_reject += s_c.cyc_rej;
        cnt->cycles_update += s_c.cyc_upd;
        cnt->m_ema = m_ema;
        if (s_c.hops - s_c.hops0 >= 32ull)
            cnt->rate = (float)(s_c.attempts - s_c.attempts0) / (float)(s_c.hops - s_c.hops0);
        cnt->status = status;
    }
}

}  // namespace cg
