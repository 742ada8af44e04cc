// cg_pr_random.cuh -- the label of the random-site chain (partner lookup,
// theta, the binary64 energy change), shared by the single-CTA kernel
// (cg_pr_random.cu) and its cluster form (cg_pr_random_cluster.cu).
#pragma once

#include "cg_pr_common.cuh"

namespace cg {

struct RCand {
    unsigned i, j;
    double dE;
};

struct RLabel {
    unsigned i, j, x2;
    double2 gx;               // 1/r_ij and E dx_ij
    float cv;                 // 1/r_ij + E dx_ij or up to 1/64 of it above
    bool theta;
};

// Label k's site, partner and theta.  An empty site i has theta = 0 whatever
// its partner, so the partner is looked up for occupied sites only: the
// smallest m of i's list with x1 < C_m.  One 64-byte load of i's guide record
// gives the list's bounds, its last running weight (x1 at or above it: a null
// proposal) and the bucket of pairs x1 >> 28 can select; a four-way search
// (three independent probes per step) narrows a bucket of more than eight, and
// the rest is counted from up to three aligned loads of four weights (C_m - 1,
// 32 bits).  The chosen pair's partner with a bound on its 1/r + E dx, and 1/r
// and E dx themselves, are two more loads side by side: five sectors per label
// where whole records, read with their 1/r and E dx in the scan, took seven.
// (1/r and E dx loaded for the few labels that need them would save one sector
// but put one more load into the chain of a hop: 24 replicas of L = 64 4.20
// against 4.11 ms per 128 hops at T = 0.05, 4.35 against 4.20 at T = 0.3; one
// of L = 32 at T = 0.3 2.53 against 2.43.)
// gsm: the compacted guide records in shared memory (two uint4 per site:
// {first, last lo, length | last hi << 16, 0} and the 16 bucket starts as
// bytes), or null for the 64-byte records in global memory.
__device__ __forceinline__ RLabel propose_random(const DevReplica &Rg, const unsigned *occ,
                                                 unsigned k, const PhiloxPrefix &PP,
                                                 uint32_t key0, uint32_t key1, unsigned N,
                                                 bool valid, const uint4 *gsm = nullptr)
{
    RLabel p;
    p.theta = false;
    p.i = p.j = 0;
    p.x2 = 0;
    p.gx = make_double2(0.0, 0.0);
    p.cv = 0.0f;
    if (!valid) return p;
    uint32_t x[4];
    philox_finish(k, PP, key0, key1, x);
    p.i = __umulhi(x[0], N);
    p.x2 = x[2];
    if (!((occ[p.i >> 5] >> (p.i & 31)) & 1u)) return p;
    const unsigned long long x1 = x[1];
    const uint32_t w1 = x[1];
    const unsigned b = x[1] >> 28, b1 = b + 1;
    int first, end, glo, ghi;
    unsigned long long last;
    if (gsm) {
        const uint4 ra = gsm[2 * p.i], rb = gsm[2 * p.i + 1];
        first = (int)ra.x;
        end = first + (int)(ra.z & 0xffffu);
        last = (unsigned long long)ra.y | ((unsigned long long)((ra.z >> 16) & 1u) << 32);
        if (first == end || x1 >= last) return p;
        // byte b of words 4..7: the start of bucket b
        const unsigned wb = (b >> 2) == 0 ? rb.x : (b >> 2) == 1 ? rb.y : (b >> 2) == 2 ? rb.z : rb.w;
        const unsigned wb1 = (b1 >> 2) == 0 ? rb.x : (b1 >> 2) == 1 ? rb.y
                           : (b1 >> 2) == 2 ? rb.z : rb.w;
        glo = first + (int)((wb >> (8 * (b & 3))) & 0xffu);
        ghi = b1 < (unsigned)kRandomBuckets ? first + (int)((wb1 >> (8 * (b1 & 3))) & 0xffu) : end;
    } else {
        const int4 *g4 = reinterpret_cast<const int4 *>(Rg.rguide + (size_t)p.i * kRandomGuide);
        const int4 ga = __ldg(g4), gb = __ldg(g4 + 1), gc = __ldg(g4 + 2);
        first = ga.x;
        end = ga.y;                                        // [0] and [1]
        last = (unsigned long long)(uint32_t)ga.z | ((unsigned long long)(uint32_t)ga.w << 32);
        if (first == end || x1 >= last) return p;
        // the 16-bit starts of buckets b = x1 >> 28 and b + 1 (words [4..11]
        // in gb, gc; bucket 16 starts at the list's end)
        const unsigned w0 = (b >> 1) < 4 ? (unsigned)((b >> 1) == 0 ? gb.x : (b >> 1) == 1 ? gb.y
                                                      : (b >> 1) == 2 ? gb.z : gb.w)
                                         : (unsigned)((b >> 1) == 4 ? gc.x : (b >> 1) == 5 ? gc.y
                                                      : (b >> 1) == 6 ? gc.z : gc.w);
        const unsigned w1 = (b1 >> 1) < 4 ? (unsigned)((b1 >> 1) == 0 ? gb.x : (b1 >> 1) == 1 ? gb.y
                                                       : (b1 >> 1) == 2 ? gb.z : gb.w)
                                          : (unsigned)((b1 >> 1) == 4 ? gc.x : (b1 >> 1) == 5 ? gc.y
                                                       : (b1 >> 1) == 6 ? gc.z : gc.w);
        glo = first + (int)((b & 1) ? (w0 >> 16) : (w0 & 0xffffu));
        ghi = b1 < (unsigned)kRandomBuckets
                  ? first + (int)((b1 & 1) ? (w1 >> 16) : (w1 & 0xffffu))
                  : end;
    }
    int lo = glo, hi = min(ghi, end - 1) + 1;
    const uint32_t *rw = Rg.rw;
    // the answer lies in [lo, hi); x1 < C_m iff x1 <= rw[m]
    while (hi - lo > 8) {
        const int q = (hi - lo) >> 2;
        const int m1 = lo + q, m2 = m1 + q, m3 = m2 + q;
        const uint32_t c1 = __ldg(rw + m1), c2 = __ldg(rw + m2), c3 = __ldg(rw + m3);
        if (w1 <= c1) {
            hi = m1 + 1;
        } else if (w1 <= c2) {
            lo = m1 + 1;
            hi = m2 + 1;
        } else if (w1 <= c3) {
            lo = m2 + 1;
            hi = m3 + 1;
        } else {
            lo = m3 + 1;
        }
    }
    // the pairs of [lo, hi - 1) with C_m <= x1 come before the answer (the
    // weights rise along the list); a window of up to 11 from the group lo is in
    // (the last group may read up to three words past the weights, where the
    // partners' lie; they do not count)
    const int base = lo & ~3;
    const uint4 *r4 = reinterpret_cast<const uint4 *>(rw + base);
    const uint4 wa = __ldg(r4);
    uint4 wb = make_uint4(0u, 0u, 0u, 0u), wc = wb;
    if (base + 4 < hi - 1) wb = __ldg(r4 + 1);
    if (base + 8 < hi - 1) wc = __ldg(r4 + 2);
    const uint32_t w[12] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w, wc.x, wc.y, wc.z, wc.w};
    int m = lo;
#pragma unroll
    for (int t = 0; t < 12; ++t) {
        const int e = base + t;
        m += (e >= lo && e < hi - 1 && w[t] < w1) ? 1 : 0;
    }
    const uint32_t rc = __ldg(Rg.rj + m);
    p.gx = __ldg(Rg.rgx + m);
    p.j = rc & kPartnerMask;
    p.cv = __uint_as_float(rc & ~kPartnerMask);
    p.theta = !((occ[p.j >> 5] >> (p.j & 31)) & 1u);     // n_i = 1 here
    return p;
}

// Step 2 for a label whose theta holds: its dH is bounded from the energies'
// high words first (as in the lattice kernels), and the few labels below the cut
// take the binary64 one, ((eps_j - eps_i) - 1/r_ij) - E dx_ij, each step rounded,
// and the binary64 decision.  (Three binary64 adds per label on the slow pipe
// were a quarter of a chunk.)
__device__ __forceinline__ bool accept_random(double ei, double ej, const RLabel &p, float cut,
                                              double T, float invTf, double &dE)
{
    bool oi, oj;
    const float fi = hi_to_f32(__double2hiint(ei), oi), fj = hi_to_f32(__double2hiint(ej), oj);
    const float s = fabsf(fi) + fabsf(fj) + fabsf(p.cv);
    const float lo = fmaf(s, -0x1p-19f, (fj - fi) - p.cv);      // at most dH
    if (oi && oj && (!(lo < cut) || surely_rejected(lo, p.x2, invTf))) return false;
    dE = d_sub(d_sub(d_sub(ej, ei), p.gx.x), p.gx.y);
    return metropolis64(dE, p.x2, T, invTf);
}

// Stage the compacted guide records of all N sites into shared memory (two
// uint4 per site, from the 64-byte records; every list below 256 pairs).
template <int kThreads>
__device__ __forceinline__ void stage_guide(uint4 *gsm, const DevReplica &Rg, int N, int tid)
{
    for (int s = tid; s < N; s += kThreads) {
        const int4 *g4 = reinterpret_cast<const int4 *>(Rg.rguide + (size_t)s * kRandomGuide);
        const int4 ga = g4[0], gb = g4[1], gc = g4[2];
        const unsigned w16[8] = {(unsigned)gb.x, (unsigned)gb.y, (unsigned)gb.z, (unsigned)gb.w,
                                 (unsigned)gc.x, (unsigned)gc.y, (unsigned)gc.z, (unsigned)gc.w};
        unsigned bytes[4] = {0u, 0u, 0u, 0u};
#pragma unroll
        for (int b = 0; b < kRandomBuckets; ++b) {
            const unsigned off = (b & 1) ? (w16[b >> 1] >> 16) : (w16[b >> 1] & 0xffffu);
            bytes[b >> 2] |= (off & 0xffu) << (8 * (b & 3));
        }
        gsm[2 * s] = make_uint4((unsigned)ga.x, (unsigned)ga.z,
                                (unsigned)(ga.y - ga.x) | (((unsigned)ga.w & 1u) << 16), 0u);
        gsm[2 * s + 1] = make_uint4(bytes[0], bytes[1], bytes[2], bytes[3]);
    }
}

}  // namespace cg
