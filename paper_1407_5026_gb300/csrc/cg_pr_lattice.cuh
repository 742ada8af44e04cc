// cg_pr_lattice.cuh -- the persistent parallel-rejection kernel with one CTA
// per replica (square lattice: cg_pr_kernel.cu, cubic lattice:
// cg_pr_kernel3d.cu; with two-electron hops: cg_pr_kernel_pair.cu,
// cg_pr_kernel_pair_time.cu and cg_pr_kernel3d_pair.cu).
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
// What bounds it (L = 128, T = 0.01, 304 replicas, two CTAs per SM): 32 labels
// cost 97 warp instructions (counted), 50 of them on the integer pipe, 28 on the
// multiply pipe and 6 loads; Philox alone is 40 of the 78.  Half of the issue
// slots are taken; fixed latencies, the chunks' barriers and shared-memory latency
// come first among the waits.  Labels run at 120 G/s over a launch and 151 G/s
// over the rejection phase, the generator by itself at 464.  More warps change
// nothing.  So the per-label work
// was cut: only a label whose theta holds and whose dH is below the cut (one in
// a few hundred) reaches the exponential, the near-tie test and, in binary64,
// the slow binary64 pipe (its dH is first bounded from the energies' high
// words); the tower is one byte of a 16,384-entry table for 99.5% of the words
// x1; every lane runs the loads without a branch.  A chunk with an accept needs
// no second barrier: the accepting warps write their proposals and lower a
// shared minimum before the one that ends the chunk.
// ms per run call of the kernel before (150 instructions per label, 512 threads
// throughout) and of this one, same chains: L = 128 binary32 12.12 -> 9.77,
// binary64 (152 replicas) 2.95 -> 1.36; 24 binary64 chains of L = 64 4.25 ->
// 2.38; L = 32 to 96 mixed 3.16 -> 1.69; 32^3 2.24 -> 1.94; L = 64 with a fifth
// pair labels 2.53 -> 1.89.  Four labels per lane in place of two gained
// nothing (9.60 to 9.68 against 9.66; mixed 1.65 against 1.62), and neither did a search
// without barriers, which evaluates labels past the accepting one.
#pragma once

#include <type_traits>

#include "cg_pr_update.cuh"

namespace cg {

// b of the chunk rule C ~ sqrt(m b)
constexpr float kLatChunkCost = 256.0f;

// Hop vector of a packed displacement word (see rec below): with a
// power-of-two L the fields are dx mod L, dy mod L (and dz mod L), otherwise
// dx | dy << 16 (square) or 10-bit fields (cubic).
template <bool kPow2, int kDim>
__device__ __forceinline__ void vec_fields(unsigned w, int L, int log2L, int &dx, int &dy, int &dz)
{
    dz = 0;
    if (kPow2) {
        if (kDim == 3) {
            dz = (int)(w >> (2 * log2L));
            dz -= (dz >= (L >> 1)) ? L : 0;
        }
        dx = (int)(w & (unsigned)(L - 1));
        dx -= (dx >= (L >> 1)) ? L : 0;
        dy = (int)((w >> log2L) & (unsigned)(L - 1));
        dy -= (dy >= (L >> 1)) ? L : 0;
    } else if (kDim == 3) {
        dx = (int)(w << 22) >> 22;
        dy = (int)(w << 12) >> 22;
        dz = (int)w >> 20;
    } else {
        dx = (int)(short)(w & 0xffffu);
        dy = (int)w >> 16;
    }
}

// The displacement word of (dx, dy, dz), and of a packed hop vector dxy
// (cg_internal.h).
template <bool kPow2, int kDim>
__device__ __forceinline__ unsigned vec_word(int dx, int dy, int dz, int L, int log2L)
{
    if (!kPow2)
        return kDim == 3 ? ((unsigned)dx & 0x3ffu) | (((unsigned)dy & 0x3ffu) << 10) |
                               ((unsigned)dz << 20)
                         : ((unsigned)dx & 0xffffu) | ((unsigned)dy << 16);
    const unsigned m = (unsigned)(L - 1);
    const unsigned yx = (((unsigned)dy & m) << log2L) | ((unsigned)dx & m);
    return kDim == 3 ? (((unsigned)dz & m) << (2 * log2L)) | yx : yx;
}

template <bool kPow2, int kDim>
__device__ __forceinline__ unsigned vec_word(int dxy, int L, int log2L)
{
    if (kDim == 3)
        return vec_word<kPow2, kDim>((dxy << 22) >> 22, (dxy << 12) >> 22, dxy >> 20, L, log2L);
    return vec_word<kPow2, kDim>((int)(short)(dxy & 0xffff), dxy >> 16, 0, L, log2L);
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

// The tower's tables into shared memory.
template <int kThreads, bool kPow2, int kDim>
__device__ __forceinline__ void stage_tower(const LatLayout &lay, const DevReplica &Rg,
                                            int guide_bits, int L, int log2L)
{
    const int tid = threadIdx.x, V = Rg.V;
    // the device table has 2^kLatGuideBits entries; a coarser bucket
    // holds its entries' common value, or 255
    const int per = 1 << (kLatGuideBits - guide_bits);
    for (int b = tid; b < (1 << guide_bits); b += kThreads) {
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

// dH above which no acceptance variate accepts, with a margin: binary32
// variates are at least 2^-24 (ln: -16.64), binary64 ones 2^-33, and the
// binary64 test calls e^y zero below y = -23.  The binary32 form decides
// |dH| < 1e-5 apart.
template <bool kF64>
__device__ __forceinline__ float lat_cut(double T)
{
    return kF64 ? (float)(23.1 * T) : fmaxf((float)(17.0 * T), 1.1e-5f);
}

// Room for the rounding of cv and of fixed-point energies to binary32.
__device__ __forceinline__ float lat_slack(double E, int L)
{
    return (float)((8.0 + fabs(E) * (double)(L / 2)) * 0x1p-21);
}

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

// The vector of a word x1: the guide's, or the search's where it has none; false
// for a null proposal (v is then some vector's index).
__device__ __forceinline__ bool lat_draw(const LatLayout &S, uint32_t x1, int gshift, int vbase,
                                         int vlast, unsigned thr_last, int &v)
{
    const int g = (int)sm<unsigned char>(S.off_guide, x1 >> gshift);
    v = g + vbase;
    if (g != 255) return true;
    v = vlast;
    return lat_search(S, x1, thr_last, v);
}

// What a label's evaluation reads that stays fixed over a launch.
struct LatConst {
    LatLayout S;
    Cand *cand;                // per warp: its lowest accepting label's proposal
    int L, log2L, vbase, vlast, gshift, warp, lane;
    unsigned N, magic, M, thr_last;
    uint32_t key0, key1;
    float cut, slack, invTf;   // slack: binary64's bound on what binary32 loses of dH
    double T;
    // two-electron hops
    PairProp *pcand;           // per warp: the second electron of its candidate
    unsigned pair_T;
    int pair_R;
    const double *tab64;       // the binary64 table in global memory
};

// Two-electron hops: a label whose fourth word is below pair_T proposes a pair.
// From the Philox block of counter (k, r lo, r hi | 2^31, replica), y0, y2 (and
// y3 on the cubic lattice) give the offset e of the second electron k = i + e,
// each axis floor(y W / 2^32) - R with W = 2R + 1, and y1 its hop vector d2 by
// the same tower, l = k + d2.  theta also needs n_k = 1, n_l = 0,
// 0 < |e|^2 <= R^2 and 0 < |e'|^2 <= R^2 for the reverse offset
// e' = e + d2 - d1, so that a pair and its reverse are proposed with the same
// probability.  w1: the displacement word of the first electron's hop.
struct LatPair {
    unsigned k, l, w2;
    int v2;
    float cv2;
    bool ok;
};

template <bool kPow2, int kDim>
__device__ __forceinline__ LatPair lat_pair(const LatConst &K, unsigned label,
                                            const PhiloxPrefix &PP2, unsigned i, unsigned w1)
{
    LatPair q;
    uint32_t y[4];
    philox_finish(label, PP2, K.key0, K.key1, y);
    const int R = K.pair_R;
    const unsigned W = (unsigned)(2 * R + 1);
    const int ex = (int)__umulhi(y[0], W) - R, ey = (int)__umulhi(y[2], W) - R;
    const int ez = kDim == 3 ? (int)__umulhi(y[3], W) - R : 0;
    const bool live = lat_draw(K.S, y[1], K.gshift, K.vbase, K.vlast, K.thr_last, q.v2);
    const uint2 rc = sm<uint2>(K.S.off_rec, q.v2);
    q.cv2 = __uint_as_float(rc.x);
    q.w2 = rc.y;
    int dx1, dy1, dz1, dx2, dy2, dz2;
    vec_fields<kPow2, kDim>(w1, K.L, K.log2L, dx1, dy1, dz1);
    vec_fields<kPow2, kDim>(q.w2, K.L, K.log2L, dx2, dy2, dz2);
    q.k = hop_target<kPow2, kDim>(i, vec_word<kPow2, kDim>(ex, ey, ez, K.L, K.log2L), K.L, K.log2L,
                                  K.N, K.magic);
    q.l = hop_target<kPow2, kDim>(q.k, q.w2, K.L, K.log2L, K.N, K.magic);
    const int fx = ex + dx2 - dx1, fy = ey + dy2 - dy1, fz = ez + dz2 - dz1;
    const int e2 = ex * ex + ey * ey + ez * ez, f2 = fx * fx + fy * fy + fz * fz, R2 = R * R;
    const unsigned wk = sm<unsigned>(K.S.off_occ, q.k >> 5), wl = sm<unsigned>(K.S.off_occ, q.l >> 5);
    q.ok = live && e2 > 0 && e2 <= R2 && f2 > 0 && f2 <= R2 && ((wk >> (q.k & 31u)) & 1u) &&
           !((wl >> (q.l & 31u)) & 1u);
    return q;
}

// eps_s as binary64.
template <typename Store>
__device__ __forceinline__ double lat_energy(int off_eps, unsigned s)
{
    if constexpr (std::is_same<Store, long long>::value)
        return fix_to_double(sm<long long>(off_eps, s));
    else
        return (double)sm<Store>(off_eps, s);
}

// Step 2 for a pair whose theta holds; dE is its dH in binary64 (binary32
// energies: from the widened ones, as for the executed pair).  The binary32
// form decides by the same sum in binary32, and near ties (|dH| < 1e-5) by the
// binary64 one.
template <typename Store, bool kPow2, int kDim>
__device__ __forceinline__ bool lat_accept_pair(const LatConst &K, const LatPair &q, unsigned i,
                                                unsigned j, int v, float cv, uint32_t x2,
                                                double &dE)
{
    const int H1 = K.L / 2 + 1;
    // -1: undecided (binary64 decides), else the binary32 form's decision
    int take = -1;
    if constexpr (sizeof(Store) == 4) {
        const float *t32 = &sm<float>(K.S.off_tinv);
        const float ei = sm<float>(K.S.off_eps, i), ej = sm<float>(K.S.off_eps, j);
        const float ek = sm<float>(K.S.off_eps, q.k), el = sm<float>(K.S.off_eps, q.l);
        const float d1 = __fsub_rn(__fsub_rn(ej, ei), cv);
        const float d2 = __fsub_rn(__fsub_rn(el, ek), q.cv2);
        const float cr = __fsub_rn(
            __fsub_rn(tinv_sites<float, kPow2, kDim>(t32, q.l, j, K.L, K.log2L, K.magic, H1),
                      tinv_sites<float, kPow2, kDim>(t32, q.l, i, K.L, K.log2L, K.magic, H1)),
            __fsub_rn(tinv_sites<float, kPow2, kDim>(t32, q.k, j, K.L, K.log2L, K.magic, H1),
                      tinv_sites<float, kPow2, kDim>(t32, q.k, i, K.L, K.log2L, K.magic, H1)));
        const float dEf = __fadd_rn(__fadd_rn(d1, d2), cr);
        if (!(fabsf(dEf) < 1e-5f))
            take = dEf <= 0.0f ||
                   (float)(x2 >> 9) < __fmaf_rn(__expf(-dEf * K.invTf), 0x1p23f, -0.5f);
        if (take == 0) return false;
    }
    dE = pair_dE64_vals<kPow2, kDim>(
        K.tab64, lat_energy<Store>(K.S.off_eps, i), lat_energy<Store>(K.S.off_eps, j),
        lat_energy<Store>(K.S.off_eps, q.k), lat_energy<Store>(K.S.off_eps, q.l),
        sm<double>(K.S.off_vr64, v), sm<double>(K.S.off_edx64, v), sm<double>(K.S.off_vr64, q.v2),
        sm<double>(K.S.off_edx64, q.v2), i, j, q.k, q.l, K.L, K.log2L, K.magic, H1);
    return take > 0 || metropolis64(dE, x2, K.T, K.invTf);
}

// The warp's block of 32 NL labels from kb on: label kb + 32 n + lane, n < NL.
// Only labels whose theta holds and whose dH is below the cut go through the
// accept test; the lowest accepting lane writes the warp's candidate and
// lowers the CTA's best label.  True when the block holds an accept.
// Store: the type of the energies in shared memory (long long: binary64 in
// fixed point).
template <typename Store, bool kPow2, int kDim, int NL, bool kPair>
__device__ __forceinline__ bool lat_eval(const LatConst &K, unsigned kb, const PhiloxPrefix &PP,
                                         const PhiloxPrefix &PP2, unsigned *best)
{
    constexpr bool kF64 = sizeof(Store) == 8, kFix = std::is_same<Store, long long>::value;
    uint32_t x1[NL], x2[NL];
    unsigned si[NL], sj[NL];
    int v[NL];
    float cv[NL], d[NL];
    bool on[NL], cand[NL], pair[NL];
    bool odd = false;
#pragma unroll
    for (int n = 0; n < NL; ++n) {
        const unsigned k = kb + 32u * (unsigned)n + (unsigned)K.lane;
        uint32_t x[4];
        philox_finish(k, PP, K.key0, K.key1, x);
        x1[n] = x[1];
        x2[n] = x[2];
        pair[n] = kPair && x[3] < K.pair_T;
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
            // 2^-28 + 2^-22 each below 8; the cut's slack covers it
            const float fi = __int2float_rn(sm<int>(K.S.off_eps, 2 * si[n] + 1));
            const float fj = __int2float_rn(sm<int>(K.S.off_eps, 2 * sj[n] + 1));
            d[n] = fmaf(fj - fi, 0x1p-28f, -cv[n]) - K.slack;    // at most dH
            cand[n] = theta && !pair[n] && d[n] < K.cut;
        } else if constexpr (kF64) {
            bool oi, oj;
            const float fi = hi_to_f32(sm<int>(K.S.off_eps, 2 * si[n] + 1), oi);
            const float fj = hi_to_f32(sm<int>(K.S.off_eps, 2 * sj[n] + 1), oj);
            // at most dH (or nothing known: the test decides)
            d[n] = fmaf(fabsf(fi) + fabsf(fj), -0x1p-19f, (fj - fi) - cv[n]) - K.slack;
            if (!oi || !oj) d[n] = 0.0f;
            cand[n] = theta && !pair[n] && d[n] < K.cut;
        } else {
            d[n] = __fsub_rn(__fsub_rn(sm<float>(K.S.off_eps, sj[n]), sm<float>(K.S.off_eps, si[n])),
                             cv[n]);
            cand[n] = theta && !pair[n] && d[n] < K.cut;
        }
        pair[n] = pair[n] && theta;
    }
    // pair labels whose first electron can hop: one in twenty at half filling,
    // so a lane rarely has two and the block rarely takes a second turn
    unsigned pacc = 0;                         // bit n: pair label n accepts
    LatPair pq;                                // the lane's lowest accepting pair
    double pdE = 0.0;
    if constexpr (kPair) {
        unsigned todo = (pair[0] ? 1u : 0u) | (NL > 1 && pair[NL - 1] ? 2u : 0u);
        while (__any_sync(0xffffffffu, todo != 0u)) {
            const bool first = (todo & 1u) || NL == 1;
            if (todo) {
                const unsigned i = first ? si[0] : si[NL - 1], j = first ? sj[0] : sj[NL - 1];
                const int v1 = first ? v[0] : v[NL - 1];
                const LatPair q = lat_pair<kPow2, kDim>(
                    K, kb + (first ? 0u : 32u) + (unsigned)K.lane, PP2, i,
                    sm<uint2>(K.S.off_rec, v1).y);
                double dE;
                if (q.ok &&
                    lat_accept_pair<Store, kPow2, kDim>(K, q, i, j, v1, first ? cv[0] : cv[NL - 1],
                                                        first ? x2[0] : x2[NL - 1], dE) &&
                    !pacc) {
                    pacc = first ? 1u : 2u;
                    pq = q;
                    pdE = dE;
                }
                todo &= todo - 1u;
            }
        }
    }
    if (!__any_sync(0xffffffffu, cand[0] || cand[NL - 1] || pacc)) return false;
    // binary64: the bound on dH rejects most of them; what is left takes the
    // slow pipe
    if constexpr (kF64) {
#pragma unroll
        for (int n = 0; n < NL; ++n)
            cand[n] = cand[n] && !surely_rejected(d[n], x2[n], K.invTf);
        if (!__any_sync(0xffffffffu, cand[0] || cand[NL - 1] || pacc)) return false;
    }
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
    const unsigned b0 = __ballot_sync(0xffffffffu, acc[0] || (pacc & 1u));
    const unsigned b1 = NL > 1 ? __ballot_sync(0xffffffffu, acc[NL - 1] || (pacc & 2u)) : 0u;
    if (!(b0 | b1)) return false;
    if (K.lane == __ffs(b0 ? b0 : b1) - 1) {
        Cand c;
        c.i = b0 ? si[0] : si[NL - 1];
        c.j = b0 ? sj[0] : sj[NL - 1];
        c.dxy = (int)sm<uint2>(K.S.off_rec, b0 ? v[0] : v[NL - 1]).y;
        c.dE = b0 ? dE[0] : dE[NL - 1];
        // binary32: the executed hop's dH is the binary32 one, widened
        if (!kF64 && c.dE == 0.0) c.dE = (double)(b0 ? d[0] : d[NL - 1]);
        if constexpr (kPair) {
            PairProp out;
            out.k = out.l = 0xffffffffu;
            out.v2 = out.dxy2 = 0;
            out.pair = (b0 ? 1u : 2u) == pacc;
            if (out.pair) {
                out.k = pq.k;
                out.l = pq.l;
                out.v2 = pq.v2;
                out.dxy2 = (int)pq.w2;
                c.dE = pdE;
            }
            K.pcand[K.warp] = out;
        }
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
// SMs' sums of attempts come out close (304 replicas of L = 128 at T = 0.01, by
// the launch's own attempts: the largest sum is 1.10 of the mean; 1.32 in replica
// order, and the launch lasts as long as its slowest SM).  The SM only sets the preferred position: a
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

// Registers: two CTAs of 256 or 512 threads per SM (128 or 64 each).  A label
// pair in flight keeps about 90 values; at 256 threads the wider file gains more
// than the second half of the warps did (four CTAs of 256 at 64 registers help
// only batches of more than two replicas per SM: 608 of L = 64 2.1 ms against
// 2.0, 912 2.9 against 3.0).
template <typename Real, int kThreads, int kLog2L, bool kTime, int kDim = 2, bool kPair = false>
__global__ void __launch_bounds__(kThreads, (kThreads >= 1024 ? 1 : (kThreads <= 256 ? 512 : 1024) / kThreads))
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
    __shared__ PairProp s_pcand[kPair ? kWarps : 1];   // the second electron of a pair candidate
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
        stage_tower<kThreads, kPow2, kDim>(lay, Rg, a.guide_bits, L, log2L);
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
    const float cut = lat_cut<kF64>(T);

    // binary64: the energies and the table in fixed point where that is exact
    // for every one of them (the configurations' W = 1 and 2 at half filling;
    // a W that is no short binary fraction may leave small energies finer bits)
    bool fixed = false;
    if constexpr (kF64) {
        // from 1024 sites on: below, the update waits for latency, not for the
        // binary64 pipe, and the decoding costs more (L = 24: 3.4 against 3.2 us
        // a hop, L = 32: 2.95 and 2.99, L = 64: 2.9 and 4.2; 152 of L = 128: 1.94
        // against 2.40 ms per 64 hops)
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
    K.cut = cut; K.slack = lat_slack(Rg.E, L); K.invTf = invTf; K.T = T;
    K.pcand = s_pcand; K.pair_T = Rg.pair_T; K.pair_R = Rg.pair_R; K.tab64 = Rg.tinv64;

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
        const float want = sqrtf((kPair ? 0.5f : 1.0f) * kLatChunkCost * m_ema);
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
            PhiloxPrefix PP2{};
            if (kPair)
                PP2 = philox_prefix((uint32_t)rounds, (uint32_t)(rounds >> 32) | 0x80000000u, rep,
                                    key0, key1);
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
                                hit = lat_eval<Fix, kPow2, kDim, 2, kPair>(K, k, PP, PP2,
                                                                       &s_best[par]);
                        } else {
                            hit = lat_eval<Fix, kPow2, kDim, 1, kPair>(K, k0, PP, PP2,
                                                                       &s_best[par]);
                        }
                    } else if (two) {
#pragma unroll 1
                        for (unsigned k = k0; k < kb + C && !hit; k += nw * step)
                            hit = lat_eval<Real, kPow2, kDim, 2, kPair>(K, k, PP, PP2,
                                                                       &s_best[par]);
                    } else {
                        hit = lat_eval<Real, kPow2, kDim, 1, kPair>(K, k0, PP, PP2,
                                                                       &s_best[par]);
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
        PairProp cq{};                         // second electron (toy mode has none)
        if (kPair) cq = s_pcand[(wl - kb_hit) / step % nw];
        const bool cpair = kPair && !a.toy && cq.pair;
        const unsigned long long m_hop = (p - 1) * (unsigned long long)M + q;
        m_ema = 0.9f * m_ema + 0.1f * (float)m_hop;
        long long t1 = 0;
        if (tid == kBook) {
            t1 = clock64();
            s_best[par ^ 1u] = 0xffffffffu;       // last read before the previous hop's end
            if (!a.toy) {
                sm<unsigned>(lay.off_occ, ci >> 5) &= ~(1u << (ci & 31));
                sm<unsigned>(lay.off_occ, cj >> 5) |= (1u << (cj & 31));
                if (cpair) {
                    sm<unsigned>(lay.off_occ, cq.k >> 5) &= ~(1u << (cq.k & 31));
                    sm<unsigned>(lay.off_occ, cq.l >> 5) |= (1u << (cq.l & 31));
                }
            }
        }
        __syncwarp();     // or that warp would run the update twice, once for this lane

        // ---- local-energy update (step 3b) ----
        // an executed pair applies the second electron's update after the first
        // one's (each site rounds twice, in the serial order; a thread owns
        // the same sites in both)
        unsigned big = 0;
#pragma unroll 1
        for (int pass = 0; pass < (cpair ? 2 : 1); ++pass) {
            const unsigned ui = kPair && pass ? cq.k : ci, uj = kPair && pass ? cq.l : cj;
            if (kF64 && fixed) {
                if (kDim == 3)
                    update_cubic<Fix, kThreads, kPow2>(!a.toy, lay.off_eps, lay.off_tinv, ui, uj, L,
                                                       log2L, magic, big);
                else
                    update_square<Fix, kThreads, kPow2>(!a.toy, lay.off_eps, lay.off_tinv, ui, uj, L,
                                                        log2L, magic, big);
            } else {
                if (kDim == 3)
                    update_cubic<Real, kThreads, kPow2>(!a.toy, lay.off_eps, lay.off_tinv, ui, uj, L,
                                                        log2L, magic, big);
                else
                    update_square<Real, kThreads, kPow2>(!a.toy, lay.off_eps, lay.off_tinv, ui, uj,
                                                         L, log2L, magic, big);
            }
        }
        if (kF64 && fixed) {
            // an energy has reached 6 in size: back to binary64 before the
            // next hop could leave the integers' range of 8 (a hop moves it by
            // at most 1 per electron)
            if (__syncthreads_or(big >= kFixMost)) {
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
            int cdx, cdy, cdz, cdx2 = 0, cdy2 = 0;
            vec_fields<kPow2, kDim>((unsigned)c.dxy, L, log2L, cdx, cdy, cdz);
            if (kPair && cpair)
                vec_fields<kPow2, kDim>((unsigned)cq.dxy2, L, log2L, cdx2, cdy2, cdz);
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
                s_c.P += cdx + cdx2;
                s_c.energy = d_add(s_c.energy, c.dE);
            }
            if (s_c.tracing)
                trace_hop(Rg, s_c.attempts, s_c.hops, s_c.P, s_c.energy, kTime ? 1 : 0, s_c.time);
            if (s_c.log) {
                cg_hop e;
                e.i = ci; e.j = cj; e.q = q; e.p = (uint32_t)p; e.round = rounds;
                e.dx = a.toy ? 0 : cdx; e.dy = a.toy ? 0 : cdy;
                e.dE = a.toy ? 0.0 : c.dE;
                e.k = cpair ? cq.k : 0xFFFFFFFFu; e.l = cpair ? cq.l : 0xFFFFFFFFu;
                e.dx2 = cdx2; e.dy2 = cdy2;
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

// ---------------------------------------------------------------------------
// Instances.  The sides of the configurations and of their mixed batch (square
// 32, 48, 64, 96, 128; cubic 32 in binary32, the largest power of two whose eps
// fits one CTA) are fixed at compile time: the update's offsets and loop counts
// and the label's wraps become constants.  Single and two-electron hops, both
// clocks alike.  ms per run call with L at run time and fixed, 152 replicas, a
// fifth pair labels, 96 hops: L = 32 0.91 -> 0.77, 48 0.99 -> 0.84, 64 1.01 ->
// 0.85, 96 1.27 -> 1.05, 128 1.50 -> 1.20 (binary64, 64: 1.97 -> 1.82).  Any
// other L is read at run time, as a power of two or not.
// ---------------------------------------------------------------------------

using LatKernel = void (*)(const DevReplica *, const int *, RunArgs);

template <typename Real, int kThreads, bool kTime, int kDim, bool kPair>
LatKernel lattice_side(int L)
{
    if constexpr (kDim == 2) {
        switch (L) {
        case 32: return pr_lattice<Real, kThreads, 5, kTime, kDim, kPair>;
        case 48: return pr_lattice<Real, kThreads, -48, kTime, kDim, kPair>;
        case 64: return pr_lattice<Real, kThreads, 6, kTime, kDim, kPair>;
        case 96: return pr_lattice<Real, kThreads, -96, kTime, kDim, kPair>;
        case 128: return pr_lattice<Real, kThreads, 7, kTime, kDim, kPair>;
        }
    } else if constexpr (sizeof(Real) == 4) {
        if (L == 32) return pr_lattice<Real, kThreads, 5, kTime, kDim, kPair>;
    }
    return (L & (L - 1)) == 0 ? pr_lattice<Real, kThreads, 0, kTime, kDim, kPair>
                              : pr_lattice<Real, kThreads, -1, kTime, kDim, kPair>;
}

// Null for a CTA size that is not built.
template <bool kTime, int kDim, bool kPair>
LatKernel lattice_kernel(int precision, int threads, int L)
{
    if (precision == CG_FP64) {
        switch (threads) {
        case 1024: return lattice_side<double, 1024, kTime, kDim, kPair>(L);
        case 512: return lattice_side<double, 512, kTime, kDim, kPair>(L);
        case 384: return lattice_side<double, 384, kTime, kDim, kPair>(L);
        case 256: return lattice_side<double, 256, kTime, kDim, kPair>(L);
        }
    } else {
        switch (threads) {
        case 1024: return lattice_side<float, 1024, kTime, kDim, kPair>(L);
        case 512: return lattice_side<float, 512, kTime, kDim, kPair>(L);
        case 384: return lattice_side<float, 384, kTime, kDim, kPair>(L);
        case 256: return lattice_side<float, 256, kTime, kDim, kPair>(L);
        }
    }
    return nullptr;
}

template <bool kTime, int kDim, bool kPair>
cudaError_t launch_lattice(int precision, const DevReplica *d_reps, const int *d_index, int n_ctas,
                           int threads, int smem_bytes, const RunArgs &args, cudaStream_t st,
                           int L)
{
    const LatKernel k = lattice_kernel<kTime, kDim, kPair>(precision, threads, L);
    if (!k) return cudaErrorInvalidValue;
    k<<<n_ctas, threads, smem_bytes, st>>>(d_reps, d_index, args);
    return cudaGetLastError();
}

// Room for `bytes` of dynamic shared memory in every instance of one precision.
template <bool kTime, int kDim, bool kPair>
cudaError_t set_lattice_limit(int precision, int bytes)
{
    for (int threads : {256, 384, 512, 1024})
        for (int L : {4, 6, 32, 48, 64, 96, 128}) {
            const LatKernel k = lattice_kernel<kTime, kDim, kPair>(precision, threads, L);
            const cudaError_t e =
                cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
            if (e) return e;
        }
    return cudaSuccess;
}

}  // namespace cg
