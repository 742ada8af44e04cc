// cg_pr_update.cuh -- the local-energy update (step 3b) of the single-CTA
// lattice kernels: eps_l += 1/r_lj - 1/r_li for every site l, in shared memory,
// each site rounding in the serial chain's order.
#pragma once

#include "cg_pr_common.cuh"

namespace cg {

// Element i of the array at byte `off` of the CTA's dynamic shared memory.
// The kernels pass offsets, not pointers, to their inlined parts: indexing the
// array where it is declared shared keeps each access a shared-memory one with
// a 32-bit address.
template <typename T>
__device__ __forceinline__ T &sm(int off, int i = 0)
{
    extern __shared__ __align__(16) unsigned char smem[];
    return reinterpret_cast<T *>(smem + off)[i];
}

// ---- binary64 energies in fixed point ----
// GB300 adds binary64 numbers at 1/64 of its binary32 rate, and the update's
// two adds per site were 63% of a hop of the L = 128 batch.  An energy that is
// a multiple of 2^-60 below 6 in size, and the table's 1/r (a multiple of 2^-60
// for r <= 256), are exact in a 64-bit integer of that unit (below 8: a hop moves
// an energy by at most 1 per electron), so the two
// roundings of eps + (1/r_lj - 1/r_li) become integer shifts and adds with the
// same bits: an integer sum, rounded to 53 significant bits, ties to even.
constexpr int kFixBits = 60;
constexpr unsigned kFixMost = 6u << (kFixBits - 32);   // high word of the bound 6

// Both conversions in integer arithmetic (the binary64 pipe is the slow one).
__device__ __forceinline__ double fix_to_double(long long e)
{
    if (e == 0) return 0.0;
    const unsigned long long u = (unsigned long long)(e < 0 ? -e : e);
    const int k = 63 - __clzll((long long)u);          // leading bit; at most 53 follow
    const unsigned long long m = k > 52 ? u >> (k - 52) : u << (52 - k);
    const unsigned long long ex = (unsigned long long)(1023 - kFixBits + k) << 52;
    return __longlong_as_double((long long)((e < 0 ? 1ull << 63 : 0ull) | ex |
                                            (m & 0x000fffffffffffffull)));
}

// x as an integer of 2^-60; ok is cleared unless that is exact, sign of zero
// included, and |x| < 6.
__device__ __forceinline__ long long fix_from_double(double x, bool &ok)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    if (b == 0) return 0;
    const int ex = (int)((b >> 52) & 0x7ffull), sh = ex - (1023 - kFixBits + 52);
    const unsigned long long m = (b & 0x000fffffffffffffull) | 0x0010000000000000ull;
    // ex <= 1025: below 8 (inf and NaN fail here); sh > -53: not below 2^-60
    // (subnormals and -0 fail here); no bit below 2^-60
    if (ex > 1025 || sh <= -53 || (sh < 0 && (m & ((1ull << -sh) - 1ull)))) {
        ok = false;
        return 0;
    }
    const long long e = (long long)(sh >= 0 ? m << sh : m >> -sh);
    if ((unsigned)((unsigned long long)e >> 32) >= kFixMost) ok = false;
    return (b >> 63) ? -e : e;
}

// s rounded to 53 significant bits, ties to even; big takes the largest high word
// (kFixMost or more: |s| may be 6 or more).  The position of the leading bit is taken from
// the one's complement of a negative s: it differs from |s|'s for s = -2^k
// alone, which either rounding keeps.
__device__ __forceinline__ long long fix_round53(long long s, unsigned &big)
{
    const unsigned lo = (unsigned)s, hi = (unsigned)((unsigned long long)s >> 32);
    const unsigned h = hi ^ (unsigned)((int)hi >> 31);
    big = max(big, h);
    unsigned msb;
    asm("bfind.u32 %0, %1;" : "=r"(msb) : "r"(h));    // 0xffffffff for h = 0
    const int sh = max((int)msb - 20, 0);             // bits below the 53 kept (at most 10)
    const unsigned mask = (1u << sh) - 1u;
    // half a unit less one, plus the last kept bit (none when nothing is cut)
    const unsigned r = (mask >> 1) + ((lo >> sh) & mask & 1u);
    const unsigned long long t = (unsigned long long)s + r;
    return (long long)((t & 0xffffffff00000000ull) | ((unsigned)t & ~mask));
}

// e + (a - b), each step rounded to T's precision (fixed point: binary64's).
__device__ __forceinline__ float site_add(float e, float a, float b, unsigned &)
{
    return __fadd_rn(e, __fsub_rn(a, b));
}
__device__ __forceinline__ double site_add(double e, double a, double b, unsigned &)
{
    return d_add(e, d_sub(a, b));
}
__device__ __forceinline__ long long site_add(long long e, long long a, long long b, unsigned &big)
{
    long long d = a - b;
    // |a - b| < 2^53 units (1/128): exact as it is; only sites within about
    // 11 sqrt(hop length) of the hop need the first rounding
    if ((unsigned)((unsigned long long)d >> 32) + (1u << 21) >= (1u << 22)) {
        unsigned none = 0;
        d = fix_round53(d, none);
    }
    return fix_round53(e + d, big);
}

// Square lattice: thread -> base column bx < L/2, base rows by0, by0 + rpp, ...
// A base site serves (x, y), (x + L/2, y), (x, y + L/2), (x + L/2, y + L/2): on
// an even ring fold(d + L/2) = L/2 - fold(d), so one folded offset per axis
// serves all four.
// big: see fix_round53 (long long energies).
template <typename Real, int kThreads, bool kPow2>
__device__ __forceinline__ void update_square(bool on, int off_eps, int off_tinv, unsigned ui,
                                              unsigned uj, int L, int log2L, unsigned magic,
                                              unsigned &big)
{
    const int tid = threadIdx.x;
    const int Lh = L >> 1, H1 = Lh + 1;
    const int rpp = kThreads / Lh;
    if (on && tid < rpp * Lh) {
        const int bx = tid % Lh, by0 = tid / Lh;
        const int yi = kPow2 ? (int)(ui >> log2L) : (int)__umulhi(ui, magic);
        const int yj = kPow2 ? (int)(uj >> log2L) : (int)__umulhi(uj, magic);
        const int xi = (int)ui - yi * L, xj = (int)uj - yj * L;
        const int fxj = fold_axis(bx - xj, L), fxi = fold_axis(bx - xi, L);
        // columns of (x, .) and (x + L/2, .) relative to j and to i
        const Real *tinv = &sm<Real>(off_tinv);
        const Real *cj0 = tinv + fxj, *cj1 = tinv + (Lh - fxj);
        const Real *ci0 = tinv + fxi, *ci1 = tinv + (Lh - fxi);
        const int LhH1 = Lh * H1, LhL = Lh * L;
        Real *e = &sm<Real>(off_eps, by0 * L + bx);
#pragma unroll 4
        for (int y = by0; y < Lh; y += rpp, e += rpp * L) {
            int fyj, fyi;
            if (kPow2) {
                const int dj = (y - yj) & (L - 1), di = (y - yi) & (L - 1);
                fyj = min(dj, L - dj);
                fyi = min(di, L - di);
            } else {
                fyj = fold_axis(y - yj, L);
                fyi = fold_axis(y - yi, L);
            }
            // rows fold(y - .) and L/2 - fold(y - .) = fold(y + L/2 - .)
            const int oj0 = fyj * H1, oj1 = LhH1 - oj0;
            const int oi0 = fyi * H1, oi1 = LhH1 - oi0;
            const Real a00 = cj0[oj0], b00 = ci0[oi0];
            const Real a10 = cj1[oj0], b10 = ci1[oi0];
            const Real a01 = cj0[oj1], b01 = ci0[oi1];
            const Real a11 = cj1[oj1], b11 = ci1[oi1];
            e[0] = site_add(e[0], a00, b00, big);
            e[Lh] = site_add(e[Lh], a10, b10, big);
            e[LhL] = site_add(e[LhL], a01, b01, big);
            e[LhL + Lh] = site_add(e[LhL + Lh], a11, b11, big);
        }
    }
}

// Cubic lattice: thread -> base column bx < L/2 and base (y, z) planes p0,
// p0 + rpp, ...; each base site (x, y, z) < L/2 serves the eight sites
// (x + a L/2, y + b L/2, z + c L/2), a, b, c in {0, 1}.
template <typename Real, int kThreads, bool kPow2>
__device__ __forceinline__ void update_cubic(bool on, int off_eps, int off_tinv, unsigned ui,
                                             unsigned uj, int L, int log2L, unsigned magic,
                                             unsigned &big)
{
    const int tid = threadIdx.x;
    const int Lh = L >> 1, H1 = Lh + 1;
    const int rpp = kThreads / Lh;
    if (on && tid < rpp * Lh) {
        const int bx = tid % Lh, p0 = tid / Lh;
        int xi, yi, zi, xj, yj, zj;
        if (kPow2) {
            const int m = L - 1;
            xi = (int)ui & m; yi = (int)(ui >> log2L) & m; zi = (int)(ui >> (2 * log2L));
            xj = (int)uj & m; yj = (int)(uj >> log2L) & m; zj = (int)(uj >> (2 * log2L));
        } else {
            const unsigned qi = __umulhi(ui, magic), qj = __umulhi(uj, magic);
            xi = (int)(ui - qi * (unsigned)L); zi = (int)__umulhi(qi, magic);
            yi = (int)qi - zi * L;
            xj = (int)(uj - qj * (unsigned)L); zj = (int)__umulhi(qj, magic);
            yj = (int)qj - zj * L;
        }
        const int fxj = fold_axis(bx - xj, L), fxi = fold_axis(bx - xi, L);
        const Real *tinv = &sm<Real>(off_tinv);
        const Real *cj0 = tinv + fxj, *cj1 = tinv + (Lh - fxj);
        const Real *ci0 = tinv + fxi, *ci1 = tinv + (Lh - fxi);
        const int LL = L * L;
#pragma unroll 2
        for (int pz = p0; pz < Lh * Lh; pz += rpp) {
            int by, bz, fyj, fyi, fzj, fzi;
            if (kPow2) {
                // power-of-two L: shifts, masks and a min for the folds
                by = pz & (Lh - 1);
                bz = pz >> (log2L - 1);
                const int m = L - 1;
                const int dyj = (by - yj) & m, dyi = (by - yi) & m;
                const int dzj = (bz - zj) & m, dzi = (bz - zi) & m;
                fyj = min(dyj, L - dyj); fyi = min(dyi, L - dyi);
                fzj = min(dzj, L - dzj); fzi = min(dzi, L - dzi);
            } else {
                by = pz % Lh;
                bz = pz / Lh;
                fyj = fold_axis(by - yj, L); fyi = fold_axis(by - yi, L);
                fzj = fold_axis(bz - zj, L); fzi = fold_axis(bz - zi, L);
            }
            // rows (fz H1 + fy) H1 of the folded table for the four
            // (z, y) images of the base site, relative to j and to i
            int oj[2][2], oi[2][2];
#pragma unroll
            for (int cz = 0; cz < 2; ++cz)
#pragma unroll
                for (int cy = 0; cy < 2; ++cy) {
                    oj[cz][cy] = ((cz ? Lh - fzj : fzj) * H1 + (cy ? Lh - fyj : fyj)) * H1;
                    oi[cz][cy] = ((cz ? Lh - fzi : fzi) * H1 + (cy ? Lh - fyi : fyi)) * H1;
                }
            Real *e = &sm<Real>(off_eps, (bz * L + by) * L + bx);
            // odd base rows take the two x-images in swapped order, so
            // the half-warps of consecutive rows (L/2 = 16) touch
            // opposite halves of the banks at each access
            const int sw = p0 & 1;
#pragma unroll
            for (int cz = 0; cz < 2; ++cz)
#pragma unroll
                for (int cy = 0; cy < 2; ++cy)
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        const int cx = c ^ sw;
                        const Real ta = (cx ? cj1 : cj0)[oj[cz][cy]];
                        const Real tb = (cx ? ci1 : ci0)[oi[cz][cy]];
                        Real *ep = e + cz * Lh * LL + cy * Lh * L + cx * Lh;
                        *ep = site_add(*ep, ta, tb, big);
                    }
        }
    }
}

}  // namespace cg
