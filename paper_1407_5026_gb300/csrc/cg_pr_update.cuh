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

// Square lattice: thread -> base column bx < L/2, base rows by0, by0 + rpp, ...
// A base site serves (x, y), (x + L/2, y), (x, y + L/2), (x + L/2, y + L/2): on
// an even ring fold(d + L/2) = L/2 - fold(d), so one folded offset per axis
// serves all four.
template <typename Real, int kThreads, bool kPow2>
__device__ __forceinline__ void update_square(bool on, int off_eps, int off_tinv, unsigned ui, unsigned uj,
                                              int L, int log2L, unsigned magic)
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
            e[0] = Prec<Real>::add(e[0], Prec<Real>::sub(a00, b00));
            e[Lh] = Prec<Real>::add(e[Lh], Prec<Real>::sub(a10, b10));
            e[LhL] = Prec<Real>::add(e[LhL], Prec<Real>::sub(a01, b01));
            e[LhL + Lh] = Prec<Real>::add(e[LhL + Lh], Prec<Real>::sub(a11, b11));
        }
    }
}

// Cubic lattice: thread -> base column bx < L/2 and base (y, z) planes p0,
// p0 + rpp, ...; each base site (x, y, z) < L/2 serves the eight sites
// (x + a L/2, y + b L/2, z + c L/2), a, b, c in {0, 1}.
template <typename Real, int kThreads, bool kPow2>
__device__ __forceinline__ void update_cubic(bool on, int off_eps, int off_tinv, unsigned ui, unsigned uj,
                                             int L, int log2L, unsigned magic)
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
                        *ep = Prec<Real>::add(*ep, Prec<Real>::sub(ta, tb));
                    }
        }
    }
}

}  // namespace cg
