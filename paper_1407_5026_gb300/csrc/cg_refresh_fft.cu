// cg_refresh_fft.cu -- the binary32 refresh of eps from its definition below
// Eq. 2 by the convolution theorem.  On the periodic lattice
//     eps_s - phi_s = sum_t g(s - t) (n_t - nu),
// g the minimum-image 1/r with g(0) = 0, is a circular convolution, so
// eps - phi = IDFT(DFT(n - nu) . DFT(g)).  g is even, so DFT(g) is real and
// two replicas share one complex transform: z = a + i b (a, b = n - nu of the
// two) gives IDFT(DFT(z) . DFT(g)) = (a * g) + i (b * g).
//
// Two forms.  The sides of refresh_fft_plane keep a whole plane in one CTA (below,
// "Planes in one CTA").  The other
// sides 2^m and 3 2^m (the smallest ones and those past that range) run in
// passes: transforms in binary32 along one axis per pass, W lines
// per CTA in shared memory.  L = 2^m: a forward pass loads in bit-reversed
// order and runs radix-2 decimation-in-time butterflies (natural-order
// output); an inverse pass runs decimation-in-frequency butterflies on
// natural-order input and stores from the bit-reversed positions.  L = 3M
// (M = 2^m), both directions: with n = M n1 + n2 and k = k1 + 3 k2,
//     X[k1 + 3 k2] = sum_n2 W_M^(n2 k2) W_L^(n2 k1) sum_n1 W_3^(n1 k1) x[M n1 + n2],
// a radix-3 step over the thirds of the line with the twiddles W_L^(n2 k1),
// then an M-point decimation-in-frequency transform of each third; X[k]
// sits at (k mod 3) M + bitrev(k / 3).  Passes:
//   square lattice: forward x (from the bitmasks) | forward y, times
//                   DFT(g)/N, inverse y | inverse x (into eps);
//   cubic lattice:  forward x | forward y | forward z, times DFT(g)/N,
//                   inverse z | inverse y | inverse x (into eps).
// The last pass adds phi (all of its 53 bits; see refresh_site), stores eps
// rounded once to binary32 and records the largest |eps_old - eps_new| of each replica, as the other
// refresh paths do.  The product's table DFT(g)/N and the twiddles
// exp(-2 pi i k / L) are computed on the host in binary64.
#include "cg_device.cuh"
#include "cg_internal.h"

namespace cg {

namespace {

constexpr int kFftThreads = 256;

struct FftArgs {
    const DevReplica *reps;
    const int *index;     // the group's replicas, in group order
    int R, L, log2L, W;   // replicas; side (log2L: of a power-of-two L); lines per CTA
    int M3, log2M;        // L = 3 M3 (0 for a power-of-two L), log2 M3
    float2 *buf;          // ceil(R/2) x N complex values
    const float *ghat;    // N: DFT(g) / N
    const float2 *tw;     // L: exp(-2 pi i k / L)
};

__device__ __forceinline__ float2 cmul(float2 a, float2 b)
{
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}

__device__ __forceinline__ unsigned bitrev(unsigned k, int log2L)
{
    return __brev(k) >> (32 - log2L);
}

// Element (w, k) of line group g of pair p along `axis`: its site index.
// axis 0: rows g W + w, element k along x; axis 1: z = g / (L/W), columns
// x0 + w, element k along y; axis 2: y = g / (L/W), columns x0 + w,
// element k along z.
__device__ __forceinline__ unsigned site_of(int axis, int g, int w, int k, int L, int W)
{
    if (axis == 0) return (unsigned)((g * W + w) * L + k);
    const int per = L / W;
    const int o = g / per, x0 = (g - o * per) * W;
    if (axis == 1) return (unsigned)((o * L + k) * L + x0 + w);
    return (unsigned)((k * L + o) * L + x0 + w);
}

// Radix-2 decimation in time on W lines of length L in shared memory (line
// stride Ls), input in bit-reversed order; conj: the inverse transform.
__device__ __forceinline__ void dit(float2 *s, int Ls, const FftArgs &a, bool conj)
{
    const int L = a.L, half = L >> 1, nb = a.W * half;
    for (int st = 0; st < a.log2L; ++st) {
        const int h = 1 << st;
        for (int b = threadIdx.x; b < nb; b += kFftThreads) {
            const int w = b >> (a.log2L - 1), j = b & (half - 1);
            const int pos = j & (h - 1), i0 = ((j >> st) << (st + 1)) + pos, i1 = i0 + h;
            float2 t = a.tw[pos << (a.log2L - 1 - st)];
            if (conj) t.y = -t.y;
            float2 *l = s + w * Ls;
            const float2 x0 = l[i0], u = cmul(l[i1], t);
            l[i0] = make_float2(x0.x + u.x, x0.y + u.y);
            l[i1] = make_float2(x0.x - u.x, x0.y - u.y);
        }
        __syncthreads();
    }
}

// Radix-2 decimation in frequency, natural-order input, bit-reversed output.
__device__ __forceinline__ void dif(float2 *s, int Ls, const FftArgs &a, bool conj)
{
    const int L = a.L, half = L >> 1, nb = a.W * half;
    for (int st = a.log2L - 1; st >= 0; --st) {
        const int h = 1 << st;
        for (int b = threadIdx.x; b < nb; b += kFftThreads) {
            const int w = b >> (a.log2L - 1), j = b & (half - 1);
            const int pos = j & (h - 1), i0 = ((j >> st) << (st + 1)) + pos, i1 = i0 + h;
            float2 t = a.tw[pos << (a.log2L - 1 - st)];
            if (conj) t.y = -t.y;
            float2 *l = s + w * Ls;
            const float2 x0 = l[i0], x1 = l[i1];
            l[i0] = make_float2(x0.x + x1.x, x0.y + x1.y);
            l[i1] = cmul(make_float2(x0.x - x1.x, x0.y - x1.y), t);
        }
        __syncthreads();
    }
}

// L = 3 M: the radix-3 step with its twiddles, then an M-point
// decimation-in-frequency transform of each third (natural-order input;
// X[k] at (k mod 3) M + bitrev(k / 3)).  conj: the inverse transform.
__device__ __forceinline__ void mixed3(float2 *s, int Ls, const FftArgs &a, bool conj)
{
    const int M = a.M3, lm = a.log2M, nb3 = a.W * M;
    const float c = 0.8660254037844386f;                  // sqrt(3) / 2
    for (int b = threadIdx.x; b < nb3; b += kFftThreads) {
        const int w = b >> lm, n2 = b & (M - 1);
        float2 *l = s + w * Ls;
        const float2 x0 = l[n2], x1 = l[M + n2], x2 = l[2 * M + n2];
        const float2 s1 = make_float2(x1.x + x2.x, x1.y + x2.y);
        const float2 d1 = make_float2(x1.x - x2.x, x1.y - x2.y);
        const float2 t = make_float2(fmaf(-0.5f, s1.x, x0.x), fmaf(-0.5f, s1.y, x0.y));
        const float sg = conj ? -1.0f : 1.0f;
        float2 y1 = make_float2(fmaf(sg * c, d1.y, t.x), fmaf(-sg * c, d1.x, t.y));
        float2 y2 = make_float2(fmaf(-sg * c, d1.y, t.x), fmaf(sg * c, d1.x, t.y));
        float2 w1 = a.tw[n2], w2 = a.tw[2 * n2];
        if (conj) {
            w1.y = -w1.y;
            w2.y = -w2.y;
        }
        l[n2] = make_float2(x0.x + s1.x, x0.y + s1.y);
        l[M + n2] = cmul(y1, w1);
        l[2 * M + n2] = cmul(y2, w2);
    }
    __syncthreads();
    const int half = M >> 1, nb = a.W * 3 * half;
    for (int st = lm - 1; st >= 0; --st) {
        const int h = 1 << st;
        for (int b = threadIdx.x; b < nb; b += kFftThreads) {
            const int sub = b >> (lm - 1), j = b & (half - 1);
            const int w = sub / 3, k1 = sub - 3 * w;
            const int pos = j & (h - 1), i0 = ((j >> st) << (st + 1)) + pos, i1 = i0 + h;
            float2 t = a.tw[3 * (pos << (lm - 1 - st))];        // W_M^(pos M / 2h)
            if (conj) t.y = -t.y;
            float2 *l = s + w * Ls + k1 * M;
            const float2 x0 = l[i0], x1 = l[i1];
            l[i0] = make_float2(x0.x + x1.x, x0.y + x1.y);
            l[i1] = cmul(make_float2(x0.x - x1.x, x0.y - x1.y), t);
        }
        __syncthreads();
    }
}

// Position in the line of output element k after a transform: L = 3 M
// (either direction), or L = 2^m after the inverse (decimation in frequency).
__device__ __forceinline__ int out_pos(int k, const FftArgs &a, bool dif_out)
{
    if (a.M3) {
        const int k2 = k / 3;
        return (k - 3 * k2) * a.M3 + (int)bitrev((unsigned)k2, a.log2M);
    }
    return dif_out ? (int)bitrev((unsigned)k, a.log2L) : k;
}

// a + b and its rounding error (Knuth's two-sum: the pair's sum is a + b exactly).
__device__ __forceinline__ float2 two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    return make_float2(s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb)));
}

// The transforms took n - nu with nu rounded to binary32; sum_t g(s-t) = C0 for
// every s, so (nu_f - nu) C0 restores the exact nu.
__device__ __forceinline__ double nu_shift(const DevReplica &R)
{
    return d_mul(d_sub((double)(float)R.nu, R.nu), R.C0);
}

// What a CTA keeps of its pair in shared memory.  Values and maxima that take
// binary64 are formed once per CTA: 28 conversions and sums in every thread
// filled a third of the kernel's time with that pipe (304 replicas of L = 128:
// 50 us).
struct PairShared {
    float2 shift[2];               // nu_shift as the sum of two binary32 numbers
    float nu[2];
    unsigned long long err[2];     // largest change of refresh_site64, binary64 bits
    float3 most[2][32];            // the warps' largest other changes
};

// By the first two threads of a CTA; a barrier before the first use.
__device__ __forceinline__ void pair_consts(PairShared &k, const DevReplica &Ra,
                                            const DevReplica &Rb)
{
    if (threadIdx.x < 2) {
        const DevReplica &R = threadIdx.x ? Rb : Ra;
        const double c = nu_shift(R);
        const float h = (float)c;
        k.shift[threadIdx.x] = make_float2(h, (float)d_sub(c, (double)h));
        k.nu[threadIdx.x] = (float)R.nu;
        k.err[threadIdx.x] = 0ull;
    }
}

// eps_new of a site in binary64, for the values that refresh_site leaves out; the
// change goes into err (NaN is not counted).
__device__ __noinline__ float refresh_site64(double phi, float v, const DevReplica &R,
                                             float eps_old, unsigned long long *err)
{
    const double e = d_add(phi, d_add((double)v, nu_shift(R)));
    const double change = fabs(d_sub((double)eps_old, e));
    if (change >= 0.0) atomicMax(err, (unsigned long long)__double_as_longlong(change));
    return __double2float_rn(e);
}

// eps_new = phi + (v + c) rounded once to binary32, c = c.x + c.y = nu_shift, and
// the change |eps_old - (phi + (v + c))|, kept in `most` as the sum of three
// binary32 numbers if it is the thread's largest so far.  phi's 53 bits are taken
// apart into 24 + 15 + 14 and summed with v and c by two-sums, whose errors are
// kept down to the fourth: what is lost is below 2^-63 of the terms, where the
// same sum in binary64 loses 2^-53 (over W = 0 to 14 and c up to 2e-5, the largest
// error of a change near 1e-6: 9e-19 against 1.3e-15).  In binary64 the step is ten
// operations per site at 1/64 of the binary32 rate; with 24 bits of each part, and
// the change in binary32, a resume is 1 to 5% faster (304 replicas of L = 128 230
// against 234 us, 128 of L = 112 124 against 130) and a change 1e3 to 1e5 times as
// far off.  A phi that is not 0 and outside
// 2^-74 to 2^78, and an eps_old past 2^100, are left to binary64.
__device__ __forceinline__ float refresh_site(double phi, float v, float2 c, float eps_old,
                                              const DevReplica &R, unsigned long long *err,
                                              float3 &most)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(phi);
    const bool zero = (b << 1) == 0ull;
    const int ex = zero ? 949 : (int)((b >> 52) & 0x7ffull);
    if ((unsigned)(ex - 949) > 1100u - 949u || !(fabsf(eps_old) < 0x1p100f))
        return refresh_site64(phi, v, R, eps_old, err);
    const unsigned sign = (unsigned)(b >> 63) << 31;
    const float hi = zero ? 0.0f
                          : __uint_as_float(sign | ((unsigned)(ex - 896) << 23) |
                                            ((unsigned)(b >> 29) & 0x7fffffu));
    const float unit = __uint_as_float(sign | ((unsigned)(ex - 948) << 23));  // 2^(ex - 1075)
    // the lower 29 bits as 15 + 14: integers below 2^23 in the mantissa of 2^23
    // (a conversion instruction runs at an eighth of this rate)
    const float i1 = __uint_as_float(0x4b000000u | (((unsigned)b >> 14) & 0x7fffu)) - 0x1p23f;
    const float i2 = __uint_as_float(0x4b000000u | ((unsigned)b & 0x3fffu)) - 0x1p23f;
    const float l1 = __fmul_rn(i1 * 0x1p14f, unit), l2 = __fmul_rn(i2, unit);
    const float2 p = two_sum(hi, v), q = two_sum(l1, c.x), t = two_sum(p.y, q.x);
    const float u = __fadd_rn(__fadd_rn(q.y, t.y), __fadd_rn(l2, c.y));
    const float2 r = two_sum(p.x, t.x);
    const float2 d = two_sum(eps_old, -r.x), k = two_sum(d.y, -r.y), x = two_sum(d.x, k.x);
    float2 y = two_sum(x.y, __fsub_rn(k.y, u));
    const bool neg = x.x < 0.0f || (x.x == 0.0f && y.x < 0.0f);
    const float m = fabsf(x.x), n = neg ? -y.x : y.x;
    if (m > most.x || (m == most.x && n > most.y)) most = make_float3(m, n, neg ? -y.y : y.y);
    return __fadd_rn(r.x, __fadd_rn(r.y, u));
}

// The larger of two changes (sums of three binary32 numbers, largest first).
__device__ __forceinline__ float3 larger(float3 a, float3 b)
{
    return b.x > a.x || (b.x == a.x && b.y > a.y) ? b : a;
}
__device__ __forceinline__ float3 warp_most(float3 c)
{
#pragma unroll
    for (int o = 16; o; o >>= 1)
        c = larger(c, make_float3(__shfl_xor_sync(0xffffffffu, c.x, o),
                                  __shfl_xor_sync(0xffffffffu, c.y, o),
                                  __shfl_xor_sync(0xffffffffu, c.z, o)));
    return c;
}

// The block's maxima of the changes of two replicas into their counters.
__device__ __forceinline__ void record_change(float3 ca, float3 cb, bool two, bool count,
                                              DevCounters *da, DevCounters *db, PairShared &ps)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    ca = warp_most(ca);
    cb = warp_most(cb);
    if (lane == 0) {
        ps.most[0][warp] = ca;
        ps.most[1][warp] = cb;
    }
    __syncthreads();
    if (warp) return;
    for (int r = 0; r < (two ? 2 : 1); ++r) {
        const float3 c = warp_most(ps.most[r][lane < (int)(blockDim.x >> 5) ? lane : 0]);
        if (lane) continue;
        DevCounters *d = r ? db : da;
        // non-negative binary64 numbers order as their bits
        const double v = d_add((double)c.x, d_add((double)c.y, (double)c.z));
        const unsigned long long b = (unsigned long long)__double_as_longlong(v);
        atomicMax(&d->max_err_bits, b > ps.err[r] ? b : ps.err[r]);
        if (count) atomicAdd(&d->refreshes, 1ull);
    }
}

// The refresh's record of the largest change starts again (thread 0 of a CTA
// that runs before every record_change of the pair).
__device__ __forceinline__ void clear_change(bool two, DevCounters *da, DevCounters *db)
{
    if (threadIdx.x == 0) {
        da->max_err_bits = 0ull;
        if (two) db->max_err_bits = 0ull;
    }
}

// One pass over W lines of one pair.  kMode: 0 forward x from the bitmasks;
// 1 forward (buffer to buffer); 2 forward, product with DFT(g)/N, inverse
// (the last axis); 3 inverse (buffer to buffer); 4 inverse x into eps.
// grid.x = pairs x line groups per pair.
template <int kMode>
__global__ void __launch_bounds__(kFftThreads) fft_pass_kernel(FftArgs a, int axis)
{
    extern __shared__ float2 s[];
    __shared__ PairShared ps;
    const int L = a.L, W = a.W, Ls = L + 1;     // padded line stride (banks)
    const int groups = (int)(gridDim.x / (unsigned)((a.R + 1) / 2));
    const int p = blockIdx.x / groups, g = blockIdx.x - p * groups;
    const DevReplica &Ra = a.reps[a.index[2 * p]];
    const bool two = 2 * p + 1 < a.R;
    const DevReplica &Rb = a.reps[a.index[two ? 2 * p + 1 : 2 * p]];
    const unsigned Nr = (unsigned)Ra.N;                    // L^2 or L^3
    float2 *buf = a.buf + (size_t)p * Nr;
    const int n = W * L;
    const bool mixed = a.M3 != 0;
    // natural-order load for the inverse and for every L = 3 M transform
    const bool natural_in = kMode >= 3 || mixed;
    // ---- load ----
    for (int e = threadIdx.x; e < n; e += kFftThreads) {
        int w, k;
        if (axis == 0) { w = e / L; k = e - w * L; } else { k = e / W; w = e - k * W; }
        const unsigned site = site_of(axis, g, w, k, L, W);
        float2 v;
        if (kMode == 0) {
            const float na = (float)((Ra.occ[site >> 5] >> (site & 31)) & 1u) - (float)Ra.nu;
            const float nb = two ? (float)((Rb.occ[site >> 5] >> (site & 31)) & 1u) - (float)Rb.nu
                                 : 0.0f;
            v = make_float2(na, nb);
        } else {
            v = buf[site];
        }
        s[w * Ls + (natural_in ? k : (int)bitrev((unsigned)k, a.log2L))] = v;
    }
    if (kMode == 4) pair_consts(ps, Ra, Rb);
    __syncthreads();
    // ---- transform ----
    float2 *out = s;                                       // where the result lies
    if (!mixed) {
        if (kMode <= 2) dit(s, Ls, a, false);
        if (kMode == 2) {
            for (int e = threadIdx.x; e < n; e += kFftThreads) {
                int w, k;
                if (axis == 0) { w = e / L; k = e - w * L; } else { k = e / W; w = e - k * W; }
                const float gh = a.ghat[site_of(axis, g, w, k, L, W)];
                float2 &v = s[w * Ls + k];
                v = make_float2(v.x * gh, v.y * gh);
            }
            __syncthreads();
        }
        if (kMode >= 2) dif(s, Ls, a, true);
    } else {
        mixed3(s, Ls, a, kMode >= 3);
        if (kMode == 2) {
            // the product in natural order into the second buffer, then the
            // inverse transform there
            float2 *s2 = s + W * Ls;
            for (int e = threadIdx.x; e < n; e += kFftThreads) {
                int w, k;
                if (axis == 0) { w = e / L; k = e - w * L; } else { k = e / W; w = e - k * W; }
                const float gh = a.ghat[site_of(axis, g, w, k, L, W)];
                const float2 v = s[w * Ls + out_pos(k, a, false)];
                s2[w * Ls + k] = make_float2(v.x * gh, v.y * gh);
            }
            __syncthreads();
            mixed3(s2, Ls, a, true);
            out = s2;
        }
    }
    // ---- store ----
    float3 err_a = make_float3(0.0f, 0.0f, 0.0f), err_b = err_a;
    if (kMode != 4) {
        for (int e = threadIdx.x; e < n; e += kFftThreads) {
            int w, k;
            if (axis == 0) { w = e / L; k = e - w * L; } else { k = e / W; w = e - k * W; }
            const unsigned site = site_of(axis, g, w, k, L, W);
            buf[site] = out[w * Ls + out_pos(k, a, kMode >= 2)];
        }
    } else {
        // axis x: element e of the CTA is site g W L + e.  phi and eps of
        // different sites are independent, so four elements' loads are in
        // flight at once (restrict: eps is not phi)
        const unsigned site0 = (unsigned)(g * W) * (unsigned)L;
        const double *__restrict__ pa = Ra.phi + site0;
        const double *__restrict__ pb = Rb.phi + site0;
        float *__restrict__ ea = reinterpret_cast<float *>(Ra.eps) + site0;
        float *__restrict__ eb = reinterpret_cast<float *>(Rb.eps) + site0;
        const float2 ca = ps.shift[0], cb = ps.shift[1];
#pragma unroll 4
        for (int e = threadIdx.x; e < n; e += kFftThreads) {
            const int w = e / L, k = e - w * L;
            const float2 v = out[w * Ls + out_pos(k, a, true)];
            ea[e] = refresh_site(pa[e], v.x, ca, ea[e], Ra, &ps.err[0], err_a);
            if (two) eb[e] = refresh_site(pb[e], v.y, cb, eb[e], Rb, &ps.err[1], err_b);
        }
        record_change(err_a, err_b, two, g == 0, Ra.ctr, Rb.ctr, ps);
    }
}

// ---------------------------------------------------------------------------
// Planes in one CTA: refresh_fft_plane's sides.  On the square lattice one CTA does the whole refresh of a replica
// pair: its L x L complex values stay in shared memory (132 KiB at L = 128)
// through all the transforms, where the passes above write and read them through
// L2 between launches and run a barrier per radix-2 stage (304 replicas of
// L = 128: 0.15 -> 0.05 ms on the device).  Cubic lattices take three launches over planes
// instead of five passes (152 of 32^3: 0.243 -> 0.067 ms; 16 of 48^3: 0.104 ->
// 0.050).  Sides that are neither 2^m nor 3 2^m take the place of
// the tensor-core contraction (128 of L = 112, a resume with its copies: 329 ->
// 135 us).  What bounds it: latency of the seven sweeps and their barriers at one
// or two CTAs per SM, then the 18 N bytes of phi, eps and table from memory.
//
// A line of L = R1 8 elements transforms in two steps, in place:
//     X[c + R1 d] = sum_b W_8^(b d) W_L^(b c) sum_a W_R1^(a c) x[8 a + b]
// step 1, for each b: an R1-point transform over a (elements 8 a + b) times
// the twiddles; step 2, for each c: an 8-point transform over b (elements
// 8 c + b), leaving X[c + R1 d] at 8 c + d.  The inverse takes the steps
// backwards from that order, so nothing is ever reordered: only the product
// looks DFT(g) up by the permuted wave numbers, between the forward and the
// inverse 8-point steps of the y axis, in registers.  Seven sweeps of shared
// memory in all; the first reads the bitmasks, the last writes eps.
//
// Element (y, x) lies at y (L + 1) + (x with its low three bits xored by the
// next three): columns are contiguous across a half-warp, and the 8-element
// groups of a line spread over the banks.
// ---------------------------------------------------------------------------

template <bool kInv>
__device__ __forceinline__ float2 rot90(float2 v)         // times -i (inverse: i)
{
    return kInv ? make_float2(-v.y, v.x) : make_float2(v.y, -v.x);
}
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
// v times (wr, -wi) (inverse: its conjugate)
template <bool kInv>
__device__ __forceinline__ float2 ctw(float2 v, float wr, float wi)
{
    return cmul(v, make_float2(wr, kInv ? wi : -wi));
}

// v times exp(-i pi / 4) (inverse: exp(i pi / 4)): the sums first (exact for the
// first axis' n - nu), then 1/sqrt 2 in two parts, one rounding each.
template <bool kInv>
__device__ __forceinline__ float2 rot45(float2 v)
{
    constexpr float kS = 0.7071067811865476f;
    constexpr float kSlo = (float)(0.70710678118654752440 - (double)kS);
    const float a = v.x + v.y, b = kInv ? v.x - v.y : v.y - v.x;
    const float sa = fmaf(a, kS, a * kSlo), sb = fmaf(b, kS, b * kSlo);
    return kInv ? make_float2(sb, sa) : make_float2(sa, sb);
}

template <bool kInv>
__device__ __forceinline__ void dft2(float2 &a, float2 &b)
{
    const float2 t = csub(a, b);
    a = cadd(a, b);
    b = t;
}

template <bool kInv>
__device__ __forceinline__ void dft3(float2 &a, float2 &b, float2 &c)
{
    const float h = 0.8660254037844386f;                  // sqrt(3) / 2
    const float2 s = cadd(b, c), d = rot90<kInv>(csub(b, c));
    const float2 t = make_float2(fmaf(-0.5f, s.x, a.x), fmaf(-0.5f, s.y, a.y));
    a = cadd(a, s);
    b = make_float2(fmaf(h, d.x, t.x), fmaf(h, d.y, t.y));
    c = make_float2(fmaf(-h, d.x, t.x), fmaf(-h, d.y, t.y));
}

template <bool kInv>
__device__ __forceinline__ void dft4(float2 &a, float2 &b, float2 &c, float2 &d)
{
    const float2 t0 = cadd(a, c), t1 = csub(a, c), t2 = cadd(b, d), t3 = rot90<kInv>(csub(b, d));
    a = cadd(t0, t2);
    b = cadd(t1, t3);
    c = csub(t0, t2);
    d = csub(t1, t3);
}

// R-point transform of v in registers, natural order in and out.
template <int R, bool kInv>
__device__ __forceinline__ void dft(float2 (&v)[R])
{
    constexpr float kS = 0.7071067811865476f;             // cos(pi / 4)
    if constexpr (R == 2) {
        dft2<kInv>(v[0], v[1]);
    } else if constexpr (R == 3) {
        dft3<kInv>(v[0], v[1], v[2]);
    } else if constexpr (R == 4) {
        dft4<kInv>(v[0], v[1], v[2], v[3]);
    } else if constexpr (R == 6) {
        // n = 2 a + b, k = c + 3 d
        dft3<kInv>(v[0], v[2], v[4]);
        dft3<kInv>(v[1], v[3], v[5]);
        v[3] = ctw<kInv>(v[3], 0.5f, 0.8660254037844386f);
        v[5] = ctw<kInv>(v[5], -0.5f, 0.8660254037844386f);
        float2 o[6];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            o[c] = cadd(v[2 * c], v[2 * c + 1]);
            o[c + 3] = csub(v[2 * c], v[2 * c + 1]);
        }
#pragma unroll
        for (int k = 0; k < 6; ++k) v[k] = o[k];
    } else if constexpr (R == 8) {
        dft4<kInv>(v[0], v[2], v[4], v[6]);
        dft4<kInv>(v[1], v[3], v[5], v[7]);
        v[3] = rot45<kInv>(v[3]);
        v[5] = rot90<kInv>(v[5]);
        v[7] = rot45<kInv>(rot90<kInv>(v[7]));
        float2 o[8];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            o[c] = cadd(v[2 * c], v[2 * c + 1]);
            o[c + 4] = csub(v[2 * c], v[2 * c + 1]);
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) v[k] = o[k];
    } else if constexpr (R == 12 || R == 16) {
        // n = 4 a + b, k = c + (R/4) d: R/4-point transforms over a, the
        // twiddles W_R^(b c), 4-point transforms over b
        constexpr int P = R / 4;
        constexpr float c16[10] = {1.0f, 0.9238795325112867f, kS, 0.3826834323650898f, 0.0f,
                                   -0.3826834323650898f, -kS, -0.9238795325112867f, -1.0f,
                                   -0.9238795325112867f};
        constexpr float s16[10] = {0.0f, 0.3826834323650898f, kS, 0.9238795325112867f, 1.0f,
                                   0.9238795325112867f, kS, 0.3826834323650898f, 0.0f,
                                   -0.3826834323650898f};
        constexpr float c12[7] = {1.0f, 0.8660254037844386f, 0.5f, 0.0f, -0.5f,
                                  -0.8660254037844386f, -1.0f};
        constexpr float s12[7] = {0.0f, 0.5f, 0.8660254037844386f, 1.0f, 0.8660254037844386f, 0.5f,
                                  0.0f};
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            if constexpr (P == 4)
                dft4<kInv>(v[b], v[4 + b], v[8 + b], v[12 + b]);
            else
                dft3<kInv>(v[b], v[4 + b], v[8 + b]);
#pragma unroll
            for (int c = 1; c < P; ++c)
                if (b) {
                    const int e = b * c;
                    v[4 * c + b] = P == 4 ? ctw<kInv>(v[4 * c + b], c16[e % 10], s16[e % 10])
                                          : ctw<kInv>(v[4 * c + b], c12[e % 7], s12[e % 7]);
                }
        }
        float2 o[R];
#pragma unroll
        for (int c = 0; c < P; ++c) {
            dft4<kInv>(v[4 * c], v[4 * c + 1], v[4 * c + 2], v[4 * c + 3]);
#pragma unroll
            for (int d = 0; d < 4; ++d) o[c + P * d] = v[4 * c + d];
        }
#pragma unroll
        for (int k = 0; k < R; ++k) v[k] = o[k];
    }
}

// CTA size of a plane's transforms: one item per thread in the 8-point steps of
// up to 512 threads (128 registers; R1 > 12 holds 4 R1 of them), L = 128 on 1024.
template <int L>
constexpr int fft_plane_threads()
{
    return L == 128 ? 1024 : L * L / 8 >= 512 ? 512 : (L * L / 8 + 31) / 32 * 32;
}

// R-point transform of v for the R1 that dft has no steps for: the plain sum,
// W_R^k = W_L^(8 k) from the shared twiddles (the same word for the whole warp).
template <int L, bool kInv>
__device__ __forceinline__ void dft_r1(float2 (&v)[L / 8], const float2 *tw)
{
    constexpr int R = L / 8;
    if constexpr (R == 2 || R == 3 || R == 4 || R == 6 || R == 8 || R == 12 || R == 16) {
        dft<R, kInv>(v);
    } else {
        float2 o[R];
#pragma unroll
        for (int k = 0; k < R; ++k) o[k] = v[0];
#pragma unroll
        for (int n = 1; n < R; ++n) {
            o[0] = cadd(o[0], v[n]);
#pragma unroll
            for (int k = 1; k < R; ++k) {
                float2 w = tw[8 * ((n * k) % R)];
                if (kInv) w.y = -w.y;
                o[k].x = fmaf(v[n].x, w.x, fmaf(-v[n].y, w.y, o[k].x));
                o[k].y = fmaf(v[n].x, w.y, fmaf(v[n].y, w.x, o[k].y));
            }
        }
#pragma unroll
        for (int k = 0; k < R; ++k) v[k] = o[k];
    }
}

// The sweeps of one L x L plane of a pair in shared memory (see above).
template <int L>
struct Plane {
    static constexpr int R1 = L / 8, kT = fft_plane_threads<L>(), Ls = L + 1;
    static constexpr int kSmem = (L * Ls + L) * (int)sizeof(float2);
    float2 *s, *tw;
    PairShared *ps;

    __device__ __forceinline__ float2 &at(int y, int x) const
    {
        return s[y * Ls + (x & ~7) + ((x ^ (x >> 3)) & 7)];
    }
    // rows r and r + 8 share a half-warp: their 8-element runs fall in opposite
    // halves of the banks
    static __device__ __forceinline__ int row_of(int r)
    {
        return L % 16 ? r : (r & ~15) | ((r & 1) << 3) | ((r >> 1) & 7);
    }
    // item -> (row, c) of the 8-element groups of the rows
    static __device__ __forceinline__ void group_of(int it, int &y, int &c)
    {
        if (R1 % 8 == 0) {
            const int rest = it >> 4;
            c = (it & 7) + 8 * (rest % (R1 / 8));
            y = 2 * (rest / (R1 / 8)) + ((it >> 3) & 1);
        } else {
            c = it % R1;
            y = it / R1;
        }
    }
    __device__ __forceinline__ void twiddles(const float2 *g) const
    {
        for (int k = threadIdx.x; k < L; k += kT) tw[k] = g[k];
    }
    __device__ __forceinline__ float2 conj_tw(int e) const
    {
        return make_float2(tw[e].x, -tw[e].y);
    }
    // x, both forward steps, from the bitmasks of the plane at site0
    __device__ __forceinline__ void x_from_bits(const DevReplica &Ra, const DevReplica &Rb, bool two,
                                                unsigned site0) const
    {
        const float na = ps->nu[0], nb = ps->nu[1];
        for (int it = threadIdx.x; it < L * 8; it += kT) {
            const int b = it & 7, y = row_of(it >> 3);
            float2 v[R1];
#pragma unroll
            for (int k = 0; k < R1; ++k) {
                const unsigned site = site0 + (unsigned)(y * L + 8 * k + b);
                const unsigned wa = __ldg(Ra.occ + (site >> 5)), wb = __ldg(Rb.occ + (site >> 5));
                v[k] = make_float2((float)((wa >> (site & 31u)) & 1u) - na,
                                   two ? (float)((wb >> (site & 31u)) & 1u) - nb : 0.0f);
            }
            dft_r1<L, false>(v, tw);
#pragma unroll
            for (int c = 0; c < R1; ++c) at(y, 8 * c + b) = c ? cmul(v[c], tw[b * c]) : v[c];
        }
        __syncthreads();
        for (int it = threadIdx.x; it < L * R1; it += kT) {
            int y, c;
            group_of(it, y, c);
            float2 v[8];
#pragma unroll
            for (int b = 0; b < 8; ++b) v[b] = at(y, 8 * c + b);
            dft<8, false>(v);
#pragma unroll
            for (int d = 0; d < 8; ++d) at(y, 8 * c + d) = v[d];
        }
    }
    // columns, step 1 (kGlobal: read from rows of the buffer, `row` values apart)
    template <bool kGlobal>
    __device__ __forceinline__ void col_step1(const float2 *g, size_t row) const
    {
        for (int it = threadIdx.x; it < L * 8; it += kT) {
            const int x = it % L, b = it / L;
            float2 v[R1];
#pragma unroll
            for (int k = 0; k < R1; ++k) v[k] = kGlobal ? g[(8 * k + b) * row + x] : at(8 * k + b, x);
            dft_r1<L, false>(v, tw);
#pragma unroll
            for (int c = 0; c < R1; ++c) at(8 * c + b, x) = c ? cmul(v[c], tw[b * c]) : v[c];
        }
    }
    // columns, step 2, the product with DFT(g)/N and the inverse's first step;
    // wave numbers of slot x and c + R1 d: gh[(c + R1 d) gstride + kx]
    __device__ __forceinline__ void col_product(const float *gh, size_t gstride) const
    {
        for (int it = threadIdx.x; it < L * R1; it += kT) {
            const int x = it % L, c = it / L, kx = (x >> 3) + R1 * (x & 7);
            float2 v[8];
#pragma unroll
            for (int b = 0; b < 8; ++b) v[b] = at(8 * c + b, x);
            dft<8, false>(v);
#pragma unroll
            for (int d = 0; d < 8; ++d) {
                const float g = __ldg(gh + (c + R1 * d) * gstride + kx);
                v[d] = make_float2(v[d].x * g, v[d].y * g);
            }
            dft<8, true>(v);
#pragma unroll
            for (int b = 0; b < 8; ++b) at(8 * c + b, x) = cmul(v[b], conj_tw(b * c));
        }
    }
    // columns, the inverse's second step (kGlobal: into rows of the buffer)
    template <bool kGlobal>
    __device__ __forceinline__ void col_inverse2(float2 *g, size_t row) const
    {
        for (int it = threadIdx.x; it < L * 8; it += kT) {
            const int x = it % L, b = it / L;
            float2 v[R1];
#pragma unroll
            for (int c = 0; c < R1; ++c) v[c] = at(8 * c + b, x);
            dft_r1<L, true>(v, tw);
#pragma unroll
            for (int k = 0; k < R1; ++k) {
                if (kGlobal)
                    g[(8 * k + b) * row + x] = v[k];
                else
                    at(8 * k + b, x) = v[k];
            }
        }
    }
    // columns, step 2 forward into the buffer, and back from it
    __device__ __forceinline__ void col_step2_store(float2 *g) const
    {
        for (int it = threadIdx.x; it < L * R1; it += kT) {
            const int x = it % L, c = it / L;
            float2 v[8];
#pragma unroll
            for (int b = 0; b < 8; ++b) v[b] = at(8 * c + b, x);
            dft<8, false>(v);
#pragma unroll
            for (int d = 0; d < 8; ++d) g[(8 * c + d) * L + x] = v[d];
        }
    }
    __device__ __forceinline__ void col_inverse1_load(const float2 *g) const
    {
        for (int it = threadIdx.x; it < L * R1; it += kT) {
            const int x = it % L, c = it / L;
            float2 v[8];
#pragma unroll
            for (int d = 0; d < 8; ++d) v[d] = g[(8 * c + d) * L + x];
            dft<8, true>(v);
#pragma unroll
            for (int b = 0; b < 8; ++b) at(8 * c + b, x) = cmul(v[b], conj_tw(b * c));
        }
    }
    // x, the inverse's first step
    __device__ __forceinline__ void x_inverse1() const
    {
        for (int it = threadIdx.x; it < L * R1; it += kT) {
            int y, c;
            group_of(it, y, c);
            float2 v[8];
#pragma unroll
            for (int d = 0; d < 8; ++d) v[d] = at(y, 8 * c + d);
            dft<8, true>(v);
#pragma unroll
            for (int b = 0; b < 8; ++b) at(y, 8 * c + b) = cmul(v[b], conj_tw(b * c));
        }
    }
    // x, the inverse's second step, into eps of the plane at site0; the largest
    // changes of the thread's sites
    __device__ __forceinline__ void x_into_eps(const DevReplica &Ra, const DevReplica &Rb, bool two,
                                               unsigned site0, float3 &err_a,
                                               float3 &err_b) const
    {
        const double *__restrict__ pa = Ra.phi + site0, *__restrict__ pb = Rb.phi + site0;
        float *__restrict__ ea = reinterpret_cast<float *>(Ra.eps) + site0;
        float *__restrict__ eb = reinterpret_cast<float *>(Rb.eps) + site0;
        const float2 ca = ps->shift[0], cb = ps->shift[1];
        for (int it = threadIdx.x; it < L * 8; it += kT) {
            const int b = it & 7, y = row_of(it >> 3), site = y * L + b;
            float2 v[R1];
#pragma unroll
            for (int c = 0; c < R1; ++c) v[c] = at(y, 8 * c + b);
            dft_r1<L, true>(v, tw);
            // a few elements' loads in flight at a time
            constexpr int kBatch = R1 % 4 == 0 ? 4 : R1 % 3 == 0 ? 3 : R1 % 5 == 0 ? 5 : R1 % 2 == 0 ? 2 : 1;
#pragma unroll
            for (int k0 = 0; k0 < R1; k0 += kBatch) {
                double fa[kBatch], fb[kBatch];
                float oa[kBatch], ob[kBatch];
#pragma unroll
                for (int k = 0; k < kBatch; ++k) {
                    const int e = site + 8 * (k0 + k);
                    fa[k] = pa[e];
                    oa[k] = ea[e];
                    fb[k] = two ? pb[e] : 0.0;
                    ob[k] = two ? eb[e] : 0.0f;
                }
#pragma unroll
                for (int k = 0; k < kBatch; ++k) {
                    const int e = site + 8 * (k0 + k);
                    ea[e] = refresh_site(fa[k], v[k0 + k].x, ca, oa[k], Ra, &ps->err[0], err_a);
                    if (two)
                        eb[e] = refresh_site(fb[k], v[k0 + k].y, cb, ob[k], Rb, &ps->err[1], err_b);
                }
            }
        }
    }
    // phi and eps of the plane, which the last sweep reads, on their way into L2
    __device__ __forceinline__ void prefetch(const DevReplica &R, unsigned site0) const
    {
        const char *f = reinterpret_cast<const char *>(R.phi + site0);
        const char *e = reinterpret_cast<const char *>(reinterpret_cast<const float *>(R.eps) + site0);
        for (int k = threadIdx.x * 128; k < L * L * 8; k += kT * 128)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(f + k));
        for (int k = threadIdx.x * 128; k < L * L * 4; k += kT * 128)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(e + k));
    }
};

// The square lattice: the whole refresh of a pair.
template <int L>
__global__ void __launch_bounds__(fft_plane_threads<L>()) fft_square_kernel(FftArgs a)
{
    extern __shared__ float2 s[];
    __shared__ PairShared ps;
    const Plane<L> P{s, s + L * Plane<L>::Ls, &ps};
    const int p = blockIdx.x;
    const DevReplica &Ra = a.reps[a.index[2 * p]];
    const bool two = 2 * p + 1 < a.R;
    const DevReplica &Rb = a.reps[a.index[two ? 2 * p + 1 : 2 * p]];
    P.twiddles(a.tw);
    pair_consts(ps, Ra, Rb);
    clear_change(two, Ra.ctr, Rb.ctr);
    __syncthreads();
    P.prefetch(Ra, 0u);
    if (two) P.prefetch(Rb, 0u);
    P.x_from_bits(Ra, Rb, two, 0u);
    __syncthreads();
    P.template col_step1<false>(nullptr, 0);
    __syncthreads();
    P.col_product(a.ghat, L);
    __syncthreads();
    P.template col_inverse2<false>(nullptr, 0);
    __syncthreads();
    P.x_inverse1();
    __syncthreads();
    float3 err_a = make_float3(0.0f, 0.0f, 0.0f), err_b = err_a;
    P.x_into_eps(Ra, Rb, two, 0u, err_a, err_b);
    record_change(err_a, err_b, two, true, Ra.ctr, Rb.ctr, ps);
}

// The cubic lattice in three launches over L x L planes: x and y of a z-plane
// from the bitmasks into the buffer (kStep 0); z of a (z, x) plane, the product
// and back (1); y and x back into eps (2).  The buffer holds the slots as the
// transforms leave them; only the product looks the wave numbers up.
template <int L, int kStep>
__global__ void __launch_bounds__(fft_plane_threads<L>()) fft_cubic_kernel(FftArgs a)
{
    extern __shared__ float2 s[];
    __shared__ PairShared ps;
    constexpr int R1 = L / 8;
    const Plane<L> P{s, s + L * Plane<L>::Ls, &ps};
    const int p = blockIdx.x / L, o = blockIdx.x - p * L;
    const DevReplica &Ra = a.reps[a.index[2 * p]];
    const bool two = 2 * p + 1 < a.R;
    const DevReplica &Rb = a.reps[a.index[two ? 2 * p + 1 : 2 * p]];
    float2 *buf = a.buf + (size_t)p * L * L * L;
    const unsigned site0 = (unsigned)(o * L * L);
    P.twiddles(a.tw);
    if (kStep != 1) pair_consts(ps, Ra, Rb);
    __syncthreads();
    if (kStep == 0) {
        if (o == 0) clear_change(two, Ra.ctr, Rb.ctr);
        P.x_from_bits(Ra, Rb, two, site0);
        __syncthreads();
        P.template col_step1<false>(nullptr, 0);
        __syncthreads();
        P.col_step2_store(buf + site0);
    } else if (kStep == 1) {
        // slot o of y holds wave number o / 8 + R1 (o mod 8)
        const int ky = (o >> 3) + R1 * (o & 7);
        float2 *g = buf + o * L;
        P.template col_step1<true>(g, (size_t)L * L);
        __syncthreads();
        P.col_product(a.ghat + ky * L, (size_t)L * L);
        __syncthreads();
        P.template col_inverse2<true>(g, (size_t)L * L);
    } else {
        P.prefetch(Ra, site0);
        if (two) P.prefetch(Rb, site0);
        P.col_inverse1_load(buf + site0);
        __syncthreads();
        P.template col_inverse2<false>(nullptr, 0);
        __syncthreads();
        P.x_inverse1();
        __syncthreads();
        float3 err_a = make_float3(0.0f, 0.0f, 0.0f), err_b = err_a;
        P.x_into_eps(Ra, Rb, two, site0, err_a, err_b);
        record_change(err_a, err_b, two, o == 0, Ra.ctr, Rb.ctr, ps);
    }
}

template <int L>
cudaError_t launch_square(const FftArgs &a, int pairs, cudaStream_t st)
{
    const cudaError_t e = cudaFuncSetAttribute(
        fft_square_kernel<L>, cudaFuncAttributeMaxDynamicSharedMemorySize, Plane<L>::kSmem);
    if (e) return e;
    fft_square_kernel<L><<<pairs, Plane<L>::kT, Plane<L>::kSmem, st>>>(a);
    return cudaGetLastError();
}

template <int L>
cudaError_t launch_cubic(const FftArgs &a, int pairs, cudaStream_t st)
{
    // planes of up to 64 x 64 values: 33 KiB
    fft_cubic_kernel<L, 0><<<pairs * L, Plane<L>::kT, Plane<L>::kSmem, st>>>(a);
    fft_cubic_kernel<L, 1><<<pairs * L, Plane<L>::kT, Plane<L>::kSmem, st>>>(a);
    fft_cubic_kernel<L, 2><<<pairs * L, Plane<L>::kT, Plane<L>::kSmem, st>>>(a);
    return cudaGetLastError();
}

template <int kMode>
cudaError_t launch_pass(const FftArgs &a, int axis, int pairs, int groups, cudaStream_t st)
{
    // L = 3 M: the middle pass keeps a second buffer for the product
    const int smem = (a.M3 && kMode == 2 ? 2 : 1) * a.W * (a.L + 1) * (int)sizeof(float2);
    cudaError_t e = cudaFuncSetAttribute(fft_pass_kernel<kMode>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e) return e;
    fft_pass_kernel<kMode><<<pairs * groups, kFftThreads, smem, st>>>(a, axis);
    return cudaGetLastError();
}

}  // namespace

// lines per CTA: the largest power of two up to 16 that divides L (the y and
// z passes take W adjacent columns) with W L <= 8192 values of shared memory
static int refresh_fft_lines(int L)
{
    int W = 16;
    while (W > 1 && (L % W != 0 || W * L > 8192)) W >>= 1;
    return W;
}

// The sides 2^m (4 <= L <= 1024) and 3 2^m (6 <= L <= 192).
bool refresh_fft_size_ok(int L)
{
    if (L >= 4 && L <= 1024 && (L & (L - 1)) == 0) return true;
    const int M = L / 3;
    return L % 3 == 0 && L >= 6 && L <= 192 && (M & (M - 1)) == 0;
}

// Sides of the per-plane transforms: multiples of 16 to 160 and 24 (square), and
// 16, 24, 32, 48, 64 (cubic: at 40 and 56 the contraction's binary16 split is the
// more exact).  They clear the replicas' error records themselves (else
// launch_reset_refresh_err comes first).
bool refresh_fft_plane(int L, int dim)
{
    if (L == 24 && dim == 2) return true;
    if (dim == 3) return refresh_fft_size_ok(L) && L >= 16 && L <= 64;
    return L % 16 == 0 && L >= 16 && L <= 160;
}

cudaError_t launch_refresh_fft(const DevReplica *d_reps, const int *d_index, int R, int L,
                               int dim, const float *d_ghat, const float2 *d_tw, float2 *d_buf,
                               cudaStream_t st)
{
    if (!d_ghat || !d_tw || !d_buf) return cudaErrorInvalidValue;
    if (R < 1 || !(refresh_fft_size_ok(L) || refresh_fft_plane(L, dim)) || (dim != 2 && dim != 3)) return cudaErrorInvalidValue;
    FftArgs a;
    a.reps = d_reps;
    a.index = d_index;
    a.R = R;
    a.L = L;
    const bool pow2 = (L & (L - 1)) == 0;
    a.log2L = pow2 ? __builtin_ctz((unsigned)L) : 0;
    a.M3 = pow2 ? 0 : L / 3;              // (read by the passes alone)
    a.log2M = pow2 ? 0 : __builtin_ctz((unsigned)(L / 3));
    a.W = refresh_fft_lines(L);
    a.buf = d_buf;
    a.ghat = d_ghat;
    a.tw = d_tw;
    const int pairs = (R + 1) / 2;
    const int lines = dim == 3 ? L * L : L;              // lines per axis per pair
    const int groups = lines / a.W;
    cudaError_t e;
    if (dim == 2) {
        // a pair per CTA where its values fit shared memory (206 KiB at L = 160)
        switch (L) {
#define CG_SIDE(n) case n: return launch_square<n>(a, pairs, st);
        CG_SIDE(16) CG_SIDE(24) CG_SIDE(32) CG_SIDE(48) CG_SIDE(64) CG_SIDE(80) CG_SIDE(96)
        CG_SIDE(112) CG_SIDE(128) CG_SIDE(144) CG_SIDE(160)
#undef CG_SIDE
        }
        if ((e = launch_pass<0>(a, 0, pairs, groups, st))) return e;
        if ((e = launch_pass<2>(a, 1, pairs, groups, st))) return e;
        return launch_pass<4>(a, 0, pairs, groups, st);
    }
    switch (L) {
#define CG_SIDE(n) case n: return launch_cubic<n>(a, pairs, st);
    CG_SIDE(16) CG_SIDE(24) CG_SIDE(32) CG_SIDE(48) CG_SIDE(64)
#undef CG_SIDE
    }
    if ((e = launch_pass<0>(a, 0, pairs, groups, st))) return e;
    if ((e = launch_pass<1>(a, 1, pairs, groups, st))) return e;
    if ((e = launch_pass<2>(a, 2, pairs, groups, st))) return e;
    if ((e = launch_pass<3>(a, 1, pairs, groups, st))) return e;
    return launch_pass<4>(a, 0, pairs, groups, st);
}

size_t refresh_fft_buffer_bytes(int N, int R) { return (size_t)((R + 1) / 2) * (size_t)N * 8; }

}  // namespace cg
