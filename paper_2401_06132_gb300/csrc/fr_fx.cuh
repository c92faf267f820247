// fr_fx.cuh -- 64-bit block fixed-point arithmetic for the linear operators of the FP64 kernels.
//
// GB300 issues 1.6 FP64 multiply-adds per clock and SM, but 32 wide integer multiplications
// (32 x 32 -> 64 bits; both measured, dependent-free streams), so about ten terms of a fixed-point
// sum (eight in the kernels' loops). The interpolation, projection,
// differentiation and trace operators are constant matrices applied to a block of values (one field of
// one element), so they run in fixed point: the block is scaled by one power of two, taken from its
// largest magnitude, to integers below 2^56, and every product-sum is exact in 64-bit integers down
// to 2^-58 of the block's bound, where an FP64 sum rounds each step at 2^-53 of its running value.
// The power of two travels beside the block; values return to FP64 for the pointwise fluxes.
//
// A value X is held as two limbs X = h 2^28 + l (0 <= l < 2^28), a coefficient C = round(c 2^(58-k))
// as C = H 2^28 + L (|L| <= 2^27; k is the operator's scale, FX_KD, FX_KP or FX_KL). A term of a sum
// takes three wide products, each added to a 64-bit sum: hh += H h, mm += H l + L h; the dropped L l is below 2^-57 of the
// term's bound. The sum is Y = hh + (mm >> 28), in units of X 2^(k - 2). Bounds, for operators whose
// absolute row sums are at most 2 after scaling and |X| < 2^59: |h| < 2^31, |hh| < 2^62, |mm| < 2^62.
//
// The state blocks of the prismatic, tetrahedral and pyramidal volume kernels are held FX_WS bits wider,
// |X| < 2^58: with operators of at most 30 terms, scaled to row sums of at most 1 where a sum ends in limbs
// and of 4 where it ends in FP64, |hh| < 2^62 and |mm| < 2^60 + 30 2^57 < 2^63. Their gradients take a
// scale of 2^5 or 2^6 and then the room of the metric's three terms. (The prisms' line interpolation, row sums
// below 1.6, ends in limbs below 1.6 2^58 and meets row sums of at most 2.)
#pragma once

#include <cstdint>

#define FX_MASK 0x0fffffffu
#define FX_WS 2

// One coefficient or value in two limbs.
struct fx2 { int h, l; };

// c 2^(58 - k) in two limbs (host); |c| 2^-k < 2.
inline fx2 fx_coef(double c, int k)
{
    double s = c;
    for (int i = 0; i < 58 - k; i++) s *= 2.0;   // exact
    const long long C = (long long)(s < 0 ? s - 0.5 : s + 0.5);
    const long long H = (C + (1LL << 27)) >> 28;
    return fx2{(int)H, (int)(C - H * (1LL << 28))};
}

// The smallest scale k for which `largest` 2^-k < 1.9 (a coefficient's limb fits 32 bits) and
// `rowsum` 2^-k <= limit (host).
inline int fx_scale(double largest, double rowsum, double limit)
{
    int k = 0;
    for (double s = 1.0; largest * s >= 1.9 || rowsum * s > limit; s *= 0.5) k++;
    return k;
}

#ifdef __CUDACC__
// A running product-sum.
struct fxacc { long long hh, mm; };

__device__ __forceinline__ void fx_mac(fxacc &s, fx2 c, fx2 x)
{
    long long p, q, r;
    asm("mul.wide.s32 %0, %1, %2;" : "=l"(p) : "r"(c.h), "r"(x.h));
    asm("mul.wide.s32 %0, %1, %2;" : "=l"(q) : "r"(c.h), "r"(x.l));
    asm("mul.wide.s32 %0, %1, %2;" : "=l"(r) : "r"(c.l), "r"(x.h));
    asm("add.s64 %0, %0, %1;" : "+l"(s.hh) : "l"(p));
    asm("add.s64 %0, %0, %1;" : "+l"(s.mm) : "l"(q));
    asm("add.s64 %0, %0, %1;" : "+l"(s.mm) : "l"(r));
}
// The sum in units of 2^(k - 2) X.
__device__ __forceinline__ long long fx_sum(const fxacc &s) { return s.hh + (s.mm >> 28); }
// A sum back to limbs at the scale of the operator's input (times 2^-k): Y / 4, rounded if the
// accumulator started at FX_HALF.
#define FX_HALF 2
__device__ __forceinline__ fx2 fx_limbs(long long y)
{
    return fx2{(int)(y >> 30), (int)((unsigned)(y >> 2) & FX_MASK)};
}

// f x for one factor, at the scale of x (times 2^-k of the factor).
__device__ __forceinline__ fx2 fx_mul(fx2 f, fx2 x)
{
    fxacc s{FX_HALF, 0};
    fx_mac(s, f, x);
    return fx_limbs(fx_sum(s));
}

// Exponent field of the largest magnitude is formed from the high words: abs(hi) of a value.
__device__ __forceinline__ int fx_mag(double v) { return __double2hiint(v) & 0x7fffffff; }

// v of a block with biased exponent E (of its largest magnitude) as X = v 2^(1078 + W - E), |X| < 2^(56 + W).
template <int W = 0>
__device__ __forceinline__ long long fx_int(double v, int E)
{
    const int hi = __double2hiint(v), e = (hi >> 20) & 0x7ff;
    const unsigned mh = e ? ((unsigned)(hi & 0xfffff) | 0x100000u) : 0u;   // subnormal values count as zero
    unsigned long long m = ((unsigned long long)mh << 32) | (e ? (unsigned)__double2loint(v) : 0u);
    m = (m << (3 + W)) >> min(E - e, 63);
    return hi < 0 ? -(long long)m : (long long)m;
}
__device__ __forceinline__ fx2 fx_split(long long x) { return fx2{(int)(x >> 28), (int)((unsigned)x & FX_MASK)}; }
template <int W = 0>
__device__ __forceinline__ fx2 fx_from(double v, int E) { return fx_split(fx_int<W>(v, E)); }

// y 2^e2 rounded to FP64; NaN for a block that held a non-finite value.
__device__ __forceinline__ double fx_double(long long y, int e2, bool bad)
{
    const unsigned long long m = y < 0 ? 0ull - (unsigned long long)y : (unsigned long long)y;
    const int lz = __clzll((long long)m);
    const unsigned long long z = m << (lz & 63);
    int ex = min(max(1085 + e2 - lz, 0), 2046);
    if ((long long)z >= 0) ex = 0;   // y = 0
    const unsigned long long b = ((unsigned long long)(unsigned)ex << 52) + (z >> 11) + ((z >> 10) & 1ull);
    int hi = (int)(b >> 32) | ((int)(y >> 32) & 0x80000000);
    hi = bad ? 0x7ff80000 : hi;
    return __hiloint2double(hi, (int)(unsigned)b);
}

// One warp: the n values at src (n <= 32 KR) to limbs at dst, scaled by their largest magnitude; its
// exponent field goes to *E (by lane 0).
template <int KR>
__device__ __forceinline__ void fx_warp_block(const double *src, int n, fx2 *dst, int *E)
{
    const int lane = threadIdx.x & 31;
    double v[KR];
    int m = 0;
#pragma unroll
    for (int k = 0; k < KR; k++) {
        v[k] = lane + 32 * k < n ? src[lane + 32 * k] : 0.0;
        m = max(m, fx_mag(v[k]));
    }
    const int e = (int)__reduce_max_sync(0xffffffffu, (unsigned)m) >> 20;
    if (lane == 0) *E = e;
#pragma unroll
    for (int k = 0; k < KR; k++)
        if (lane + 32 * k < n) dst[lane + 32 * k] = fx_from(v[k], e);
}

// A CTA of one element: the values v[rd][alpha] of flux points threadIdx.x + rd NT (below NF) to limbs at
// dst[alpha NF + s], each variable scaled by its largest magnitude (exponent fields in E). mx: two sets of
// five words, zero at first, used in turn (par). Two barriers.
template <int NF, int NT, int RD>
__device__ __forceinline__ void fx_stage5(const double (&v)[RD][5], fx2 *dst, int (*mx)[5], int &par, int (&E)[5])
{
#pragma unroll
    for (int a = 0; a < 5; a++) {
        int m = 0;
#pragma unroll
        for (int rd = 0; rd < RD; rd++) m = max(m, fx_mag(v[rd][a]));
        m = (int)__reduce_max_sync(0xffffffffu, (unsigned)m) >> 20;
        if ((threadIdx.x & 31) == 0) atomicMax(&mx[par][a], m);
    }
    __syncthreads();
#pragma unroll
    for (int a = 0; a < 5; a++) E[a] = mx[par][a];
    if (threadIdx.x < 5) mx[par ^ 1][threadIdx.x] = 0;
    par ^= 1;
#pragma unroll
    for (int rd = 0; rd < RD; rd++) {
        const int s = threadIdx.x + rd * NT;
        if (s < NF) {
#pragma unroll
            for (int a = 0; a < 5; a++) dst[a * NF + s] = fx_from(v[rd][a], E[a]);
        }
    }
    __syncthreads();
}

// A run-time factor c (of an element's metric) in limbs for the common exponent E of its block:
// c 2^(1080 - E), below 2^58.
__device__ __forceinline__ fx2 fx_factor(double c, int E)
{
    const long long C = fx_int(c, E) << 2;
    const int H = (int)((C + (1LL << 27)) >> 28);
    return fx2{H, (int)(C - ((long long)H << 28))};
}

// Exponent of the factors J^-1[d][k], d = 0..2, that form component k of a gradient (Ji: [3 d + k]), with the
// room of three terms. Each component has its own: on an element of aspect ratio A the columns differ by A, and
// at the largest one's exponent the gradient along the long direction would lose log2(A) bits.
__device__ __forceinline__ int fx_column_exp(const double *Ji, int k)
{
    return (max(max(fx_mag(Ji[k]), fx_mag(Ji[3 + k])), fx_mag(Ji[6 + k])) >> 20) + 2;
}
// Exponent of field f (5 variables, then the gradients 5 + 3 alpha + d) relative to its variable's.
__device__ __forceinline__ int fx_field_exp(int f, const int (&qe)[3])
{
    const int d = (f - 5) % 3;
    return f < 5 ? 0 : (d == 0 ? qe[0] : (d == 1 ? qe[1] : qe[2]));
}
#endif
