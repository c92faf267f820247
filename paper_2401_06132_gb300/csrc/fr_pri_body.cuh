// fr_pri_body.cuh -- the prismatic (p = 3) phase bodies of the anti-aliased Navier-Stokes FR
// right-hand side (face solution, volume group, interface group; Sec. 4.1 factorisation), as device
// functions over the elements first, first + stride, ... of a launch: fr_pri.cu launches them on
// their own, and fr_hex.cu inside the launches that serve several element groups at once.
#pragma once

#include <cuda_runtime.h>

#include "fr_internal.h"
#include "fr_physics.cuh"
#include "fr_tcgen05.cuh"

namespace pri {
namespace {

constexpr int NT_ = FR_PT, NZ = FR_PE, MZ = 5, NQT = FR_PQ;
constexpr int NU = NT_ * NZ;                  // 40
constexpr int NF = 2 * NT_ + 3 * NZ * NZ;     // 68
constexpr int NQ = NQT * MZ;                  // 125

__device__ __forceinline__ int face_of(int s) { return s < 10 ? 0 : s < 20 ? 1 : 2 + (s - 20) / 16; }

// The FP32 volume kernel's operators in constant memory (one copy per translation unit that includes this
// file, filled by set_const_ops on each device): read with compile-time indices, its entries are
// constant-bank operands of the multiply-adds instead of a shared-memory load per coefficient.
__constant__ PriC32 c_prib32;

inline int set_const_ops(const PriC32 &h)
{
    return cudaMemcpyToSymbol(c_prib32, &h, sizeof(h)) == cudaSuccess ? 0 : -1;
}

template <typename T>
__device__ __forceinline__ void pri_normal(const Geo<T> &g, int f, T *n, T &mag)
{
    const T r2 = T(0.70710678118654752440);
    T nr[3] = {T(0), T(0), T(0)};
    if (f == 0) nr[2] = T(-1);
    else if (f == 1) nr[2] = T(1);
    else if (f == 2) nr[1] = T(-1);
    else if (f == 3) { nr[0] = r2; nr[1] = r2; }
    else nr[0] = T(-1);
    T ns[3];
#pragma unroll
    for (int k = 0; k < 3; k++) ns[k] = g.det * (g.Ji[k] * nr[0] + g.Ji[3 + k] * nr[1] + g.Ji[6 + k] * nr[2]);
    mag = sqrt(ns[0] * ns[0] + ns[1] * ns[1] + ns[2] * ns[2]);
    const T im = T(1) / mag;
#pragma unroll
    for (int k = 0; k < 3; k++) n[k] = ns[k] * im;
}

// Value at flux point s of a field stored at solution points (stride 1, index t + 10 k).
template <typename T>
__device__ __forceinline__ T face_value(const PriOps<T> &op, const T *fld, int s)
{
    T v = T(0);
    if (s < 20) {
        const int t = s % 10;
        const T *l = s < 10 ? op.lzL : op.lzR;
#pragma unroll
        for (int k = 0; k < NZ; k++) v += l[k] * fld[t + 10 * k];
    } else {
        const int f = (s - 20) / 16, loc = (s - 20) % 16, a = loc % 4, b = loc / 4;
#pragma unroll
        for (int t = 0; t < NT_; t++) v += op.Ef[f][a][t] * fld[t + 10 * b];
    }
    return v;
}

// An entry of the float-float table: its hi part and the lo part at the same offset.
__device__ __forceinline__ ff ffop(const PriOpsFF &o, const float &hi)
{
    // the lo part sits at the same offset in the second table
    const float *h = &hi;
    return ff{hi, *(reinterpret_cast<const float *>(&o.lo) + (h - reinterpret_cast<const float *>(&o.hi)))};
}

// Same, of the field minus a constant, with the float-float table (a compensated dot product, Dot2):
// the face value to about 48 bits before its final rounding to FP32.
__device__ __forceinline__ ff face_value_ff_off(const PriOpsFF &o, const float *fld, int s, float off)
{
    float sh, c;
    if (s < 20) {
        const int t = s % 10;
        const float *l = s < 10 ? o.hi.lzL : o.hi.lzR;
        dot2_first(ffop(o, l[0]), fld[t] - off, sh, c);
#pragma unroll
        for (int k = 1; k < NZ; k++) dot2_next(ffop(o, l[k]), fld[t + 10 * k] - off, sh, c);
    } else {
        const int f = (s - 20) / 16, loc = (s - 20) % 16, a = loc % 4, b = loc / 4;
        dot2_first(ffop(o, o.hi.Ef[f][a][0]), fld[10 * b] - off, sh, c);
#pragma unroll
        for (int t = 1; t < NT_; t++) dot2_next(ffop(o, o.hi.Ef[f][a][t]), fld[t + 10 * b] - off, sh, c);
    }
    return fast_two_sum(sh, c);
}

template <typename T, int NTH>
__device__ __forceinline__ void load_ops(const PriOps<T> *g, PriOps<T> &s)
{
    const int n = sizeof(PriOps<T>) / sizeof(T);
    const T *src = reinterpret_cast<const T *>(g);
    T *dst = reinterpret_cast<T *>(&s);
    for (int i = threadIdx.x; i < n; i += NTH) dst[i] = src[i];
}


// Shared-memory operands of the tensor-core contractions (bytes, 128-byte aligned pieces), for the
// split form TCM (1: FP16 in three K segments, 2: BF16 in six; tc::SplitForm).
constexpr int TC_ROWS_I = 20 * MZ, TC_ROWS_P = 15 * MZ;    // 100 and 75 rows of M = 128
constexpr int TC_ST = 11;                                  // row stride of the projected rows
template <int TCM>
struct PriTC {
    static constexpr int KI = tc::split_k<TCM>(NT_), NI = 32;    // interpolation: K = segments x 10 (padded), N = 25 (+7)
    static constexpr int KP = tc::split_k<TCM>(NQT), NP = 16;    // projection: K = segments x 25 (padded), N = 10 (+6)
    static constexpr int SBO_I = KI / 8 * 128, SBO_P = KP / 8 * 128;
    // The A tile holds the rows an element writes (the larger layout of the two); the MMA reads
    // all 128 rows, and the ones past the element's last run on into the buffers that follow the
    // tile (the operator tiles and the kernel's arrays), feeding accumulator lanes never read.
    static constexpr int A_I = (TC_ROWS_I + 7) / 8 * SBO_I, A_P = (TC_ROWS_P + 7) / 8 * SBO_P;
    static constexpr int A_BYTES = ((A_I > A_P ? A_I : A_P) + 127) / 128 * 128;
    static constexpr int BI_BYTES = NI / 8 * SBO_I, BP_BYTES = NP / 8 * SBO_P;
    static constexpr int HEAD = A_BYTES + BI_BYTES + BP_BYTES + 128 * 4 + 16;   // tiles, row shifts, barrier, TMEM slot
    static constexpr int BYTES = HEAD + 128;                                     // + alignment slack
    static constexpr uint32_t IDESC_I = tc::idesc_f16(TCM - 1, 128, NI), IDESC_P = tc::idesc_f16(TCM - 1, 128, NP);
    static_assert(TC_ROWS_I <= 128 && TC_ROWS_P <= 128, "one M = 128 tile per element");
    static_assert(16 * SBO_I <= HEAD + (5 * NU + 15 * NU + 5 * NF + 20 * NQ) * 4 &&
                      16 * SBO_P <= HEAD + (5 * NU + 15 * NU + 5 * NF + 20 * NQ) * 4,
                  "the 128 rows an MMA reads stay inside the CTA's shared memory");
};

// -------------------------------------------------------------------------------------------------
// Phase A: disu
// -------------------------------------------------------------------------------------------------
// The reduced precisions evaluate the face values with the float-float operator table (compensated:
// exact products, TwoSum accumulation) and round once: the quad-face rows of the triangle
// interpolation extrapolate from interior points (row sums of |Ef| well above 1), and at low Mach
// the Rusanov dissipation (1/2)(|v.n| + c)(u_L - u_R), with c about 10 |v|, lifts any rounding of a
// face value into R. Low-Mach form (ph.dev): the face solution of the deviations from the reference
// state, and the own-normal mass flux n.(rho v) at every flux point in float-float.
__device__ __forceinline__ void pri_disu_body(const HexArgs<float> &a, const PriOpsFF *opsff, long long first, long long stride)
{
    using T = float;
    __shared__ __align__(16) unsigned char raw[sizeof(PriOpsFF)];
    {
        const float *src = reinterpret_cast<const float *>(opsff);
        float *dst = reinterpret_cast<float *>(raw);
        for (int i = threadIdx.x; i < (int)(sizeof(PriOpsFF) / sizeof(float)); i += 256) dst[i] = src[i];
    }
    __syncthreads();
    fr_grid_wait();
    const long long total = a.ne * NF;
    for (long long it = first * (long long)blockDim.x + threadIdx.x; it < total; it += (long long)stride * blockDim.x) {
        // one thread per (element, flux point), all five variables
        const int s = (int)(it % NF);
        const long long e = it / NF;
#ifdef FR_DEBUG_BOUNDS
        {
            const long long u0 = elem_u0(a, e, NU), f0 = elem_f0(a, e, NF);
            if (u0 < 0 || u0 + (long long)FR_NV * NU > a.nU || f0 < 0 || f0 + NF > a.nfpt) {
                atomicOr(a.status, 4);
                continue;
            }
        }
#endif
        const T *u = a.U + elem_u0(a, e, NU);
        const long long fo = elem_f0(a, e, NF) + s;
        {
            const PriOpsFF &o = *reinterpret_cast<const PriOpsFF *>(raw);
            const Phys<T> ph = elem_phys(a, e);
            const bool dev = ph.dev != 0;
            ff v[FR_NV];
#pragma unroll
            for (int alpha = 0; alpha < FR_NV; alpha++) {
                const float off = dev ? (alpha == 0 ? ph.rref : (alpha == 4 ? ph.eref : 0.0f)) : 0.0f;
                v[alpha] = face_value_ff_off(o, u + alpha * NU, s, off);
                a.UF[alpha * a.nfpt + fo] = v[alpha].hi + v[alpha].lo;
            }
            if (dev) {
                const ff *nt = a.fnrm64 + (e * 6 + face_of(s)) * 4;
                ff mf = ff_of(0.0f);
#pragma unroll
                for (int k = 0; k < 3; k++)
                    if (nt[k].hi != 0.0f) mf = ff_fma(nt[k], v[1 + k], mf);
                a.MF[fo] = mf;
            }
        }
    }
    fr_grid_done();
}


// The same in FP64, with the traces in block fixed point (fr_fx.cuh): EB elements per CTA of 256 threads
// (18^3 mixed box, face phase 77 -> 38 us).
__device__ __forceinline__ void pri_disu_fx_body(const HexArgs<double> &a, const PriOps<double> *gops, long long first, long long stride)
{
    constexpr int EB = 3, NTH = 256;   // 204 flux points
    __shared__ fx2 s_u[EB * FR_NV * NU], s_ef[3][NZ][NT_], s_lz[2][NZ];
    __shared__ int s_E[EB * FR_NV];
    const PriFxS &op = reinterpret_cast<const PriFx *>(gops + 1)->s;
    for (int i = threadIdx.x; i < 3 * NZ * NT_; i += NTH) (&s_ef[0][0][0])[i] = (&op.Ef[0][0][0])[i];
    for (int i = threadIdx.x; i < 2 * NZ; i += NTH) s_lz[i / NZ][i % NZ] = i < NZ ? op.lzL[i] : op.lzR[i - NZ];
    const int kF = op.kF;
    __syncthreads();
    fr_grid_wait();
    for (long long e0 = first * EB; e0 < a.ne; e0 += stride * EB) {
        const int nb = (int)(a.ne - e0 < EB ? a.ne - e0 : EB);
        {
            bool blk_ok = true;
            for (int k = 0; k < nb; k++) blk_ok = blk_ok && fr_elem_ok(a, e0 + k, NU, NF);
            if (!blk_ok) continue;
        }
        for (int b = threadIdx.x / 32; b < nb * FR_NV; b += NTH / 32)   // one variable of one element per warp
            fx_warp_block<(NU + 31) / 32>(a.U + elem_u0(a, e0 + b / FR_NV, NU) + (b % FR_NV) * NU, NU, s_u + b * NU, s_E + b);
        __syncthreads();
        for (int it = threadIdx.x; it < nb * NF; it += NTH) {
            const int el = it / NF, s = it % NF;
            double *o = a.UF + elem_f0(a, e0 + el, NF) + s;
            const int f = (s - 20) / 16, loc = (s - 20) % 16;
            const fx2 *l = s < 20 ? s_lz[s / 10] : s_ef[f][loc % 4];
            const fx2 *u = s_u + el * FR_NV * NU + (s < 20 ? s % 10 : 10 * (loc / 4));
            const int n = s < 20 ? NZ : NT_, str = s < 20 ? 10 : 1;
            fxacc t[FR_NV] = {{0, 0}, {0, 0}, {0, 0}, {0, 0}, {0, 0}};
#pragma unroll 2
            for (int j = 0; j < n; j++) {
                const fx2 c = l[j];
#pragma unroll
                for (int alpha = 0; alpha < FR_NV; alpha++) fx_mac(t[alpha], c, u[alpha * NU + j * str]);
            }
#pragma unroll
            for (int alpha = 0; alpha < FR_NV; alpha++, o += a.nfpt) {
                const int E = s_E[el * FR_NV + alpha];
                *o = fx_double(fx_sum(t[alpha]), E - 1080 + kF, E >= 2047);
            }
        }
        __syncthreads();
    }
    fr_grid_done();
}

// -------------------------------------------------------------------------------------------------
// Phase B: volume group
// -------------------------------------------------------------------------------------------------
template <typename T, int NTH, int TCM>
__device__ __forceinline__ void pri_B_body(const HexArgs<T> &a, const PriOps<T> *gops, const PriOpsFF *opsff, long long first, long long stride)
{
    static_assert(TCM != 0 && NTH == 128 && sizeof(T) == 4, "tensor-core form: FP32, one warpgroup per element");
    using PT = PriTC<TCM>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ ff s_mf[sizeof(T) == 4 ? 3 * NU : 1];   // low-Mach form: transformed mass flux
    __shared__ short s_plist[NF];                         // flux points that need the viscous flux
    __shared__ int s_pcnt;
    PriOps<T> &op = *reinterpret_cast<PriOps<T> *>(smem_raw);
    unsigned char *arr = smem_raw + ((sizeof(PriOps<T>) + 15) / 16) * 16;
    // tensor-core state (TCM != 0): the tiles come first, so that the MMA's rows past an element's
    // last run on into the arrays below
    unsigned char *tA = nullptr, *tBi = nullptr, *tBp = nullptr;
    int *s_sh = nullptr;
    uint64_t *mbar = nullptr;
    uint32_t *s_tmem = nullptr, tmem = 0, parity = 0;
    bool tc_fail = false, first_wait = true;
    if constexpr (TCM != 0) {
        const uint32_t raw = tc::smem_u32(arr);
        tA = arr + ((128 - (raw & 127)) & 127);
        tBi = tA + PT::A_BYTES;
        tBp = tBi + PT::BI_BYTES;
        s_sh = reinterpret_cast<int *>(tBp + PT::BP_BYTES);
        mbar = reinterpret_cast<uint64_t *>(s_sh + 128);
        s_tmem = reinterpret_cast<uint32_t *>(mbar + 1);
        arr = tA + PT::HEAD;
    }
    T *s_u = reinterpret_cast<T *>(arr);
    T *s_q = s_u + 5 * NU;
    T *s_c = s_q + 15 * NU;
    T *s_w = s_c + 5 * NF;
    T *s_t = s_w + 20 * NQ;
    load_ops<T, NTH>(gops, op);
    if constexpr (TCM != 0) {
        tc::setup(mbar, s_tmem, 32);
        __syncthreads();   // operators in shared memory
        // operator tiles in the split form's segments (FP16: [B_hi | B_hi | B_lo])
        using SF = tc::SplitForm<TCM>;
        for (int i = threadIdx.x; i < PT::NI * PT::KI; i += NTH) {
            const int n = i / PT::KI, k = i % PT::KI, sg = k / NT_;
            uint16_t pp[3] = {0, 0, 0};
            if (n < NQT && sg < SF::SEGS) tc::split_parts<TCM>((float)op.Bt[n][k % NT_], pp);
            *reinterpret_cast<uint16_t *>(tBi + tc::core_offset(n, k, PT::SBO_I)) = sg < SF::SEGS ? pp[SF::y_part(sg)] : (uint16_t)0;
        }
        for (int i = threadIdx.x; i < PT::NP * PT::KP; i += NTH) {
            const int n = i / PT::KP, k = i % PT::KP, sg = k / NQT;
            uint16_t pp[3] = {0, 0, 0};
            if (n < NT_ && sg < SF::SEGS) tc::split_parts<TCM>((float)op.Pt[n][k % NQT], pp);
            *reinterpret_cast<uint16_t *>(tBp + tc::core_offset(n, k, PT::SBO_P)) = sg < SF::SEGS ? pp[SF::y_part(sg)] : (uint16_t)0;
        }
        tc::fence_async_smem();
        tc::fence_before_sync();
        __syncthreads();
        tc::fence_after_sync();
        tmem = *s_tmem;
    }
    for (long long e = first; e < a.ne; e += stride) {
        if (!fr_elem_ok(a, e, NU, NF)) continue;
        const Geo<T> g = a.geo[e];
        const Phys<T> ph = elem_phys(a, e);
        const T *U = a.U + elem_u0(a, e, NU);
        const long long gf0 = elem_f0(a, e, NF);
        bool dev = false;
        if constexpr (sizeof(T) == 4) dev = ph.dev != 0;
        for (int it = threadIdx.x; it < 5 * NU; it += NTH) {
            T v = U[it];
            if (dev) v -= it < NU ? ph.rref : (it >= 4 * NU ? ph.eref : T(0));
            s_u[it] = v;
        }
        if (threadIdx.x == 0) s_pcnt = 0;
        for (int it = threadIdx.x; it < 5 * NF; it += NTH) {   // con_u
            const int alpha = it / NF, s = it % NF;
            const uint32_t pc = a.partner[gf0 + s];
            const bool isL = (pc & FR_LFLAG) != 0;
            const long long pg = fr_partner(a, pc, gf0 + s);
            const T own = a.UF[alpha * a.nfpt + gf0 + s], oth = a.UF[alpha * a.nfpt + pg];
            const T uL = isL ? own : oth, uR = isL ? oth : own;
            s_c[it] = (T(0.5) - ph.beta) * uL + (T(0.5) + ph.beta) * uR;
        }
        __syncthreads();
        // low-Mach form: volume part of R~_rho in float-float (rho v lies in the solution space, so
        // its projection is itself and the corrected divergence applies at the solution points).
        // The tensor-core forms run it while the projection's MMA chain is in flight.
        auto mass_channel = [&]() {
            if constexpr (sizeof(T) == 4) {
                if (dev) {
                    const ff *cm = a.geo64[e].cm;   // det J J^-1, per element
                    for (int z = threadIdx.x; z < NU; z += NTH) {
                        const float m0 = s_u[NU + z], m1 = s_u[2 * NU + z], m2 = s_u[3 * NU + z];
#pragma unroll
                        for (int d = 0; d < 3; d++)
                            s_mf[d * NU + z] = ff_add(ff_add(ff_mul_f(cm[3 * d], m0), ff_mul_f(cm[3 * d + 1], m1)), ff_mul_f(cm[3 * d + 2], m2));
                    }
                    __syncthreads();
                    const PriOpsFF &o = *opsff;
                    const long long pbase = elem_u0(a, e, NU) / FR_NV;
                    for (int z = threadIdx.x; z < NU; z += NTH) {
                        const int k = z / NT_, t = z % NT_;
                        float sh = 0.0f, c = 0.0f;   // compensated dot product (Dot2)
#pragma unroll
                        for (int j = 0; j < NT_; j++) {
                            dot2ff_next(ffop(o, o.hi.Dhx[t][j]), s_mf[j + 10 * k], sh, c);
                            dot2ff_next(ffop(o, o.hi.Dhy[t][j]), s_mf[NU + j + 10 * k], sh, c);
                        }
#pragma unroll
                        for (int j = 0; j < NZ; j++) dot2ff_next(ffop(o, o.hi.Dhz[k][j]), s_mf[2 * NU + t + 10 * j], sh, c);
                        a.RL[pbase + z] = two_sum(sh, c);
                    }
                }
            }
        };
        // corrected gradient: z lines (alpha, t) and triangle planes (alpha, k, t)
        for (int it = threadIdx.x; it < 5 * NT_; it += NTH) {
            const int alpha = it / NT_, t = it % NT_;
            T u[NZ];
#pragma unroll
            for (int k = 0; k < NZ; k++) u[k] = s_u[alpha * NU + t + 10 * k];
            const T cB = s_c[alpha * NF + t], cT = s_c[alpha * NF + 10 + t];
#pragma unroll
            for (int k = 0; k < NZ; k++) {
                T v = op.liftzR[k] * cT - op.liftzL[k] * cB;
#pragma unroll
                for (int j = 0; j < NZ; j++) v += op.Dhz[k][j] * u[j];
                s_q[(alpha * 3 + 2) * NU + t + 10 * k] = v;
            }
        }
        for (int it = threadIdx.x; it < 5 * NU; it += NTH) {
            const int alpha = it / NU, r = it % NU, k = r / NT_, t = r % NT_;
            const T *u = s_u + alpha * NU + 10 * k;
            T vx = T(0), vy = T(0);
#pragma unroll
            for (int j = 0; j < NT_; j++) { vx += op.Dhx[t][j] * u[j]; vy += op.Dhy[t][j] * u[j]; }
#pragma unroll
            for (int f = 0; f < 3; f++) {
                T l = T(0);
#pragma unroll
                for (int b = 0; b < NZ; b++) l += op.Lf[f][t][b] * s_c[alpha * NF + 20 + 16 * f + b + 4 * k];
                vx += op.nf[f][0] * l;
                vy += op.nf[f][1] * l;
            }
            s_q[(alpha * 3 + 0) * NU + t + 10 * k] = vx;
            s_q[(alpha * 3 + 1) * NU + t + 10 * k] = vy;
        }
        __syncthreads();
        for (int it = threadIdx.x; it < 5 * NU; it += NTH) {   // gradcoru
            const int alpha = it / NU, z = it % NU;
            T *q = s_q + alpha * 3 * NU + z;
            const T q0 = q[0], q1 = q[NU], q2 = q[2 * NU];
#pragma unroll
            for (int k = 0; k < 3; k++) q[k * NU] = g.Ji[k] * q0 + g.Ji[3 + k] * q1 + g.Ji[6 + k] * q2;
        }
        __syncthreads();
        // viscous normal flux at own flux points, on the side whose LDG weight 1/2 +- beta is not
        // zero (the other side's is never used); the points are compacted so whole warps work
        // (the tensor-core forms run it while the interpolation's MMA chain is in flight)
        auto viscous_faces = [&]() {
            for (int s = threadIdx.x; s < NF; s += NTH) {
                const bool isL = (a.partner[gf0 + s] & FR_LFLAG) != 0;
                const T wgt = isL ? T(0.5) + ph.beta : T(0.5) - ph.beta;
                if (wgt == T(0)) {
#pragma unroll
                    for (int k = 0; k < 4; k++) a.FV[k * a.nfpt + gf0 + s] = T(0);
                } else {
                    s_plist[atomicAdd(&s_pcnt, 1)] = (short)s;
                }
            }
            __syncthreads();
            const int nplist = s_pcnt;
            for (int li = threadIdx.x; li < nplist; li += NTH) {
                const int s = s_plist[li];
                T uf[5], qf[5][3];
#pragma unroll
                for (int alpha = 0; alpha < 5; alpha++) {
                    uf[alpha] = face_value(op, s_u + alpha * NU, s);
#pragma unroll
                    for (int d = 0; d < 3; d++) qf[alpha][d] = face_value(op, s_q + (alpha * 3 + d) * NU, s);
                }
                const T *nt = a.fnrm + (e * 6 + face_of(s)) * 4;
                T n[3] = {nt[0], nt[1], nt[2]};
                if (dev) { uf[0] += ph.rref; uf[4] += ph.eref; }
                T fvn[4];
                viscous_normal_flux(ph, uf, qf, n, fvn);
#pragma unroll
                for (int k = 0; k < 4; k++) a.FV[k * a.nfpt + gf0 + s] = fvn[k];
            }
        };
        {
            // z first (CUDA cores): row r = 5 f + c holds field f (s_q follows s_u) at z level c on
            // the 10 triangle points; then the triangle interpolation of all 100 rows on the tensor core.
            const int r = threadIdx.x;
            if (r < TC_ROWS_I) {
                const int f = r / MZ, c = r % MZ;
                const T *src = s_u + f * NU;
                float x[NT_], mx = 0.f;
#pragma unroll
                for (int t = 0; t < NT_; t++) {
                    float v = 0.f;
#pragma unroll
                    for (int k = 0; k < NZ; k++) v += (float)op.Bz[c][k] * (float)src[t + 10 * k];
                    x[t] = v;
                    mx = fmaxf(mx, fabsf(v));
                }
                const int sh = tc::row_shift(mx);
                const float sc = tc::pow2f(sh);
#pragma unroll
                for (int t = 0; t < NT_; t++) x[t] *= sc;
                tc::store_split_parts<TCM, PT::KI, NT_>(tA, r, x);
                s_sh[r] = sh;
            }
            tc::mma_issue<PT::KI / 16>(tmem, tA, PT::SBO_I, tBi, PT::SBO_I, PT::IDESC_I, mbar);
            viscous_faces();   // CUDA-core work while the chain runs (touches no operand tile)
            if (!tc::mma_wait(mbar, parity, tc::first_limit(first_wait, a.dbg_wait0))) {
                tc_fail = true;
                break;
            }
            {
                float v0[16], v1[16];
                const uint32_t ta = tmem + ((uint32_t)(32 * (threadIdx.x >> 5)) << 16);
                tc::ld16(ta, v0);
                tc::ld16(ta + 16, v1);
                if (r < TC_ROWS_I) {
                    const float isc = tc::pow2f(-s_sh[r]);
                    T *dst = s_w + NQT * r;                    // field f, level c: f NQ + 25 c = 25 r
#pragma unroll
                    for (int q = 0; q < 16; q++) dst[q] = (T)(v0[q] * isc);
#pragma unroll
                    for (int q = 16; q < NQT; q++) dst[q] = (T)(v1[q - 16] * isc);
                }
            }
            __syncthreads();
        }
        bool ok = true;
        for (int q = threadIdx.x; q < NQ; q += NTH) {          // tdisf
            T u[5], gq[5][3], f[3][5];
#pragma unroll
            for (int alpha = 0; alpha < 5; alpha++) {
                u[alpha] = s_w[alpha * NQ + q];
#pragma unroll
                for (int d = 0; d < 3; d++) gq[alpha][d] = s_w[(5 + alpha * 3 + d) * NQ + q];
            }
            if constexpr (sizeof(T) == 4) {
                if (dev) ok &= total_flux_dev(ph, u, gq, f);
                else ok &= total_flux(ph, u, gq, f);
            } else {
                ok &= total_flux(ph, u, gq, f);
            }
#pragma unroll
            for (int alpha = 0; alpha < 5; alpha++)
#pragma unroll
                for (int d = 0; d < 3; d++)
                    s_w[(alpha * 3 + d) * NQ + q] = g.det * (g.Ji[3 * d] * f[0][alpha] + g.Ji[3 * d + 1] * f[1][alpha] + g.Ji[3 * d + 2] * f[2][alpha]);
        }
        flag_status(a.status, ok);
        __syncthreads();
        {
            // triangle projection of the 75 rows (flux component f, quadrature level c) on the tensor
            // core, then z (CUDA cores)
            const int r = threadIdx.x;
            if (r < TC_ROWS_P) {
                const T *src = s_w + NQT * r;
                float x[NQT], mx = 0.f;
#pragma unroll
                for (int q = 0; q < NQT; q++) { x[q] = (float)src[q]; mx = fmaxf(mx, fabsf(x[q])); }
                const int sh = tc::row_shift(mx);
                const float sc = tc::pow2f(sh);
#pragma unroll
                for (int q = 0; q < NQT; q++) x[q] *= sc;
                tc::store_split_parts<TCM, PT::KP, NQT>(tA, r, x);
                s_sh[r] = sh;
            }
            tc::mma_issue<PT::KP / 16>(tmem, tA, PT::SBO_P, tBp, PT::SBO_P, PT::IDESC_P, mbar);
            // CUDA-core work while the chain runs: it reads the state and writes only static shared
            // memory and global memory, which the chain's rows (they run on past the operand tile
            // into the dynamic shared arrays) never reach
            mass_channel();
            if (!tc::mma_wait(mbar, parity, tc::first_limit(first_wait, a.dbg_wait0))) {
                tc_fail = true;
                break;
            }
            {
                float v0[16];
                tc::ld16(tmem + ((uint32_t)(32 * (threadIdx.x >> 5)) << 16), v0);
                if (r < TC_ROWS_P) {
                    const float isc = tc::pow2f(-s_sh[r]);
#pragma unroll
                    for (int t = 0; t < NT_; t++) s_t[TC_ST * r + t] = (T)(v0[t] * isc);
                }
            }
            __syncthreads();
            for (int it = threadIdx.x; it < 15 * NU; it += NTH) {
                const int f = it / NU, rr = it % NU, k = rr / NT_, t = rr % NT_;
                T v = T(0);
#pragma unroll
                for (int c = 0; c < MZ; c++) v += op.Pz[k][c] * s_t[TC_ST * (MZ * f + c) + t];
                s_q[f * NU + t + 10 * k] = v;
            }
            __syncthreads();
        }
        T *R = a.R + elem_u0(a, e, NU);
        for (int it = threadIdx.x; it < 5 * NU; it += NTH) {   // corrected divergence
            const int alpha = it / NU, r = it % NU, k = r / NT_, t = r % NT_;
            const T *F = s_q + alpha * 3 * NU;
            T v = T(0);
#pragma unroll
            for (int j = 0; j < NT_; j++) v += op.Dhx[t][j] * F[j + 10 * k] + op.Dhy[t][j] * F[NU + j + 10 * k];
#pragma unroll
            for (int j = 0; j < NZ; j++) v += op.Dhz[k][j] * F[2 * NU + t + 10 * j];
            R[it] = v;
        }
        __syncthreads();
    }
    if constexpr (TCM != 0) {
        // a chain that did not complete within the bound is reported; the tensor memory is released
        if (tc_fail && threadIdx.x == 0) atomicOr(a.status, 2);
        tc::teardown(mbar, parity, tc_fail, tmem, 32);
    }
}


constexpr int P32_TS = 12, P32_WS = 28;   // padded triangle rows: whole 16-byte vectors
static_assert(sizeof(PriOpsFF) % 16 == 0, "PriS32 follows at a 16-byte boundary");
constexpr size_t P32_SMEM = sizeof(float) * (20 * NU + 5 * NF + 20 * MZ * P32_TS + 20 * NF);
static_assert(20 * MZ * P32_TS + 20 * NF >= 15 * MZ * P32_WS && 20 * NU + 5 * NF >= 15 * MZ * NT_ && (20 * NU + 5 * NF) % 4 == 0,
              "staging fits over consumed buffers, in 16-byte rows");

// -------------------------------------------------------------------------------------------------
// Phase B in FP32 on the CUDA cores, one element per CTA
// -------------------------------------------------------------------------------------------------
// A line, a triangle plane or a quadrature point per thread wherever it can be held in registers, with
// the operators as constant-bank operands: the gradient's planes and lines on their own warps, the line
// interpolation first so that a thread interpolates its own quadrature point's 20 fields in the triangle
// plane and keeps them in registers through the flux, the corrected derivatives on the projection
// (Dhx Pt, Dhy Pt, Dhz Pz), one warp per component direction, with the mass channel beside them. With a
// pass per operator the kernel issued 11,000 warp instructions per element behind 18 barriers; now 7,900
// behind 9. Measured, 24^3 mixed box (13,824 prisms): 202 -> 148 us per launch.
template <int NTH>
__device__ __forceinline__ void pri_B32_body(const HexArgs<float> &a, const PriOpsFF *opsff, long long first, long long stride)
{
    static_assert(NTH == 128 && NU + NF <= NTH, "four warps; one thread per quadrature point, state and flux point");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float *s_u = reinterpret_cast<float *>(smem_raw);        // state, then the physical gradient (5 + 3 alpha + d)
    float *s_c = s_u + 20 * NU;                              // common solution
    float *s_t = s_c + 5 * NF;                               // [20][c][12] line-interpolated fields
    float *s_tr = s_t + 20 * MZ * P32_TS;                    // [listed flux point][20] traces
    float *s_w = s_t;                                        // [15][c][28] transformed flux
    float *s_p = s_u;                                        // [15][c][t] projected in the triangle plane
    __shared__ ff s_mf[3 * NU];                              // low-Mach form: transformed mass flux
    // plane operators and traces, read by loops over their outputs or rows selected at run time
    // (unrolled with constant operands, the planes missed in the instruction cache)
    __shared__ __align__(16) PriS32 so;
    __shared__ short s_plist[NF];
    __shared__ int s_pcnt;
    const PriC32 &op = c_prib32;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    {
        const float4 *src = reinterpret_cast<const float4 *>(opsff + 1);
        float4 *dst = reinterpret_cast<float4 *>(&so);
        for (int i = tid; i < (int)(sizeof(PriS32) / 16); i += NTH) dst[i] = src[i];
    }
    float bt[NT_];   // this thread's row of the triangle interpolation
    const int tq = tid % NQT, tc_ = tid / NQT;
#pragma unroll
    for (int t = 0; t < NT_; t++) bt[t] = opsff->hi.Bt[tq][t];
    if (tid == 0) s_pcnt = 0;
    __syncthreads();
    fr_grid_wait();
    for (long long e = first; e < a.ne; e += stride) {
        if (!fr_elem_ok(a, e, NU, NF)) continue;
        const Geo<float> g = a.geo[e];
        const Phys<float> ph = elem_phys(a, e);
        const bool dev = ph.dev != 0;
        const int a0 = dev ? 1 : 0;   // low-Mach form: the mass has no flux on this path
        const long long u0 = elem_u0(a, e, NU), gf0 = elem_f0(a, e, NF);
        // 1. state (deviations in the low-Mach form; with the transformed mass flux) and common solution, one
        //    point and five variables per thread, and the flux points whose side carries LDG weight
        if (tid < NU) {
            const float *U = a.U + u0 + tid;
            const float m0 = U[NU], m1 = U[2 * NU], m2 = U[3 * NU];
            s_u[tid] = U[0] - (dev ? ph.rref : 0.f);
            s_u[NU + tid] = m0; s_u[2 * NU + tid] = m1; s_u[3 * NU + tid] = m2;
            s_u[4 * NU + tid] = U[4 * NU] - (dev ? ph.eref : 0.f);
            if (dev) {
                const ff *cm = a.geo64[e].cm;   // det J J^-1
#pragma unroll
                for (int d = 0; d < 3; d++)
                    s_mf[d * NU + tid] = ff_add(ff_add(ff_mul_f(cm[3 * d], m0), ff_mul_f(cm[3 * d + 1], m1)), ff_mul_f(cm[3 * d + 2], m2));
            }
        } else if (tid < NU + NF) {
            const int s = tid - NU;
            const long long og = gf0 + s;
            const uint32_t pc = a.partner[og];
            const bool isL = (pc & FR_LFLAG) != 0;
            const long long pg = fr_partner(a, pc, og);
            const float *uL = a.UF + (isL ? og : pg), *uR = a.UF + (isL ? pg : og);
            const float wl = 0.5f - ph.beta, wr = 0.5f + ph.beta;
#pragma unroll
            for (int alpha = 0; alpha < 5; alpha++, uL += a.nfpt, uR += a.nfpt) s_c[alpha * NF + s] = wl * *uL + wr * *uR;
            if ((isL ? wr : wl) == 0.f) {
                float *fv = a.FV + og;
#pragma unroll
                for (int k = 0; k < 4; k++, fv += a.nfpt) *fv = 0.f;
            } else {
                s_plist[atomicAdd(&s_pcnt, 1)] = (short)s;
            }
        }
        __syncthreads();
        const int nplist = s_pcnt;
        // 2. corrected gradient: x and y of the triangle planes (alpha, k) on warps 0 and 1, z lines
        //    (alpha, t) on warps 2 and 3
        if (warp < 2) {
            if (lane < 5 * NZ) {
                const int alpha = lane / NZ, k = lane % NZ;
                const float *x = s_u + alpha * NU + 10 * k, *c = s_c + alpha * NF + 20 + 4 * k;
                float u[NT_], cf[12];
#pragma unroll
                for (int t = 0; t < NT_; t++) u[t] = x[t];
#pragma unroll
                for (int b = 0; b < 12; b++) cf[b] = c[16 * (b / 4) + b % 4];
                float *q = s_u + (5 + alpha * 3 + warp) * NU + 10 * k;
#pragma unroll 1
                for (int t = 0; t < NT_; t++) {
                    float L[24];
#pragma unroll
                    for (int i = 0; i < 6; i++) {
                        const float4 y = *reinterpret_cast<const float4 *>(&so.dl[warp][t][4 * i]);
                        L[4 * i] = y.x; L[4 * i + 1] = y.y; L[4 * i + 2] = y.z; L[4 * i + 3] = y.w;
                    }
                    float v = 0.f;
#pragma unroll
                    for (int j = 0; j < NT_; j++) v += L[j] * u[j];
#pragma unroll
                    for (int b = 0; b < 12; b++) v += L[NT_ + b] * cf[b];
                    q[t] = v;
                }
            }
        } else {
            const int l = tid - 64;
            if (l < 5 * NT_) {
                const int alpha = l / NT_, t = l % NT_;
                float u[NZ];
#pragma unroll
                for (int k = 0; k < NZ; k++) u[k] = s_u[alpha * NU + t + 10 * k];
                const float cB = s_c[alpha * NF + t], cT = s_c[alpha * NF + 10 + t];
#pragma unroll
                for (int k = 0; k < NZ; k++) {
                    float v = op.liftzR[k] * cT - op.liftzL[k] * cB;
#pragma unroll
                    for (int j = 0; j < NZ; j++) v += op.Dhz[k][j] * u[j];
                    s_u[(5 + alpha * 3 + 2) * NU + t + 10 * k] = v;
                }
            }
        }
        __syncthreads();
        for (int it = tid; it < 5 * NU; it += NTH) {   // q = J^-T q~
            float *q = s_u + (5 + it / NU * 3) * NU + it % NU;
            const float q0 = q[0], q1 = q[NU], q2 = q[2 * NU];
#pragma unroll
            for (int k = 0; k < 3; k++) q[k * NU] = g.Ji[k] * q0 + g.Ji[3 + k] * q1 + g.Ji[6 + k] * q2;
        }
        __syncthreads();
        // 3. traces of the 20 fields at the listed flux points, four threads per point; z lines of the
        //    interpolation
        for (int it = tid; it < 4 * nplist; it += NTH) {
            const int li = it >> 2, fg = it & 3, s = s_plist[li];
            const float *x = s_u + 5 * fg * NU;
            float v[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
            if (s < 20) {
                const float *l = so.lz[s / 10];
                x += s % 10;
#pragma unroll
                for (int k = 0; k < NZ; k++)
#pragma unroll
                    for (int i = 0; i < 5; i++) v[i] += l[k] * x[i * NU + 10 * k];
            } else {
                const int f = (s - 20) / 16, loc = (s - 20) % 16;
                const float *l = so.ef[f][loc % 4];
                x += 10 * (loc / 4);
#pragma unroll
                for (int j = 0; j < NT_; j++)
#pragma unroll
                    for (int i = 0; i < 5; i++) v[i] += l[j] * x[i * NU + j];
            }
#pragma unroll
            for (int i = 0; i < 5; i++) s_tr[li * 20 + 5 * fg + i] = v[i];
        }
        for (int it = tid; it < 20 * NT_; it += NTH) {
            const int f = it / NT_, t = it % NT_;
            float u[NZ];
#pragma unroll
            for (int k = 0; k < NZ; k++) u[k] = s_u[f * NU + t + 10 * k];
#pragma unroll
            for (int c = 0; c < MZ; c++) {
                float v = 0.f;
#pragma unroll
                for (int k = 0; k < NZ; k++) v += op.Bz[c][k] * u[k];
                s_t[(f * MZ + c) * P32_TS + t] = v;
            }
        }
        __syncthreads();
        // 4. own-normal viscous flux at the listed flux points (from the upper warps down)
        for (int li = NTH - 1 - tid; li < nplist; li += NTH) {
            const int s = s_plist[li];
            const float *v = s_tr + li * 20;
            float uf[5], qf[5][3];
#pragma unroll
            for (int alpha = 0; alpha < 5; alpha++) {
                uf[alpha] = v[alpha];
#pragma unroll
                for (int d = 0; d < 3; d++) qf[alpha][d] = v[5 + alpha * 3 + d];
            }
            const float *nt = a.fnrm + (e * 6 + face_of(s)) * 4;
            const float n[3] = {nt[0], nt[1], nt[2]};
            if (dev) { uf[0] += ph.rref; uf[4] += ph.eref; }
            float fvn[4];
            viscous_normal_flux(ph, uf, qf, n, fvn);
            float *fv = a.FV + gf0 + s;
#pragma unroll
            for (int k = 0; k < 4; k++, fv += a.nfpt) *fv = fvn[k];
        }
        // 5. this thread's quadrature point: triangle-plane interpolation, flux and its transformation
        bool ok = true;
        float f[3][5];
        if (tid < NQ) {
            float u[5], gq[5][3];
#pragma unroll
            for (int i = 0; i < 20; i++) {
                const float *x = s_t + (i * MZ + tc_) * P32_TS;
                const float4 x0 = *reinterpret_cast<const float4 *>(x), x1 = *reinterpret_cast<const float4 *>(x + 4);
                const float2 x2 = *reinterpret_cast<const float2 *>(x + 8);
                float v = bt[0] * x0.x;
                v += bt[1] * x0.y; v += bt[2] * x0.z; v += bt[3] * x0.w;
                v += bt[4] * x1.x; v += bt[5] * x1.y; v += bt[6] * x1.z; v += bt[7] * x1.w;
                v += bt[8] * x2.x; v += bt[9] * x2.y;
                if (i < 5) u[i] = v;
                else gq[(i - 5) / 3][(i - 5) % 3] = v;
            }
            if (dev) ok = total_flux_dev(ph, u, gq, f);
            else ok = total_flux(ph, u, gq, f);
        }
        flag_status(a.status, ok);
        __syncthreads();   // the interpolated fields and the traces are read
        if (tid < NQ) {
#pragma unroll
            for (int alpha = 0; alpha < 5; alpha++)
                if (alpha >= a0) {
#pragma unroll
                    for (int d = 0; d < 3; d++)
                        s_w[(alpha * 3 + d) * MZ * P32_WS + tc_ * P32_WS + tq] =
                            g.det * (g.Ji[3 * d] * f[0][alpha] + g.Ji[3 * d + 1] * f[1][alpha] + g.Ji[3 * d + 2] * f[2][alpha]);
                }
        }
        __syncthreads();
        // 6. projection with the corrected divergence in the triangle planes (alpha, c), one direction per
        //    warp; the fourth warp forms the low-Mach form's volume part of R~_rho in float-float (rho v lies
        //    in the solution space, so its projection is itself)
        if (warp < 3) {
            const int alpha = a0 + lane / MZ, c = lane % MZ;
            if (alpha < 5 && lane < 25) {
                const float *x = s_w + (alpha * 3 + warp) * MZ * P32_WS + c * P32_WS;
                float *p = s_p + (alpha * 3 + warp) * MZ * NT_ + c * NT_;
                float w[NQT];
                w[24] = x[24];
#pragma unroll
                for (int i = 0; i < 6; i++) {
                    const float4 y = *reinterpret_cast<const float4 *>(x + 4 * i);
                    w[4 * i] = y.x; w[4 * i + 1] = y.y; w[4 * i + 2] = y.z; w[4 * i + 3] = y.w;
                }
#pragma unroll 1
                for (int t = 0; t < NT_; t++) {
                    float v = so.pt[warp][t][24] * w[24];
#pragma unroll
                    for (int i = 0; i < 6; i++) {
                        const float4 y = *reinterpret_cast<const float4 *>(&so.pt[warp][t][4 * i]);
                        v += y.x * w[4 * i]; v += y.y * w[4 * i + 1]; v += y.z * w[4 * i + 2]; v += y.w * w[4 * i + 3];
                    }
                    p[t] = v;
                }
            }
        } else if (dev) {
            for (int z = lane; z < NU; z += 32) {
                const int k = z / NT_, t = z % NT_;
                float sh = 0.0f, c = 0.0f;   // compensated dot product (Dot2)
#pragma unroll
                for (int j = 0; j < NT_; j++) {
                    dot2ff_next(so.dx[t][j], s_mf[j + 10 * k], sh, c);
                    dot2ff_next(so.dy[t][j], s_mf[NU + j + 10 * k], sh, c);
                }
#pragma unroll
                for (int j = 0; j < NZ; j++) dot2ff_next(so.dz[k][j], s_mf[2 * NU + t + 10 * j], sh, c);
                a.RL[u0 / FR_NV + z] = two_sum(sh, c);
            }
        }
        if (tid == 0) s_pcnt = 0;
        __syncthreads();
        // 7. z lines (alpha, t) and the sum of the three components
        if (tid < (5 - a0) * NT_) {
            const int alpha = a0 + tid / NT_, t = tid % NT_;
            float v[NZ] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int d = 0; d < 3; d++)
#pragma unroll
                for (int c = 0; c < MZ; c++) {
                    const float x = s_p[(alpha * 3 + d) * MZ * NT_ + c * NT_ + t];
#pragma unroll
                    for (int k = 0; k < NZ; k++) v[k] += op.PZ[d][k][c] * x;
                }
            float *R = a.R + u0 + alpha * NU + t;
#pragma unroll
            for (int k = 0; k < NZ; k++) R[10 * k] = v[k];
        }
        __syncthreads();
    }
    fr_grid_done();
}

// -------------------------------------------------------------------------------------------------
// Phase B in FP64: the operators in block fixed point (fr_fx.cuh), one element per CTA
// -------------------------------------------------------------------------------------------------
// As the dense elements' kernel: the operators on the integer multipliers, the pointwise fluxes on the
// FP64 pipe that bounded the kernel with every operator on it. The line interpolation comes first, so
// that a thread then interpolates its own quadrature point's 20 fields in the triangle plane and holds
// them and the flux in registers; the derivatives ride on the projection (Dhx Pt, Dhy Pt, Dhz Pz). Measured, 18^3
// mixed box (5,832 prisms beside 2,916 hexahedra), volume phase: 1.56 -> 0.50 ms.
constexpr int FX_TR = 20 * NF;                        // traces of the listed flux points
constexpr int FX_S = 20 * MZ * NT_ + FX_TR;           // line-interpolated fields and traces, then the flux
static_assert(FX_S >= 15 * NQ && 20 * NU + 5 * NF >= 15 * MZ * NT_, "staging fits over consumed buffers");
constexpr size_t FX_SMEM = sizeof(PriFxS) + sizeof(fx2) * (20 * NU + 5 * NF + FX_S);

template <int NTH>
__device__ __forceinline__ void pri_B_fx_body(const HexArgs<double> &a, const PriOps<double> *gops, long long first, long long stride)
{
    static_assert(NTH == 128, "one thread per quadrature point, state and flux point");
    static_assert(NU + NF <= NTH, "one thread per state and flux point");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ short s_plist[NF];
    __shared__ int s_pcnt, s_mx[10];
    const PriFx *gx = reinterpret_cast<const PriFx *>(gops + 1);
    const PriFxS &op = *reinterpret_cast<const PriFxS *>(smem_raw);
    const int tid = threadIdx.x;
    const bool lane0 = (tid & 31) == 0;
    {
        const int *src = reinterpret_cast<const int *>(&gx->s);
        int *dst = reinterpret_cast<int *>(smem_raw);
        for (int i = tid; i < (int)(sizeof(PriFxS) / sizeof(int)); i += NTH) dst[i] = src[i];
    }
    fx2 *s_u = reinterpret_cast<fx2 *>(smem_raw + sizeof(PriFxS));   // state, then the physical gradient (5 + 3 alpha + d)
    fx2 *s_c = s_u + 20 * NU;                                // common solution
    fx2 *s_t = s_c + 5 * NF;                                 // [20][c][t] line-interpolated fields
    double *s_tr = reinterpret_cast<double *>(s_t + 20 * MZ * NT_);
    fx2 *s_w = s_t;                                          // [15][c][q] transformed flux
    fx2 *s_p = s_u;                                          // [15][c][t] projected in the triangle plane
    const int tq = tid < NQ ? tid % NQT : 0, tc_ = tid < NQ ? tid / NQT : 0;   // this thread's quadrature point
    if (tid < 10) s_mx[tid] = 0;
    if (tid == 0) s_pcnt = 0;
    __syncthreads();
    fr_grid_wait();
    for (long long e = first; e < a.ne; e += stride) {
        if (!fr_elem_ok(a, e, NU, NF)) continue;
        const Geo<double> g = a.geo[e];
        const Phys<double> ph = elem_phys(a, e);
        const long long gf0 = elem_f0(a, e, NF);
        // 1. state and common solution (one point per thread, five variables), largest magnitudes, and
        //    the flux points whose side carries LDG weight
        double val[5] = {0, 0, 0, 0, 0};
        if (tid < NU) {
            const double *U = a.U + elem_u0(a, e, NU) + tid;
#pragma unroll
            for (int alpha = 0; alpha < 5; alpha++) val[alpha] = U[alpha * NU];
        } else if (tid < NU + NF) {
            const long long og = gf0 + (tid - NU);
            const uint32_t pc = a.partner[og];
            const bool isL = (pc & FR_LFLAG) != 0;
            const long long pg = fr_partner(a, pc, og), gL = isL ? og : pg, gR = isL ? pg : og;
#pragma unroll
            for (int alpha = 0; alpha < 5; alpha++)
                val[alpha] = fr_common(0.5 - ph.beta, 0.5 + ph.beta, a.UF[alpha * a.nfpt + gL], a.UF[alpha * a.nfpt + gR]);
            if ((isL ? 0.5 + ph.beta : 0.5 - ph.beta) == 0.0) {
#pragma unroll
                for (int k = 0; k < 4; k++) a.FV[k * a.nfpt + og] = 0.0;
            } else {
                s_plist[atomicAdd(&s_pcnt, 1)] = (short)(tid - NU);
            }
        }
#pragma unroll
        for (int alpha = 0; alpha < 5; alpha++) {
            const int m = (int)__reduce_max_sync(0xffffffffu, (unsigned)fx_mag(val[alpha]));
            if (lane0) atomicMax(&s_mx[alpha], m >> 20);
        }
        __syncthreads();
        int E[5];
#pragma unroll
        for (int alpha = 0; alpha < 5; alpha++) E[alpha] = s_mx[alpha];
        if (tid < NU) {
#pragma unroll
            for (int alpha = 0; alpha < 5; alpha++) s_u[alpha * NU + tid] = fx_from<FX_WS>(val[alpha], E[alpha]);
        } else if (tid < NU + NF) {
#pragma unroll
            for (int alpha = 0; alpha < 5; alpha++) s_c[alpha * NF + tid - NU] = fx_from<FX_WS>(val[alpha], E[alpha]);
        }
        __syncthreads();
        const int nplist = s_pcnt;
        // 2. corrected gradient: triangle planes and z lines, then q = J^-T q~
        int EJ[3], qe[3];   // gradient component k: value = X 2^(E - 1078 - FX_WS + qe[k])
#pragma unroll
        for (int k = 0; k < 3; k++) {
            EJ[k] = fx_column_exp(g.Ji, k);
            qe[k] = op.kD + EJ[k] - 1022;
        }
        for (int it = tid; it < 5 * NU; it += NTH) {
            const int alpha = it / NU, z = it % NU, k = z / NT_, t = z % NT_;
            const fx2 *u = s_u + alpha * NU, *c = s_c + alpha * NF;
            fxacc q[3] = {{FX_HALF, 0}, {FX_HALF, 0}, {FX_HALF, 0}};
#pragma unroll
            for (int j = 0; j < NT_; j++) {
                fx_mac(q[0], op.Dhx[t][j], u[j + 10 * k]);
                fx_mac(q[1], op.Dhy[t][j], u[j + 10 * k]);
            }
#pragma unroll 1
            for (int f = 0; f < 3; f++) {
                fxacc l{FX_HALF, 0};
#pragma unroll
                for (int b = 0; b < NZ; b++) fx_mac(l, op.Lf[f][t][b], c[20 + 16 * f + b + 4 * k]);
                const fx2 lf = fx_limbs(fx_sum(l));
                fx_mac(q[0], op.nf[f][0], lf);
                fx_mac(q[1], op.nf[f][1], lf);
            }
#pragma unroll
            for (int j = 0; j < NZ; j++) fx_mac(q[2], op.Dhz[k][j], u[t + 10 * j]);
            fx_mac(q[2], op.liftzR[k], c[10 + t]);
            fx_mac(q[2], op.liftzL[k], fx2{-c[t].h, -c[t].l});
            fx2 qr[3];
#pragma unroll
            for (int d = 0; d < 3; d++) qr[d] = fx_limbs(fx_sum(q[d]));
#pragma unroll
            for (int kk = 0; kk < 3; kk++) {
                fxacc s{FX_HALF, 0};
#pragma unroll
                for (int d = 0; d < 3; d++) fx_mac(s, fx_factor(g.Ji[3 * d + kk], EJ[kk]), qr[d]);
                s_u[(5 + alpha * 3 + kk) * NU + z] = fx_limbs(fx_sum(s));
            }
        }
        __syncthreads();
        // 3. traces of the 20 fields at the listed flux points, four threads per point
        for (int it = tid; it < 4 * nplist; it += NTH) {
            const int li = it >> 2, fg = it & 3, s = s_plist[li];
            fxacc t[5] = {{0, 0}, {0, 0}, {0, 0}, {0, 0}, {0, 0}};
            const fx2 *x = s_u + 5 * fg * NU;
            if (s < 20) {
                const fx2 *l = s < 10 ? op.lzL : op.lzR;
                x += s % 10;
#pragma unroll
                for (int k = 0; k < NZ; k++)
#pragma unroll
                    for (int i = 0; i < 5; i++) fx_mac(t[i], l[k], x[i * NU + 10 * k]);
            } else {
                const int f = (s - 20) / 16, loc = (s - 20) % 16;
                const fx2 *l = op.Ef[f][loc % 4];
                x += 10 * (loc / 4);
#pragma unroll 2
                for (int j = 0; j < NT_; j++)
#pragma unroll
                    for (int i = 0; i < 5; i++) fx_mac(t[i], l[j], x[i * NU + j]);
            }
#pragma unroll
            for (int i = 0; i < 5; i++) {
                const int f = 5 * fg + i, Ea = s_mx[f < 5 ? f : (f - 5) / 3];
                s_tr[li * 20 + f] = fx_double(fx_sum(t[i]), Ea - 1080 - FX_WS + op.kF + fx_field_exp(f, qe), Ea >= 2047);
            }
        }
        // 4. interpolation: z lines, then this thread's quadrature point in the triangle plane; the flux there
        for (int it = tid; it < 20 * NT_; it += NTH) {
            const int f = it / NT_, t = it % NT_;
            fx2 u[NZ];
#pragma unroll
            for (int k = 0; k < NZ; k++) u[k] = s_u[f * NU + t + 10 * k];
#pragma unroll
            for (int c = 0; c < MZ; c++) {
                fxacc s{FX_HALF, 0};
#pragma unroll
                for (int k = 0; k < NZ; k++) fx_mac(s, op.Bz[c][k], u[k]);
                s_t[(f * MZ + c) * NT_ + t] = fx_limbs(fx_sum(s));
            }
        }
        __syncthreads();
        bool ok = true;
        double f[3][5];
        int fm[5] = {0, 0, 0, 0, 0};
        if (tid < NQ) {
            fx2 b[NT_];
#pragma unroll
            for (int t = 0; t < NT_; t++) b[t] = gx->Bt[tq][t];
            double u[5], gq[5][3];
#pragma unroll
            for (int i = 0; i < 20; i++) {
                const fx2 *x = s_t + (i * MZ + tc_) * NT_;
                fxacc s{0, 0};
#pragma unroll
                for (int t = 0; t < NT_; t++) fx_mac(s, b[t], x[t]);
                const int alpha = i < 5 ? i : (i - 5) / 3;
                const double v = fx_double(fx_sum(s), E[alpha] - 1080 - FX_WS + op.kB + fx_field_exp(i, qe), E[alpha] >= 2047);
                if (i < 5) u[i] = v;
                else gq[alpha][(i - 5) % 3] = v;
            }
            ok = total_flux(ph, u, gq, f);
            // det J J^-1 f, in place
#pragma unroll
            for (int alpha = 0; alpha < 5; alpha++) {
                const double f0 = f[0][alpha], f1 = f[1][alpha], f2 = f[2][alpha];
#pragma unroll
                for (int d = 0; d < 3; d++) {
                    f[d][alpha] = g.det * (g.Ji[3 * d] * f0 + g.Ji[3 * d + 1] * f1 + g.Ji[3 * d + 2] * f2);
                    fm[alpha] = max(fm[alpha], fx_mag(f[d][alpha]));
                }
            }
        }
        flag_status(a.status, ok);
#pragma unroll
        for (int alpha = 0; alpha < 5; alpha++) {
            const int m = (int)__reduce_max_sync(0xffffffffu, (unsigned)fm[alpha]);
            if (lane0) atomicMax(&s_mx[5 + alpha], m >> 20);
        }
        // 5. own-normal viscous flux at the listed flux points
        for (int li = tid; li < nplist; li += NTH) {
            const int s = s_plist[li];
            const double *v = s_tr + li * 20;
            double uf[5], qf[5][3];
#pragma unroll
            for (int alpha = 0; alpha < 5; alpha++) {
                uf[alpha] = v[alpha];
#pragma unroll
                for (int d = 0; d < 3; d++) qf[alpha][d] = v[5 + alpha * 3 + d];
            }
            const double *nt = a.fnrm + (e * 6 + face_of(s)) * 4;
            const double n[3] = {nt[0], nt[1], nt[2]};
            double fvn[4];
            viscous_normal_flux(ph, uf, qf, n, fvn);
#pragma unroll
            for (int k = 0; k < 4; k++) a.FV[k * a.nfpt + gf0 + s] = fvn[k];
        }
        __syncthreads();
        // 6. the flux in fixed point, over the interpolated fields and the traces
        if (tid < NQ) {
#pragma unroll
            for (int alpha = 0; alpha < 5; alpha++) {
                const int Ef = s_mx[5 + alpha];
#pragma unroll
                for (int d = 0; d < 3; d++) s_w[(alpha * 3 + d) * NQ + tid] = fx_from(f[d][alpha], Ef);
            }
        }
        __syncthreads();
        // 7. projection with the corrected divergence: triangle planes (Dhx Pt, Dhy Pt, Pt), then z and the
        //    sum of the three components
        for (int it = tid; it < 5 * MZ * NT_; it += NTH) {
            const int alpha = it / (MZ * NT_), r = it % (MZ * NT_), c = r / NT_, t = r % NT_;
#pragma unroll 1
            for (int d = 0; d < 3; d++) {
                const fx2 *x = s_w + (alpha * 3 + d) * NQ + NQT * c, *l = op.PT[d][t];
                fxacc s{FX_HALF, 0};
#pragma unroll 5
                for (int q = 0; q < NQT; q++) fx_mac(s, l[q], x[q]);
                s_p[(alpha * 3 + d) * MZ * NT_ + r] = fx_limbs(fx_sum(s));
            }
        }
        __syncthreads();
        double *R = a.R + elem_u0(a, e, NU);
        for (int it = tid; it < 5 * NU; it += NTH) {
            const int alpha = it / NU, z = it % NU, k = z / NT_, t = z % NT_;
            fxacc s{0, 0};
#pragma unroll
            for (int d = 0; d < 3; d++)
#pragma unroll
                for (int c = 0; c < MZ; c++) fx_mac(s, op.PZ[d][k][c], s_p[(alpha * 3 + d) * MZ * NT_ + c * NT_ + t]);
            const int Ef = s_mx[5 + alpha];
            R[it] = fx_double(fx_sum(s), Ef - 1080 + op.kT + op.kZ, Ef >= 2047);
        }
        __syncthreads();
        if (tid < 10) s_mx[tid] = 0;
        if (tid == 0) s_pcnt = 0;
        __syncthreads();
    }
    fr_grid_done();
}

// -------------------------------------------------------------------------------------------------
// Phase C: interface group
// -------------------------------------------------------------------------------------------------
template <typename T, int NTH>
__device__ __forceinline__ void pri_C_body(const HexArgs<T> &a, const PriOps<T> *gops, const PriOpsFF *opsff, long long first, long long stride)
{
    constexpr bool FX = sizeof(T) == 8;   // FP64: the lift in block fixed point (fr_fx.cuh)
    static_assert(!FX || NF <= NTH, "one flux point per thread");
    __shared__ PriOps<typename std::conditional<FX, float, T>::type> op_;
    __shared__ T s_d[FX ? 1 : 5 * NF];
    __shared__ fx2 s_dx[FX ? 5 * NF : 1], s_lf[FX ? 3 * NT_ * NZ : 1], s_lz[FX ? 2 * NZ : 1];
    __shared__ int s_mx[2][5];
    __shared__ ff s_dff[sizeof(T) == 4 ? NF : 1];   // low-Mach form: transformed mass flux (float-float)
    const auto &op = op_;
    int par = 0, kD = 0;
    if constexpr (FX) {
        const PriFxS &ox = reinterpret_cast<const PriFx *>(gops + 1)->s;
        for (int i = threadIdx.x; i < 3 * NT_ * NZ; i += NTH) s_lf[i] = (&ox.Lf[0][0][0])[i];
        for (int i = threadIdx.x; i < 2 * NZ; i += NTH) s_lz[i] = i < NZ ? ox.liftzL[i] : ox.liftzR[i - NZ];
        if (threadIdx.x < 10) s_mx[threadIdx.x / 5][threadIdx.x % 5] = 0;
        kD = ox.kD;
    } else {
        load_ops<T, NTH>(gops, op_);
    }
    __syncthreads();
    fr_grid_wait();
    for (long long e = first; e < a.ne; e += stride) {
        if (!fr_elem_ok(a, e, NU, NF)) continue;
        const Geo<T> g = a.geo[e];
        const Phys<T> ph = elem_phys(a, e);
        const long long gf0 = elem_f0(a, e, NF);
        bool dev = false;
        if constexpr (sizeof(T) == 4) dev = ph.dev != 0;
        bool ok = true;
        T dv[1][5] = {{T(0), T(0), T(0), T(0), T(0)}};
        for (int s = threadIdx.x; s < NF; s += NTH) {
            const uint32_t pc = a.partner[gf0 + s];
            const bool isL = (pc & FR_LFLAG) != 0;
            const long long og = gf0 + s, pg = fr_partner(a, pc, og);
            // own and partner values (the own ones do not wait for the partner's index), then the pair's L and
            // R states: one flux evaluation per warp, whatever roles its points have
            T uL[5], uR[5], fvL[4], fvR[4];
#pragma unroll
            for (int k = 0; k < 5; k++) { uL[k] = a.UF[k * a.nfpt + og]; uR[k] = a.UF[k * a.nfpt + pg]; }
#pragma unroll
            for (int k = 0; k < 4; k++) { fvL[k] = a.FV[k * a.nfpt + og]; fvR[k] = a.FV[k * a.nfpt + pg]; }
#pragma unroll
            for (int k = 0; k < 5; k++) { const T o = uL[k]; uL[k] = isL ? o : uR[k]; uR[k] = isL ? uR[k] : o; }
#pragma unroll
            for (int k = 0; k < 4; k++) { const T o = fvL[k]; fvL[k] = isL ? o : fvR[k]; fvR[k] = isL ? fvR[k] : o; }
            const T *nt = a.fnrm + (e * 6 + face_of(s)) * 4;
            const T mag = nt[3];
            const T nL[3] = {isL ? nt[0] : -nt[0], isL ? nt[1] : -nt[1], isL ? nt[2] : -nt[2]};
            T F[5];
            if (dev) {
                if constexpr (sizeof(T) == 4) {
                    float sw;
                    ok &= common_flux_dev(ph, uL, uR, fvL, fvR, nL, F, sw);
                    // mass flux in float-float: 1/2 (mL - mR) + (s/2 + tau)(rho_L - rho_R),
                    // mX = own-normal n.(rho v)
                    const ff mo = a.MF[og], mp = a.MF[pg];
                    const ff mL = isL ? mo : mp, mR = isL ? mp : mo;
                    const ff Fr = ff_add(ff_mul_f(ff_sub(mL, mR), 0.5f), ff_mul_f(two_sum(uL[0], -uR[0]), 0.5f * sw + ph.tau));
                    const ff magf = a.fnrm64[(e * 6 + face_of(s)) * 4 + 3], Dr = ff_mul(magf, Fr);
                    s_dff[s] = isL ? Dr : ff_neg(Dr);
                }
            } else {
                ok &= common_flux(ph, uL, uR, fvL, fvR, nL, F);
            }
            const T sc = isL ? mag : -mag;
#pragma unroll
            for (int k = 0; k < 5; k++) {
                if constexpr (FX) dv[0][k] = sc * F[k];
                else s_d[k * NF + s] = sc * F[k];
            }
        }
        flag_status(a.status, ok);
        T *R = a.R + elem_u0(a, e, NU);
        const T idet = g.nidet;
        if constexpr (FX) {
            int E[5];
            fx_stage5<NF, NTH, 1>(dv, s_dx, s_mx, par, E);
            for (int it = threadIdx.x; it < 5 * NU; it += NTH) {
                const int alpha = it / NU, r = it % NU, k = r / NT_, t = r % NT_, Ea = s_mx[par ^ 1][alpha];
                const fx2 *D = s_dx + alpha * NF;
                fxacc x{0, 0};
                fx_mac(x, s_lz[k], D[t]);
                fx_mac(x, s_lz[NZ + k], D[10 + t]);
#pragma unroll
                for (int f = 0; f < 3; f++)
#pragma unroll
                    for (int b = 0; b < NZ; b++) fx_mac(x, s_lf[(f * NT_ + t) * NZ + b], D[20 + 16 * f + b + 4 * k]);
                const double v = (R[it] + fx_double(fx_sum(x), Ea - 1080 + kD, Ea >= 2047)) * idet;
                if (a.rkstage == 0) R[it] = v;
                else rk_fold(a, elem_u0(a, e, NU) + it, v);
            }
        } else {
            __syncthreads();
        }
        if constexpr (FX) {
        } else if (!dev) {
            for (int it = threadIdx.x; it < 5 * NU; it += NTH) {
                const int alpha = it / NU, r = it % NU, k = r / NT_, t = r % NT_;
                const T *D = s_d + alpha * NF;
                T v = R[it] + op.liftzL[k] * D[t] + op.liftzR[k] * D[10 + t];
#pragma unroll
                for (int f = 0; f < 3; f++)
#pragma unroll
                    for (int b = 0; b < NZ; b++) v += op.Lf[f][t][b] * D[20 + 16 * f + b + 4 * k];
                if (a.rkstage == 0) R[it] = v * idet;
                else rk_fold(a, elem_u0(a, e, NU) + it, v * idet);
            }
        } else if constexpr (sizeof(T) == 4) {
            // low-Mach form: R_rho in float-float, R_E = R_(E - H0 rho) + H0 R_rho
            const PriOpsFF &o = *opsff;
            const ff idet64 = a.geo64[e].idet;
            const ff H0 = ph.H0ff;
            const long long pbase = elem_u0(a, e, NU) / FR_NV;
            for (int z = threadIdx.x; z < NU; z += NTH) {
                const int k = z / NT_, t = z % NT_;
                ff r = a.RL[pbase + z];
                r = ff_fma(ffop(o, o.hi.liftzL[k]), s_dff[t], r);
                r = ff_fma(ffop(o, o.hi.liftzR[k]), s_dff[10 + t], r);
#pragma unroll
                for (int f = 0; f < 3; f++)
#pragma unroll
                    for (int b = 0; b < NZ; b++) r = ff_fma(ffop(o, o.hi.Lf[f][t][b]), s_dff[20 + 16 * f + b + 4 * k], r);
                const ff Rrho = ff_mul(r, idet64);
                float out[5];
                out[0] = Rrho.hi + Rrho.lo;
#pragma unroll
                for (int alpha = 1; alpha < 5; alpha++) {
                    const T *D = s_d + alpha * NF;
                    T v = R[alpha * NU + z] + op.liftzL[k] * D[t] + op.liftzR[k] * D[10 + t];
#pragma unroll
                    for (int f = 0; f < 3; f++)
#pragma unroll
                        for (int b = 0; b < NZ; b++) v += op.Lf[f][t][b] * D[20 + 16 * f + b + 4 * k];
                    out[alpha] = v * idet;
                }
                const ff e4 = ff_fma(H0, Rrho, ff_of(out[4]));
                out[4] = e4.hi + e4.lo;
#pragma unroll
                for (int alpha = 0; alpha < 5; alpha++) {
                    if (a.rkstage == 0) R[alpha * NU + z] = out[alpha];
                    else rk_fold(a, elem_u0(a, e, NU) + alpha * NU + z, out[alpha]);
                }
            }
        }
        __syncthreads();
    }
    fr_grid_done();
}


}  // namespace
}  // namespace pri
