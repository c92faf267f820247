// fr_dense.cu -- kernels of the anti-aliased Navier-Stokes FR right-hand side for element types
// without tensor-product structure (p = 3): tetrahedra and pyramids.
//
// Sum factorisation (Sec. 4) serves hexahedra and prisms only; for tetrahedra and pyramids (Sec. 1)
// every operator is a dense matrix applied per element: NU solution points (20 / 30), NF flux points
// on NFACE faces (4 x 10 / a 16-point base and 4 x 10), 125 quadrature points. Same three fused
// phases as the other types: A face solution, B volume group, C interface group. The volume group
// evaluates, per element, the con_u average, the corrected gradient (Dh_d u plus the face lift of the
// common solution, then J^-T), the own-normal viscous flux at the flux points whose LDG weight is not
// zero, the interpolation of the 20 fields (u and its gradient) to the quadrature points, the
// pointwise flux and its transformation det J J^-1 f, and the L2 projection with the corrected
// divergence folded in (R~ = sum_d (Dh_d Pj) f~_d: one dense NU x 125 operator per direction).
//
// The operator tables (DenseOps: 100 KB / 160 KB in FP64) stay in global memory, read through the
// L1/L2 caches; they are stored with the output index fastest, so that a warp's lanes, which compute
// consecutive outputs, read consecutive entries while the field values they multiply are one
// shared-memory broadcast per warp (16-byte vector loads along the solution-point index, whose rows
// are padded to NUS with zero operator rows).
#include <cuda_runtime.h>

#include "fr_internal.h"
#include "fr_physics.cuh"
#include "fr_tcgen05.cuh"

namespace {

constexpr int NQ = FR_TQ, NQP = FR_TQP;

// Tensor-core interpolation of the mixed forms: D[q][f] = sum_j B[q][j] x_f[j] for the 20 fields
// (state and gradient) of one element, M = 128 quadrature-point rows (125 used), N = 32 field rows
// (20 used), K = the split form's NU-wide slices (tc::SplitForm; FP16: [B_hi | B_hi | B_lo] against
// [x_hi | x_lo | x_hi]; BF16: six slices of three parts), zero-padded to a multiple of 16. The
// operator tile is split once per CTA; each element writes its 20 field rows (scaled by a power of
// two per row) and reads its quadrature point's 20 values back from tensor memory, one lane per
// thread.
template <typename OPS, int TCM>
struct DenseTC {
    static constexpr int KI = tc::split_k<TCM>(OPS::NU);       // FP16: 64 (tetrahedron), 96 (pyramid)
    static constexpr int SBO = KI / 8 * 128;
    static constexpr int A_BYTES = 16 * SBO;                   // 128 rows
    static constexpr int B_BYTES = 4 * SBO;                    // 32 rows
    static constexpr int HEAD = A_BYTES + B_BYTES + 32 * 4 + 16;   // tiles, row shifts, barrier, TMEM slot
    static constexpr int BYTES = HEAD + 128;                   // + alignment slack
    static constexpr uint32_t IDESC = tc::idesc_f16(TCM - 1, 128, 32);
};

// 16 bytes of T (4 floats or 2 doubles): one vector shared-memory load
template <typename T>
struct alignas(16) V16 {
    static constexpr int n = 16 / sizeof(T);
    T v[n];
};
template <typename T>
__device__ __forceinline__ V16<T> ld16(const T *p)
{
    return *reinterpret_cast<const V16<T> *>(p);
}

// The float-float table type of an operator table, and one entry of it as a pair (the lo part sits
// at the same offset in the second table).
template <typename OPS>
using FFOf = DenseOpsFF<DenseOps<float, OPS::NU, OPS::NF, OPS::NFACE>>;
template <typename FF>
__device__ __forceinline__ ff ffat(const FF &o, const float &hi)
{
    const float *h0 = reinterpret_cast<const float *>(&o.hi);
    return ff{hi, reinterpret_cast<const float *>(&o.lo)[&hi - h0]};
}

// -------------------------------------------------------------------------------------------------
// Phase A: disu (U^f = M0 U)
// -------------------------------------------------------------------------------------------------
// EPB elements per CTA iteration, one thread per (element, flux point). The states of the EPB
// elements are staged in shared memory with coalesced loads; each thread keeps its column of M0 in
// registers for the whole persistent loop and reads the state with 16-byte broadcast loads.
// The reduced precisions evaluate every face value as a compensated dot product (Dot2 of Ogita, Rump
// and Oishi) of the float-float M0 row (hi + lo) with the FP32 state, rounded once: at low Mach the
// Rusanov dissipation (1/2)(|v.n| + c)(u_L - u_R), c about 10 |v|, lifts any rounding of a face
// value into R. Low-Mach FP32 form (ph.dev): the face solution of the deviations from the reference
// state, and the own-normal mass flux n.(rho v) at every flux point in float-float: first
// m_f = n_f . (rho v) at the solution points per face (the face normal is constant on an affine
// element), then the same compensated dot product with m_f.
// Pyramids (224 threads per CTA): registers capped for five CTAs per SM, up from two at the
// compiler's 112 (a few spilled values; the tetrahedral form is faster uncapped). Otherwise (0) the
// compiler's own register count.
template <typename OPS, int EPB>
__global__ void __launch_bounds__(OPS::NF * EPB, OPS::NF * EPB > 192 ? 1280 / (OPS::NF * EPB) : 0)
k_dense_disu(HexArgs<float> a, const OPS *__restrict__ op, const FFOf<OPS> *__restrict__ opsff)
{
    constexpr int NU = OPS::NU, NF = OPS::NF, NUS = OPS::NUS, NFACE = OPS::NFACE, NTH = NF * EPB;
    using T = float;
    constexpr int VN = V16<T>::n;
    __shared__ __align__(16) T s_u[EPB][FR_NV * NUS];
    __shared__ __align__(16) ff s_m[EPB][NFACE * NUS];
    const int el = threadIdx.x / NF, s = threadIdx.x % NF;
    T col[NUS];
#pragma unroll
    for (int z = 0; z < NUS; z++) col[z] = op->M0t[z][s];   // pad rows are zero
    float col_lo[NUS];                              // lo parts of the FP32 column
#pragma unroll
    for (int z = 0; z < NUS; z++) col_lo[z] = opsff->lo.M0t[z][s];
    if constexpr (NUS > NU) {
        for (int i = threadIdx.x; i < EPB * FR_NV * (NUS - NU); i += NTH) {
            const int l = i / (FR_NV * (NUS - NU)), r = i % (FR_NV * (NUS - NU));
            s_u[l][(r / (NUS - NU)) * NUS + NU + r % (NUS - NU)] = T(0);
        }
    }
    fr_grid_wait();
    const long long ng = (a.ne + EPB - 1) / EPB;
    for (long long g = blockIdx.x; g < ng; g += gridDim.x) {
        const long long e0 = g * EPB;
        const int nel = (int)(a.ne - e0 < EPB ? a.ne - e0 : EPB);
        {
            bool blk_ok = true;
            for (int k = 0; k < nel; k++) blk_ok = blk_ok && fr_elem_ok(a, e0 + k, NU, NF);
            if (!blk_ok) continue;
        }
        for (int i = threadIdx.x; i < nel * FR_NV * NU; i += NTH) {
            const int l = i / (FR_NV * NU), r = i % (FR_NV * NU), alpha = r / NU;
            const long long e = e0 + l;
            T v = a.U[elem_u0(a, e, NU) + r];
            const Phys<T> ph = elem_phys(a, e);
            if (ph.dev) v -= alpha == 0 ? ph.rref : (alpha == 4 ? ph.eref : T(0));
            s_u[l][alpha * NUS + r % NU] = v;
        }
        __syncthreads();
        for (int i = threadIdx.x; i < nel * NFACE * NU; i += NTH) {
            const int l = i / (NFACE * NU), r = i % (NFACE * NU), f = r / NU, z = r % NU;
            const long long e = e0 + l;
            if (!elem_phys(a, e).dev) continue;
            const ff *nt = a.fnrm64 + (e * 6 + f) * 4;
            const float *u = s_u[l];
            ff m = ff_mul_f(nt[0], u[NUS + z]);
            m = ff_add(m, ff_mul_f(nt[1], u[2 * NUS + z]));
            s_m[l][f * NUS + z] = ff_add(m, ff_mul_f(nt[2], u[3 * NUS + z]));
        }
        __syncthreads();
        if (el < nel) {
            const long long e = e0 + el;
            const long long f0 = elem_f0(a, e, NF);
            const T *u = s_u[el];
            // sh + c = sum_z (col + col_lo)[z] x[z]: exact products (one FMA each), TwoSum
            // accumulation of the high parts, the errors summed in c
            float sh[FR_NV], c[FR_NV];
#pragma unroll
            for (int alpha = 0; alpha < FR_NV; alpha++) { sh[alpha] = 0.0f; c[alpha] = 0.0f; }
#pragma unroll
            for (int z = 0; z < NUS; z += VN) {
#pragma unroll
                for (int alpha = 0; alpha < FR_NV; alpha++) {
                    const V16<T> x = ld16(u + alpha * NUS + z);
#pragma unroll
                    for (int j = 0; j < VN; j++) {
                        const float pr = col[z + j] * x.v[j];
                        const float er = __fmaf_rn(col_lo[z + j], x.v[j], __fmaf_rn(col[z + j], x.v[j], -pr));
                        const ff t = two_sum(sh[alpha], pr);
                        sh[alpha] = t.hi;
                        c[alpha] += t.lo + er;
                    }
                }
            }
#pragma unroll
            for (int alpha = 0; alpha < FR_NV; alpha++) a.UF[alpha * a.nfpt + f0 + s] = sh[alpha] + c[alpha];
            if (elem_phys(a, e).dev) {
                const ff *m = s_m[el] + OPS::FACE(s) * NUS;
                float sh = 0.0f, c = 0.0f;
#pragma unroll
                for (int z = 0; z < NU; z++) {
                    const ff mz = m[z];
                    const float pr = col[z] * mz.hi;
                    const float er = __fmaf_rn(opsff->lo.M0t[z][s], mz.hi, __fmaf_rn(col[z], mz.lo, __fmaf_rn(col[z], mz.hi, -pr)));
                    const ff t = two_sum(sh, pr);
                    sh = t.hi;
                    c += t.lo + er;
                }
                a.MF[f0 + s] = two_sum(sh, c);
            }
        }
        __syncthreads();
    }
    fr_grid_done();
}

// The same in FP64, with the face values in block fixed point (fr_fx.cuh): on the FP64 pipe the 5 NU
// multiply-adds per flux point bounded the kernel (11^3 hexahedron/pyramid box, face phase 92 -> 38 us). A
// thread keeps its column of M0 in registers.
template <typename OPS, int EPB>
__global__ void __launch_bounds__(OPS::NF * EPB) k_dense_disu_fx(HexArgs<double> a, const OPS *__restrict__ ops)
{
    constexpr int NU = OPS::NU, NF = OPS::NF, NUS = OPS::NUS, NTH = NF * EPB;
    static_assert(NU <= 32 && NTH % 32 == 0, "one variable of one element per warp pass");
    const auto &op = ops->fx;
    __shared__ __align__(16) fx2 s_u[EPB][FR_NV * NUS];
    __shared__ int s_E[EPB * FR_NV];
    const int el = threadIdx.x / NF, s = threadIdx.x % NF, kM = op.kM;
    fx2 col[NUS];
#pragma unroll
    for (int z = 0; z < NUS; z++) col[z] = op.M0t[z][s];   // pad rows are zero
    if constexpr (NUS > NU) {
        for (int i = threadIdx.x; i < EPB * FR_NV * (NUS - NU); i += NTH) {
            const int l = i / (FR_NV * (NUS - NU)), r = i % (FR_NV * (NUS - NU));
            s_u[l][(r / (NUS - NU)) * NUS + NU + r % (NUS - NU)] = fx2{0, 0};
        }
    }
    fr_grid_wait();
    const long long ng = (a.ne + EPB - 1) / EPB;
    for (long long g = blockIdx.x; g < ng; g += gridDim.x) {
        const long long e0 = g * EPB;
        const int nel = (int)(a.ne - e0 < EPB ? a.ne - e0 : EPB);
        {
            bool blk_ok = true;
            for (int k = 0; k < nel; k++) blk_ok = blk_ok && fr_elem_ok(a, e0 + k, NU, NF);
            if (!blk_ok) continue;
        }
        for (int b = threadIdx.x / 32; b < nel * FR_NV; b += NTH / 32)
            fx_warp_block<1>(a.U + elem_u0(a, e0 + b / FR_NV, NU) + (b % FR_NV) * NU, NU, s_u[b / FR_NV] + (b % FR_NV) * NUS, s_E + b);
        __syncthreads();
        if (el < nel) {
            double *o = a.UF + elem_f0(a, e0 + el, NF) + s;
#pragma unroll 1
            for (int alpha = 0; alpha < FR_NV; alpha++, o += a.nfpt) {
                const fx2 *u = s_u[el] + alpha * NUS;
                const int E = s_E[el * FR_NV + alpha];
                fxacc t{0, 0};
#pragma unroll
                for (int z = 0; z < NUS; z += 2) {
                    const int4 y = *reinterpret_cast<const int4 *>(u + z);
                    fx_mac(t, col[z], fx2{y.x, y.y});
                    fx_mac(t, col[z + 1], fx2{y.z, y.w});
                }
                *o = fx_double(fx_sum(t), E - 1080 + kM, E >= 2047);
            }
        }
        __syncthreads();
    }
    fr_grid_done();
}

// -------------------------------------------------------------------------------------------------
// Phase B: volume group, one element per CTA of NTH threads (persistent over elements)
// -------------------------------------------------------------------------------------------------
template <int NTH, typename OPS, int TCM>
__global__ void __launch_bounds__(NTH, TCM == 0 ? 8 : 6) k_dense_B(HexArgs<float> a, const OPS *__restrict__ op, const FFOf<OPS> *__restrict__ opsff)
{
    using T = float;
    constexpr int NU = OPS::NU, NF = OPS::NF, NFACE = OPS::NFACE, NUS = OPS::NUS;
    static_assert(NTH >= NQ, "one thread per quadrature point");
    static_assert(TCM == 0 || NTH == 128, "tensor-core form: one warpgroup per element");
    using TC = DenseTC<OPS, TCM == 0 ? 1 : TCM>;
    using SF = tc::SplitForm<TCM == 0 ? 1 : TCM>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ short s_plist[NF];
    __shared__ int s_pcnt;
    __shared__ __align__(8) double s_mfb[3 * NU];   // low-Mach form: transformed mass flux
    __shared__ __align__(8) double s_rlb[3 * NU];   // low-Mach form: Dh_d of it, per d
    constexpr int VW = V16<T>::n;
    constexpr int NCH = NTH / NU;                 // quadrature-point chunks of the projection
    unsigned char *arr = smem_raw;
    // tensor-core state (TCM != 0): operator tile, field tile, row shifts, barrier, TMEM address
    unsigned char *tA = nullptr, *tB = nullptr;
    int *s_sh = nullptr;
    uint64_t *mbar = nullptr;
    uint32_t *s_tmem = nullptr, tmem = 0, parity = 0;
    bool tc_fail = false, first_wait = true;
    if constexpr (TCM != 0) {
        const uint32_t raw = tc::smem_u32(arr);
        tA = arr + ((128 - (raw & 127)) & 127);
        tB = tA + TC::A_BYTES;
        s_sh = reinterpret_cast<int *>(tB + TC::B_BYTES);
        mbar = reinterpret_cast<uint64_t *>(s_sh + 32);
        s_tmem = reinterpret_cast<uint32_t *>(mbar + 1);
        arr = tA + TC::HEAD;
        tc::setup(mbar, s_tmem, 32);
        for (int i = threadIdx.x; i < 128 * TC::KI; i += NTH) {   // the split form's slices of B, rows q
            const int n = i / TC::KI, k = i % TC::KI, sg = k / NU;
            uint16_t pp[3] = {0, 0, 0};
            if (n < NQ && sg < SF::SEGS) tc::split_parts<TCM>((float)op->Bt[k % NU][n], pp);
            *reinterpret_cast<uint16_t *>(tA + tc::core_offset(n, k, TC::SBO)) = sg < SF::SEGS ? pp[SF::y_part(sg)] : (uint16_t)0;
        }
        for (int i = threadIdx.x; i < 32 * TC::KI; i += NTH)     // field rows 20..31 and the K pad stay zero
            *reinterpret_cast<uint16_t *>(tB + tc::core_offset(i / TC::KI, i % TC::KI, TC::SBO)) = 0;
        tc::fence_async_smem();
        tc::fence_before_sync();
        __syncthreads();
        tc::fence_after_sync();
        tmem = *s_tmem;
    }
    T *s_u = reinterpret_cast<T *>(arr);        // [5][NUS] state
    T *s_q = s_u + 5 * NUS;                       // [15][NUS] physical gradient (field 5 + 3 alpha + d of s_u)
    T *s_c = s_q + 15 * NUS;                      // [5][NF] common solution
    T *s_w = s_c + 5 * NF;                        // [20][NQP] fields at quadrature points, then f~
    T *s_red = s_w + 15 * NQP;                    // [NCH][5][NU] projection partial sums (fields 15-19 are dead by then)
    static_assert(NCH * 5 * NU <= 5 * NQP, "partial sums fit in the dead quadrature-point rows");
    static_assert(NUS % VW == 0 && (NUS * sizeof(T)) % 16 == 0 && (NQP * sizeof(T)) % 16 == 0 && (NF * sizeof(T)) % 16 == 0,
                  "16-byte rows");
    // pads that meet zero operator rows in the vector loads stay zero: s_w columns NQ.. and the
    // solution-point columns NU.. of the 20 fields
    for (int it = threadIdx.x; it < 20 * (NQP - NQ); it += NTH) s_w[(it / (NQP - NQ)) * NQP + NQ + it % (NQP - NQ)] = T(0);
    if constexpr (NUS > NU)
        for (int it = threadIdx.x; it < 20 * (NUS - NU); it += NTH) s_u[(it / (NUS - NU)) * NUS + NU + it % (NUS - NU)] = T(0);
    fr_grid_wait();
    for (long long e = blockIdx.x; e < a.ne; e += gridDim.x) {
        if (!fr_elem_ok(a, e, NU, NF)) continue;
        const Geo<T> g = a.geo[e];
        const Phys<T> ph = elem_phys(a, e);
        const T *U = a.U + elem_u0(a, e, NU);
        const long long gf0 = elem_f0(a, e, NF);
        const bool dev = ph.dev != 0;
        for (int it = threadIdx.x; it < 5 * NU; it += NTH) {
            T v = U[it];
            if (dev) v -= it < NU ? ph.rref : (it >= 4 * NU ? ph.eref : T(0));
            s_u[(it / NU) * NUS + it % NU] = v;
        }
        // low-Mach form: the volume part of R~_rho, sum_d Dh_d (det J J^-1 rho v)_d, in about 48
        // bits or better (rho v lies in the solution space, so its L2 projection is itself and
        // the corrected divergence Dh applies at the solution points). First the transformed
        // mass flux (read from the state in global memory, so that it is ready at the first
        // barrier); the 3 NU products Dh_d m_d then ride along with the gradient items below.
        // The dense product costs 3 NU^2 multiply-adds per element: on the tetrahedron (NU = 20)
        // the FP64 pipe, idle in this kernel, does them faster than float-float arithmetic on
        // the busy FP32 pipe; on the pyramid (NU = 30) the FP64 pipe would become the limit, so
        // it stays in float-float.
        if (dev) {
            const GeoLM &g64 = a.geo64[e];
            for (int z = threadIdx.x; z < NU; z += NTH) {
                const float m0 = U[NU + z], m1 = U[2 * NU + z], m2 = U[3 * NU + z];
#pragma unroll
                for (int d = 0; d < 3; d++) {
                    if constexpr (NU <= 20) {
                        s_mfb[d * NU + z] = g64.det * (g64.Ji[3 * d] * (double)m0 + g64.Ji[3 * d + 1] * (double)m1 + g64.Ji[3 * d + 2] * (double)m2);
                    } else {
                        ff *s_mf = reinterpret_cast<ff *>(s_mfb);
                        s_mf[d * NU + z] = ff_add(ff_add(ff_mul_f(g64.cm[3 * d], m0), ff_mul_f(g64.cm[3 * d + 1], m1)), ff_mul_f(g64.cm[3 * d + 2], m2));
                    }
                }
            }
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
        // corrected gradient q~_d = Dh_d u + sum_f n_f,d (L_f c), then q = J^-T q~
        const int ngrad = 5 * NU + (dev ? 3 * NU : 0);
        for (int it = threadIdx.x; it < ngrad; it += NTH) {
            if (it >= 5 * NU) {   // low-Mach mass channel: (Dh_d m_d)[z]
                const int d = (it - 5 * NU) / NU, z = (it - 5 * NU) % NU;
                const FFOf<OPS> &o = *opsff;
                if constexpr (NU <= 20) {
                    double v = 0.0;
#pragma unroll 5
                    for (int j = 0; j < NU; j++) v += o.Dht64[d][j][z] * s_mfb[d * NU + j];
                    s_rlb[d * NU + z] = v;
                } else {
                    // compensated dot product (Dot2) of the float-float operator row and m_d
                    const ff *m = reinterpret_cast<const ff *>(s_mfb) + d * NU;
                    float sh = 0.0f, c = 0.0f;
#pragma unroll 5
                    for (int j = 0; j < NU; j++) {
                        const float h = o.hi.Dht[d][j][z], l = o.lo.Dht[d][j][z];
                        const ff mj = m[j];
                        const float pr = h * mj.hi;
                        const float er = __fmaf_rn(l, mj.hi, __fmaf_rn(h, mj.lo, __fmaf_rn(h, mj.hi, -pr)));
                        const ff t = two_sum(sh, pr);
                        sh = t.hi;
                        c += t.lo + er;
                    }
                    reinterpret_cast<ff *>(s_rlb)[d * NU + z] = two_sum(sh, c);
                }
                continue;
            }
            const int alpha = it / NU, z = it % NU;
            const T *u = s_u + alpha * NUS;
            const T *c = s_c + alpha * NF;
            T q0 = T(0), q1 = T(0), q2 = T(0);
#pragma unroll 4
            for (int j = 0; j < NU; j++) {
                const T uj = u[j];
                q0 += op->Dht[0][j][z] * uj;
                q1 += op->Dht[1][j][z] * uj;
                q2 += op->Dht[2][j][z] * uj;
            }
#pragma unroll
            for (int f = 0; f < NFACE; f++) {
                T l = T(0);
#pragma unroll
                for (int s = OPS::F0(f); s < OPS::F0(f + 1); s++) l += op->Lt[s][z] * c[s];
                q0 += op->nf[f][0] * l;
                q1 += op->nf[f][1] * l;
                q2 += op->nf[f][2] * l;
            }
#pragma unroll
            for (int k = 0; k < 3; k++) s_q[(alpha * 3 + k) * NUS + z] = g.Ji[k] * q0 + g.Ji[3 + k] * q1 + g.Ji[6 + k] * q2;
        }
        __syncthreads();
        if (dev) {
            const long long pbase = elem_u0(a, e, NU) / FR_NV;
            for (int z = threadIdx.x; z < NU; z += NTH) {
                if constexpr (NU <= 20) {
                    a.RL[pbase + z] = ff_from_double(s_rlb[z] + s_rlb[NU + z] + s_rlb[2 * NU + z]);
                } else {
                    const ff *r = reinterpret_cast<const ff *>(s_rlb);
                    a.RL[pbase + z] = ff_add(ff_add(r[z], r[NU + z]), r[2 * NU + z]);
                }
            }
        }
        // viscous normal flux at own flux points, on the side whose LDG weight 1/2 +- beta is not
        // zero (the other side's is never used); the points are compacted so whole warps work
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
        if constexpr (TCM != 0) {
            // the 20 field rows (s_q follows s_u) for the tensor-core interpolation, four threads per
            // row: [x_hi | x_lo | x_hi], scaled by 2^sh so that the row's largest magnitude lies in
            // [2^14, 2^15); the MMA then runs while the viscous flux below is evaluated
            if (threadIdx.x < 96) {   // warps 0-2, whole warps in the shuffles
                const int r = threadIdx.x >> 2, sub = threadIdx.x & 3;
                const bool row = r < 20;
                constexpr int NV = (NU + 3) / 4;
                float x[NV], mx = 0.f;
#pragma unroll
                for (int i = 0; i < NV; i++) {
                    const int j = sub + 4 * i;
                    x[i] = (row && j < NU) ? (float)s_u[r * NUS + j] : 0.f;
                    mx = fmaxf(mx, fabsf(x[i]));
                }
                mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
                mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
                if (row) {
                    const int sh = tc::row_shift(mx);
                    const float sc = tc::pow2f(sh);
#pragma unroll
                    for (int i = 0; i < NV; i++) {
                        const int j = sub + 4 * i;
                        if (j < NU) {
                            uint16_t pp[3];
                            tc::split_parts<TCM>(x[i] * sc, pp);
#pragma unroll
                            for (int sg = 0; sg < SF::SEGS; sg++)
                                *reinterpret_cast<uint16_t *>(tB + tc::core_offset(r, sg * NU + j, TC::SBO)) = pp[SF::x_part(sg)];
                        }
                    }
                    if (sub == 0) s_sh[r] = sh;
                }
            }
            tc::fence_async_smem();
            tc::fence_before_sync();
        }
        __syncthreads();
        if constexpr (TCM != 0) {
            if (threadIdx.x == 0) {
                tc::fence_after_sync();
                const uint32_t aA = tc::smem_u32(tA), aB = tc::smem_u32(tB);
#pragma unroll
                for (int j = 0; j < TC::KI / 16; j++)
                    tc::mma_f16(tmem, tc::sdesc(aA + 256 * j, 128, TC::SBO), tc::sdesc(aB + 256 * j, 128, TC::SBO),
                                TC::IDESC, j);
                tc::commit(mbar);
            }
        }
        const int nplist = s_pcnt;
        for (int li = threadIdx.x; li < nplist; li += NTH) {
            const int s = s_plist[li];
            T v[20];
#pragma unroll
            for (int f = 0; f < 20; f++) v[f] = T(0);
#pragma unroll 1
            for (int z0 = 0; z0 < NUS; z0 += VW) {
                T m[VW];
#pragma unroll
                for (int k = 0; k < VW; k++) m[k] = op->M0t[z0 + k][s];
#pragma unroll
                for (int f = 0; f < 20; f++) {
                    const V16<T> x = ld16(s_u + f * NUS + z0);
#pragma unroll
                    for (int k = 0; k < VW; k++) v[f] += m[k] * x.v[k];
                }
            }
            T uf[5], qf[5][3];
#pragma unroll
            for (int alpha = 0; alpha < 5; alpha++) {
                uf[alpha] = v[alpha];
#pragma unroll
                for (int d = 0; d < 3; d++) qf[alpha][d] = v[5 + alpha * 3 + d];
            }
            const T *nt = a.fnrm + (e * 6 + OPS::FACE(s)) * 4;
            T n[3] = {nt[0], nt[1], nt[2]};
            if (dev) { uf[0] += ph.rref; uf[4] += ph.eref; }
            T fvn[4];
            viscous_normal_flux(ph, uf, qf, n, fvn);
#pragma unroll
            for (int k = 0; k < 4; k++) a.FV[k * a.nfpt + gf0 + s] = fvn[k];
        }
        if constexpr (TCM != 0) {
            // the interpolation issued above: wait (bounded) and read lane q = this thread
            const bool done = tc::mbar_wait(mbar, parity, tc::first_limit(first_wait, a.dbg_wait0));
            if (!__syncthreads_and(done)) {
                tc_fail = true;
                break;
            }
            parity ^= 1;
            tc::fence_after_sync();
            float v0[16], v1[16];
            const uint32_t ta = tmem + ((uint32_t)(32 * (threadIdx.x >> 5)) << 16);   // lane = quadrature point
            tc::ld16(ta, v0);
            tc::ld16(ta + 16, v1);
            const int q = threadIdx.x;
            if (q < NQ) {
#pragma unroll
                for (int f = 0; f < 16; f++) s_w[f * NQP + q] = v0[f] * tc::pow2f(-s_sh[f]);
#pragma unroll
                for (int f = 16; f < 20; f++) s_w[f * NQP + q] = v1[f - 16] * tc::pow2f(-s_sh[f]);
            }
        } else {
            // interpolation of the 20 fields to the quadrature points: one point per thread
            for (int q = threadIdx.x; q < NQ; q += NTH) {
                T v[20];
#pragma unroll
                for (int f = 0; f < 20; f++) v[f] = T(0);
#pragma unroll 1
                for (int j0 = 0; j0 < NUS; j0 += VW) {
                    T b[VW];
#pragma unroll
                    for (int k = 0; k < VW; k++) b[k] = op->Bt[j0 + k][q];
#pragma unroll
                    for (int f = 0; f < 20; f++) {
                        const V16<T> x = ld16(s_u + f * NUS + j0);
#pragma unroll
                        for (int k = 0; k < VW; k++) v[f] += b[k] * x.v[k];
                    }
                }
#pragma unroll
                for (int f = 0; f < 20; f++) s_w[f * NQP + q] = v[f];
            }
        }
        __syncthreads();
        bool ok = true;
        for (int q = threadIdx.x; q < NQ; q += NTH) {          // tdisf, in place
            T u[5], gq[5][3], f[3][5];
#pragma unroll
            for (int alpha = 0; alpha < 5; alpha++) {
                u[alpha] = s_w[alpha * NQP + q];
#pragma unroll
                for (int d = 0; d < 3; d++) gq[alpha][d] = s_w[(5 + alpha * 3 + d) * NQP + q];
            }
            if (dev) ok &= total_flux_dev(ph, u, gq, f);
            else ok &= total_flux(ph, u, gq, f);
#pragma unroll
            for (int alpha = 0; alpha < 5; alpha++)
#pragma unroll
                for (int d = 0; d < 3; d++)
                    s_w[(alpha * 3 + d) * NQP + q] = g.det * (g.Ji[3 * d] * f[0][alpha] + g.Ji[3 * d + 1] * f[1][alpha] + g.Ji[3 * d + 2] * f[2][alpha]);
        }
        flag_status(a.status, ok);
        __syncthreads();
        // projection with the corrected divergence: R~[alpha][z] = sum_d sum_q Dv_d[z][q] f~_d[alpha][q].
        // Thread (z, chunk c of the NQP/4 groups of 4 quadrature points) sums all 5 variables over its
        // chunk (one operator load per 5 FMAs, the flux values as 16-byte broadcasts); the NCH
        // partial sums are then added in shared memory.
        if (threadIdx.x < NU * NCH) {
            const int z = threadIdx.x % NU, c = threadIdx.x / NU;
            const int gb = c * (NQP / 4) / NCH, ge = (c + 1) * (NQP / 4) / NCH;
            T acc[5] = {T(0), T(0), T(0), T(0), T(0)};
#pragma unroll 1
            for (int d = 0; d < 3; d++)
#pragma unroll 1
                for (int gq4 = gb; gq4 < ge; gq4++) {
                    const int q0 = 4 * gq4;
                    T mv[4];
#pragma unroll
                    for (int k = 0; k < 4; k++) mv[k] = op->Dvt[d][q0 + k][z];
#pragma unroll
                    for (int alpha = 0; alpha < 5; alpha++) {
                        const T *F = s_w + (alpha * 3 + d) * NQP + q0;
#pragma unroll
                        for (int h = 0; h < 4; h += VW) {
                            const V16<T> x = ld16(F + h);
#pragma unroll
                            for (int k = 0; k < VW; k++) acc[alpha] += mv[h + k] * x.v[k];
                        }
                    }
                }
#pragma unroll
            for (int alpha = 0; alpha < 5; alpha++) s_red[(c * 5 + alpha) * NU + z] = acc[alpha];
        }
        __syncthreads();
        T *R = a.R + elem_u0(a, e, NU);
        for (int it = threadIdx.x; it < 5 * NU; it += NTH) {
            T v = T(0);
#pragma unroll
            for (int c = 0; c < NCH; c++) v += s_red[c * 5 * NU + it];
            R[it] = v;
        }
        __syncthreads();
    }
    fr_grid_done();
    if constexpr (TCM != 0) {
        // a chain that did not complete within the bound is reported; the tensor memory is released
        if (tc_fail && threadIdx.x == 0) atomicOr(a.status, 2);
        tc::teardown(mbar, parity, tc_fail, tmem, 32);
    }
}

// -------------------------------------------------------------------------------------------------
// Phase B in FP32 on the CUDA cores: four elements per CTA
// -------------------------------------------------------------------------------------------------
// The dense products re-read their operators per element (the projection alone 30 KB) and were bound by
// the shared-memory and L1 data path (77% busy, FMA pipe 26%). Here an operator entry serves several
// products: the gradient's all five variables, the interpolation's two quadrature points per thread (a
// field value feeds both), and the projection is a register-tiled product, NU x 375 times 375 x (elements
// times variables), a thread holding NU/5 rows by 4 columns of one slice of the quadrature points. The
// interpolated fields stay in registers through the flux.
template <typename OPS>
struct Dense32 {
    static constexpr int EPB = 4, NTH = 128, NUS = OPS::NUS, NF = OPS::NF, NU = OPS::NU;
    static constexpr int ZT = NU / 5;                      // rows of a projection tile
    static constexpr int LOWF = EPB * (20 * NUS + 5 * NF); // state, gradient and common solution; then the partial sums
    static constexpr int SL(int ncol) { return NTH / (5 * (ncol / 4)); }   // slices of the projection's sum
    static_assert(NU % 5 == 0 && ZT % 2 == 0 && SL(16) * 16 * NU <= LOWF && SL(20) * 20 * NU <= LOWF && LOWF % 4 == 0, "tiles");
    static constexpr size_t SMEM = (size_t)(LOWF + 3 * NQ * EPB * 5) * sizeof(float);
};

template <typename OPS>
__global__ void __launch_bounds__(128, OPS::NU <= 20 ? 5 : 4) k_dense_B32(HexArgs<float> a, const OPS *__restrict__ op, const FFOf<OPS> *__restrict__ opsff)
{
    using D = Dense32<OPS>;
    constexpr int NU = OPS::NU, NF = OPS::NF, NFACE = OPS::NFACE, NUS = OPS::NUS, EPB = D::EPB, NTH = D::NTH, ZT = D::ZT;
    extern __shared__ __align__(16) float s_low[];
    float *s_c = s_low + EPB * 20 * NUS;          // [el][5][NF] common solution
    float *s_F = s_low + D::LOWF;                 // [d][q][el][variable] transformed flux
    __shared__ short s_plist[EPB * NF];
    __shared__ int s_pcnt;
    __shared__ __align__(8) double s_mfb[EPB * 3 * NU];   // low-Mach form: transformed mass flux
    __shared__ __align__(8) double s_rlb[EPB * 3 * NU];   // low-Mach form: Dh_d of it, per d
    const int tid = threadIdx.x;
    if (tid == 0) s_pcnt = 0;
    fr_grid_wait();
    const long long ng = (a.ne + EPB - 1) / EPB;
    for (long long grp = blockIdx.x; grp < ng; grp += gridDim.x) {
        const long long e0 = grp * EPB;
        const int nb = (int)(a.ne - e0 < EPB ? a.ne - e0 : EPB);
        {
            bool blk_ok = true;
            for (int k = 0; k < nb; k++) blk_ok = blk_ok && fr_elem_ok(a, e0 + k, NU, NF);
            if (!blk_ok) continue;
        }
        const bool dev = elem_phys(a, e0).dev != 0;   // a handle's instances all carry the low-Mach form or none
        const int nv = dev ? 4 : 5, ncol = EPB * nv;  // low-Mach form: the mass has no flux on this path
        __syncthreads();
        // 1. state (deviations in the low-Mach form), common solution and, in the low-Mach form, the
        //    transformed mass flux (in FP64 on the tetrahedron, where the otherwise idle FP64 pipe does its
        //    products faster; in float-float on the pyramid); the flux points whose side carries LDG weight
        for (int it = tid; it < nb * (NU + NF); it += NTH) {
            const int el = it / (NU + NF), r = it % (NU + NF);
            const Phys<float> ph = elem_phys(a, e0 + el);
            if (r < NU) {
                const float *U = a.U + elem_u0(a, e0 + el, NU) + r;
                float *u = s_low + el * 20 * NUS + r;
                const float m0 = U[NU], m1 = U[2 * NU], m2 = U[3 * NU];
                u[0] = U[0] - (dev ? ph.rref : 0.f);
                u[NUS] = m0; u[2 * NUS] = m1; u[3 * NUS] = m2;
                u[4 * NUS] = U[4 * NU] - (dev ? ph.eref : 0.f);
                if (dev) {
                    const GeoLM &g64 = a.geo64[e0 + el];
#pragma unroll
                    for (int d = 0; d < 3; d++) {
                        if constexpr (NU <= 20) {
                            s_mfb[(el * 3 + d) * NU + r] = g64.det * (g64.Ji[3 * d] * (double)m0 + g64.Ji[3 * d + 1] * (double)m1 + g64.Ji[3 * d + 2] * (double)m2);
                        } else {
                            reinterpret_cast<ff *>(s_mfb)[(el * 3 + d) * NU + r] =
                                ff_add(ff_add(ff_mul_f(g64.cm[3 * d], m0), ff_mul_f(g64.cm[3 * d + 1], m1)), ff_mul_f(g64.cm[3 * d + 2], m2));
                        }
                    }
                }
            } else {
                const int s = r - NU;
                const long long og = elem_f0(a, e0 + el, NF) + s;
                const uint32_t pc = a.partner[og];
                const bool isL = (pc & FR_LFLAG) != 0;
                const long long pg = fr_partner(a, pc, og);
                const float *uL = a.UF + (isL ? og : pg), *uR = a.UF + (isL ? pg : og);
                const float wl = 0.5f - ph.beta, wr = 0.5f + ph.beta;
                float *c = s_c + el * 5 * NF + s;
#pragma unroll
                for (int alpha = 0; alpha < 5; alpha++, uL += a.nfpt, uR += a.nfpt) c[alpha * NF] = wl * *uL + wr * *uR;
                if ((isL ? wr : wl) == 0.f) {
                    float *fv = a.FV + og;
#pragma unroll
                    for (int k = 0; k < 4; k++, fv += a.nfpt) *fv = 0.f;
                } else {
                    s_plist[atomicAdd(&s_pcnt, 1)] = (short)(el * NF + s);
                }
            }
        }
        if constexpr (NUS > NU) {   // the pads meet zero operator rows
            for (int it = tid; it < EPB * 20 * (NUS - NU); it += NTH) s_low[(it / (NUS - NU)) * NUS + NU + it % (NUS - NU)] = 0.f;
        }
        __syncthreads();
        const int nplist = s_pcnt;
        // 2. corrected gradient q~_d = Dh_d u + sum_f n_f,d (L_f c), then q = J^-T q~: one thread per
        //    (element, point), all variables
        for (int it = tid; it < nb * NU; it += NTH) {
            const int el = it / NU, z = it % NU;
            const float *u = s_low + el * 20 * NUS, *c = s_c + el * 5 * NF;
            float q[5][3];
#pragma unroll
            for (int i = 0; i < 15; i++) q[i / 3][i % 3] = 0.f;
#pragma unroll 5
            for (int j = 0; j < NU; j++) {
                const float d0 = op->Dht[0][j][z], d1 = op->Dht[1][j][z], d2 = op->Dht[2][j][z];
#pragma unroll
                for (int alpha = 0; alpha < 5; alpha++) {
                    const float x = u[alpha * NUS + j];
                    q[alpha][0] += d0 * x; q[alpha][1] += d1 * x; q[alpha][2] += d2 * x;
                }
            }
#pragma unroll 1
            for (int f = 0; f < NFACE; f++) {
                float l[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
                const int s1 = OPS::F0(f + 1);
#pragma unroll 5
                for (int s = OPS::F0(f); s < s1; s++) {
                    const float w = op->Lt[s][z];
#pragma unroll
                    for (int alpha = 0; alpha < 5; alpha++) l[alpha] += w * c[alpha * NF + s];
                }
                const float n0 = op->nf[f][0], n1 = op->nf[f][1], n2 = op->nf[f][2];
#pragma unroll
                for (int alpha = 0; alpha < 5; alpha++) { q[alpha][0] += n0 * l[alpha]; q[alpha][1] += n1 * l[alpha]; q[alpha][2] += n2 * l[alpha]; }
            }
            const Geo<float> g = a.geo[e0 + el];
            float *o = s_low + el * 20 * NUS + 5 * NUS + z;
#pragma unroll
            for (int alpha = 0; alpha < 5; alpha++)
#pragma unroll
                for (int k = 0; k < 3; k++) o[(alpha * 3 + k) * NUS] = g.Ji[k] * q[alpha][0] + g.Ji[3 + k] * q[alpha][1] + g.Ji[6 + k] * q[alpha][2];
        }
        // 3. low-Mach form: (Dh_d m_d)[z], the volume part of R~_rho (rho v lies in the solution space, so
        //    its L2 projection is itself and the corrected divergence applies at the solution points); from
        //    the upper threads down
        if (dev) {
            for (int it = NTH - 1 - tid; it < nb * 3 * NU; it += NTH) {
                const int el = it / (3 * NU), d = (it / NU) % 3, z = it % NU;
                const FFOf<OPS> &o = *opsff;
                if constexpr (NU <= 20) {
                    const double *m = s_mfb + (el * 3 + d) * NU;
                    double v = 0.0;
#pragma unroll 5
                    for (int j = 0; j < NU; j++) v += o.Dht64[d][j][z] * m[j];
                    s_rlb[it] = v;
                } else {
                    // compensated dot product (Dot2) of the float-float operator row and m_d
                    const ff *m = reinterpret_cast<const ff *>(s_mfb) + (el * 3 + d) * NU;
                    float sh = 0.0f, c = 0.0f;
#pragma unroll 5
                    for (int j = 0; j < NU; j++) dot2ff_next(ff{o.hi.Dht[d][j][z], o.lo.Dht[d][j][z]}, m[j], sh, c);
                    reinterpret_cast<ff *>(s_rlb)[it] = two_sum(sh, c);
                }
            }
        }
        __syncthreads();
        if (dev) {
            for (int it = NTH - 1 - tid; it < nb * NU; it += NTH) {
                const int el = it / NU, z = it % NU;
                const long long pbase = elem_u0(a, e0 + el, NU) / FR_NV;
                if constexpr (NU <= 20) {
                    const double *r = s_rlb + el * 3 * NU + z;
                    a.RL[pbase + z] = ff_from_double(r[0] + r[NU] + r[2 * NU]);
                } else {
                    const ff *r = reinterpret_cast<const ff *>(s_rlb) + el * 3 * NU + z;
                    a.RL[pbase + z] = ff_add(ff_add(r[0], r[NU]), r[2 * NU]);
                }
            }
        }
        // 4. own-normal viscous flux at the listed flux points
        for (int li = tid; li < nplist; li += NTH) {
            const int el = s_plist[li] / NF, s = s_plist[li] % NF;
            const float *x = s_low + el * 20 * NUS;
            float v[20];
#pragma unroll
            for (int f = 0; f < 20; f++) v[f] = 0.f;
            float mn[4];   // (fetched a step ahead)
#pragma unroll
            for (int k = 0; k < 4; k++) mn[k] = op->M0t[k][s];
#pragma unroll 1
            for (int z0 = 0; z0 < NUS; z0 += 4) {
                float m[4];
#pragma unroll
                for (int k = 0; k < 4; k++) m[k] = mn[k];
                if (z0 + 4 < NUS) {
#pragma unroll
                    for (int k = 0; k < 4; k++) mn[k] = op->M0t[z0 + 4 + k][s];
                }
#pragma unroll
                for (int f = 0; f < 20; f++) {
                    const float4 y = *reinterpret_cast<const float4 *>(x + f * NUS + z0);
                    v[f] += m[0] * y.x; v[f] += m[1] * y.y; v[f] += m[2] * y.z; v[f] += m[3] * y.w;
                }
            }
            float uf[5], qf[5][3];
#pragma unroll
            for (int alpha = 0; alpha < 5; alpha++) {
                uf[alpha] = v[alpha];
#pragma unroll
                for (int d = 0; d < 3; d++) qf[alpha][d] = v[5 + alpha * 3 + d];
            }
            const Phys<float> ph = elem_phys(a, e0 + el);
            const float *nt = a.fnrm + ((e0 + el) * 6 + OPS::FACE(s)) * 4;
            const float n[3] = {nt[0], nt[1], nt[2]};
            if (dev) { uf[0] += ph.rref; uf[4] += ph.eref; }
            float fvn[4];
            viscous_normal_flux(ph, uf, qf, n, fvn);
            float *fv = a.FV + elem_f0(a, e0 + el, NF) + s;
#pragma unroll
            for (int k = 0; k < 4; k++, fv += a.nfpt) *fv = fvn[k];
        }
        // 5. interpolation of the 20 fields to two quadrature points, q and q + H, and the flux there
        constexpr int H = (NQ + 1) / 2;
        bool ok = true;
        for (int it = tid; it < nb * H; it += NTH) {
            const int el = it / H, q = it % H;
            const bool two = q + H < NQ;
            const float *x = s_low + el * 20 * NUS;
            float v[2][20];
#pragma unroll
            for (int f = 0; f < 20; f++) v[0][f] = v[1][f] = 0.f;
            // (operator entries fetched a step ahead)
            float n0[4], n1[4];
            const int q1 = two ? q + H : q;
#pragma unroll
            for (int k = 0; k < 4; k++) { n0[k] = op->Bt[k][q]; n1[k] = op->Bt[k][q1]; }
#pragma unroll 1
            for (int j0 = 0; j0 < NUS; j0 += 4) {
                float b0[4], b1[4];
#pragma unroll
                for (int k = 0; k < 4; k++) { b0[k] = n0[k]; b1[k] = n1[k]; }
                if (j0 + 4 < NUS) {
#pragma unroll
                    for (int k = 0; k < 4; k++) { n0[k] = op->Bt[j0 + 4 + k][q]; n1[k] = op->Bt[j0 + 4 + k][q1]; }
                }
#pragma unroll
                for (int f = 0; f < 20; f++) {
                    const float4 y = *reinterpret_cast<const float4 *>(x + f * NUS + j0);
                    v[0][f] += b0[0] * y.x; v[0][f] += b0[1] * y.y; v[0][f] += b0[2] * y.z; v[0][f] += b0[3] * y.w;
                    v[1][f] += b1[0] * y.x; v[1][f] += b1[1] * y.y; v[1][f] += b1[2] * y.z; v[1][f] += b1[3] * y.w;
                }
            }
            const Phys<float> ph = elem_phys(a, e0 + el);
            const Geo<float> g = a.geo[e0 + el];
#pragma unroll
            for (int p = 0; p < 2; p++) {
                if (p == 1 && !two) break;
                float u[5], gq[5][3], f[3][5];
#pragma unroll
                for (int alpha = 0; alpha < 5; alpha++) {
                    u[alpha] = v[p][alpha];
#pragma unroll
                    for (int d = 0; d < 3; d++) gq[alpha][d] = v[p][5 + alpha * 3 + d];
                }
                if (dev) ok &= total_flux_dev(ph, u, gq, f);
                else ok &= total_flux(ph, u, gq, f);
#pragma unroll
                for (int d = 0; d < 3; d++) {
                    const float c0 = g.det * g.Ji[3 * d], c1 = g.det * g.Ji[3 * d + 1], c2 = g.det * g.Ji[3 * d + 2];
                    float *F = s_F + (d * NQ + q + p * H) * ncol + el * nv;
                    float t[5];
#pragma unroll
                    for (int alpha = 0; alpha < 5; alpha++) t[alpha] = c0 * f[0][alpha] + c1 * f[1][alpha] + c2 * f[2][alpha];
                    if (dev) *reinterpret_cast<float4 *>(F) = make_float4(t[1], t[2], t[3], t[4]);
                    else {
#pragma unroll
                        for (int alpha = 0; alpha < 5; alpha++) F[alpha] = t[alpha];
                    }
                }
            }
        }
        flag_status(a.status, ok);
        __syncthreads();
        // 6. projection with the corrected divergence, R~[z][column] = sum_k Dv[z][k] F[k][column], k = (d, q):
        //    thread (slice of k, row group of ZT, column group of 4)
        {
            const int ncg = ncol / 4, per = 5 * ncg, nsl = NTH / per;
            const int sl = tid / per, zg = (tid % per) / ncg, cg = tid % ncg;
            float acc[ZT][4];
#pragma unroll
            for (int i = 0; i < ZT; i++)
#pragma unroll
                for (int j = 0; j < 4; j++) acc[i][j] = 0.f;
            if (sl < nsl) {
#pragma unroll 1
                for (int d = 0; d < 3; d++) {
                    const int qb = sl * NQ / nsl, qe = (sl + 1) * NQ / nsl;
                    const float *w = &op->Dvt[d][qb][zg * ZT];
                    const float *F = s_F + (d * NQ + qb) * ncol + 4 * cg;
#pragma unroll 4
                    for (int q = qb; q < qe; q++, w += NU, F += ncol) {
                        float m[ZT];
#pragma unroll
                        for (int i = 0; i < ZT; i += 2) {
                            const float2 y = *reinterpret_cast<const float2 *>(w + i);
                            m[i] = y.x; m[i + 1] = y.y;
                        }
                        const float4 x = *reinterpret_cast<const float4 *>(F);
#pragma unroll
                        for (int i = 0; i < ZT; i++) { acc[i][0] += m[i] * x.x; acc[i][1] += m[i] * x.y; acc[i][2] += m[i] * x.z; acc[i][3] += m[i] * x.w; }
                    }
                }
                // partial sums [slice][row][column] over the consumed state, gradient and common solution
                float *o = s_low + (sl * NU + zg * ZT) * ncol + 4 * cg;
#pragma unroll
                for (int i = 0; i < ZT; i++) *reinterpret_cast<float4 *>(o + i * ncol) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
            }
            if (tid == 0) s_pcnt = 0;
            __syncthreads();
            for (int it = tid; it < nb * nv * NU; it += NTH) {
                const int el = it / (nv * NU), r = it % (nv * NU), al = r / NU, z = r % NU;
                const float *p = s_low + z * ncol + el * nv + al;
                float v = 0.f;
                for (int k = 0; k < nsl; k++) v += p[k * NU * ncol];
                a.R[elem_u0(a, e0 + el, NU) + (al + 5 - nv) * NU + z] = v;
            }
        }
    }
    fr_grid_done();
}

// -------------------------------------------------------------------------------------------------
// Phase B in FP64: the dense operators in block fixed point (fr_fx.cuh), one element per CTA
// -------------------------------------------------------------------------------------------------
// A dense element's operators are 0.85 (tetrahedron) to 0.9 (pyramid) of its FP64 arithmetic, which
// bounds the kernel; on the integer multipliers they run beside the pointwise fluxes that stay on the
// FP64 pipe. Blocks: each variable with its common solution; the three transformed flux components of
// a variable, which the projection adds up. The quadrature-point fields never leave the registers: a
// thread interpolates the 20 fields to its point, evaluates the flux there and keeps the 15 transformed
// components until the CTA knows their largest magnitudes. Measured, 12^3 Kuhn box (10,368 tetrahedra): 2.53 -> 0.79 ms.
template <typename OPS, int NTH>
__global__ void __launch_bounds__(NTH, 4) k_dense_B_fx(HexArgs<double> a, const OPS *__restrict__ ops)
{
    constexpr int NU = OPS::NU, NF = OPS::NF, NFACE = OPS::NFACE, NUS = OPS::NUS;
    constexpr int NCH = NTH / NU;                 // quadrature-point chunks of the projection
    static_assert(NTH == 128 && NU + NF <= NTH, "one thread per quadrature point, state and flux point");
    static_assert((3 * NQP + NCH - 1) / NCH + 6 <= 128 && NQP % 2 == 0 && NUS % 2 == 0, "terms of one 64-bit projection sum");
    const auto &op = ops->fx;
    __shared__ __align__(16) fx2 s_u[20 * NUS];          // state, then the physical gradient (5 + 3 alpha + d)
    __shared__ fx2 s_c[5 * NF];                          // common solution
    __shared__ __align__(16) fx2 s_w[15 * NQP];          // transformed flux; before it, the traces (FP64)
    __shared__ long long s_red[NCH * 5 * NU];            // projection partial sums
    __shared__ short s_plist[NF];
    __shared__ int s_pcnt, s_mx[10];
    double *s_tr = reinterpret_cast<double *>(s_w);      // [listed flux point][20]
    static_assert(NF * 20 <= 15 * NQP, "traces over the flux");
    const int tid = threadIdx.x;
    const bool lane0 = (tid & 31) == 0;
    if constexpr (NUS > NU)   // the pads meet zero operator rows
        for (int it = tid; it < 20 * (NUS - NU); it += NTH) s_u[(it / (NUS - NU)) * NUS + NU + it % (NUS - NU)] = fx2{0, 0};
    if (tid < 10) s_mx[tid] = 0;
    if (tid == 0) s_pcnt = 0;
    __syncthreads();
    fr_grid_wait();
    for (long long e = blockIdx.x; e < a.ne; e += gridDim.x) {
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
            for (int alpha = 0; alpha < 5; alpha++) s_u[alpha * NUS + tid] = fx_from<FX_WS>(val[alpha], E[alpha]);
        } else if (tid < NU + NF) {
#pragma unroll
            for (int alpha = 0; alpha < 5; alpha++) s_c[alpha * NF + tid - NU] = fx_from<FX_WS>(val[alpha], E[alpha]);
        }
        __syncthreads();
        const int nplist = s_pcnt;
        // 2. corrected gradient q~_d = Dh_d u + sum_f n_f,d (L_f c), then q = J^-T q~
        int EJ[3], qe[3];   // gradient component k: value = X 2^(E - 1078 - FX_WS + qe[k])
#pragma unroll
        for (int k = 0; k < 3; k++) {
            EJ[k] = fx_column_exp(g.Ji, k);
            qe[k] = op.kD + EJ[k] - 1022;
        }
        for (int it = tid; it < 5 * NU; it += NTH) {
            const int alpha = it / NU, z = it % NU;
            const fx2 *u = s_u + alpha * NUS, *c = s_c + alpha * NF;
            fxacc q[3] = {{FX_HALF, 0}, {FX_HALF, 0}, {FX_HALF, 0}};
#pragma unroll 4
            for (int j = 0; j < NU; j++) {
                const fx2 uj = u[j];
#pragma unroll
                for (int d = 0; d < 3; d++) fx_mac(q[d], op.Dht[d][j][z], uj);
            }
#pragma unroll 1
            for (int f = 0; f < NFACE; f++) {
                fxacc l{FX_HALF, 0};
                const int s1 = OPS::F0(f + 1);
#pragma unroll 2
                for (int s = OPS::F0(f); s < s1; s++) fx_mac(l, op.Lt[s][z], c[s]);
                const fx2 lf = fx_limbs(fx_sum(l));
#pragma unroll
                for (int d = 0; d < 3; d++) fx_mac(q[d], op.nf[f][d], lf);
            }
            fx2 qr[3];
#pragma unroll
            for (int d = 0; d < 3; d++) qr[d] = fx_limbs(fx_sum(q[d]));
#pragma unroll
            for (int k = 0; k < 3; k++) {
                fxacc s{FX_HALF, 0};
#pragma unroll
                for (int d = 0; d < 3; d++) fx_mac(s, fx_factor(g.Ji[3 * d + k], EJ[k]), qr[d]);
                s_u[(5 + alpha * 3 + k) * NUS + z] = fx_limbs(fx_sum(s));
            }
        }
        __syncthreads();
        // 3. traces of the 20 fields at the listed flux points, four threads per point
        for (int it = tid; it < 4 * nplist; it += NTH) {
            const int li = it >> 2, fg = it & 3, s = s_plist[li];
            fxacc t[5] = {{0, 0}, {0, 0}, {0, 0}, {0, 0}, {0, 0}};
#pragma unroll 2
            for (int z = 0; z < NU; z++) {
                const fx2 m = op.M0t[z][s];
#pragma unroll
                for (int k = 0; k < 5; k++) fx_mac(t[k], m, s_u[(5 * fg + k) * NUS + z]);
            }
#pragma unroll
            for (int k = 0; k < 5; k++) {
                const int f = 5 * fg + k, Ea = s_mx[f < 5 ? f : (f - 5) / 3];
                s_tr[li * 20 + f] = fx_double(fx_sum(t[k]), Ea - 1080 - FX_WS + op.kM + fx_field_exp(f, qe), Ea >= 2047);
            }
        }
        // 4. interpolation to this thread's quadrature point and the flux there
        bool ok = true;
        double f[3][5];
        int fm[5] = {0, 0, 0, 0, 0};
        if (tid < NQ) {
            fxacc t[20];
#pragma unroll
            for (int i = 0; i < 20; i++) t[i] = fxacc{0, 0};
            // two solution points per step (16-byte loads of a field's values), their operator entries
            // fetched a step ahead
            fx2 n0 = op.Bt[0][tid], n1 = op.Bt[1][tid];
#pragma unroll 1
            for (int j = 0; j < NUS; j += 2) {
                const fx2 b0 = n0, b1 = n1;
                if (j + 2 < NUS) { n0 = op.Bt[j + 2][tid]; n1 = op.Bt[j + 3][tid]; }   // (pad rows are zero)
#pragma unroll
                for (int i = 0; i < 20; i++) {
                    const int4 y = *reinterpret_cast<const int4 *>(s_u + i * NUS + j);
                    fx_mac(t[i], b0, fx2{y.x, y.y});
                    fx_mac(t[i], b1, fx2{y.z, y.w});
                }
            }
            double u[5], gq[5][3];
#pragma unroll
            for (int alpha = 0; alpha < 5; alpha++) {
                const int ex = E[alpha] - 1080 - FX_WS + op.kB;
                u[alpha] = fx_double(fx_sum(t[alpha]), ex, E[alpha] >= 2047);
#pragma unroll
                for (int d = 0; d < 3; d++) gq[alpha][d] = fx_double(fx_sum(t[5 + alpha * 3 + d]), ex + qe[d], E[alpha] >= 2047);
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
        } else {
#pragma unroll
            for (int c = 0; c < 15; c++) f[c % 3][c / 3] = 0.0;   // the pad rows meet zero operator rows
        }
        flag_status(a.status, ok);
#pragma unroll
        for (int alpha = 0; alpha < 5; alpha++) {
            const int m = (int)__reduce_max_sync(0xffffffffu, (unsigned)fm[alpha]);
            if (lane0) atomicMax(&s_mx[5 + alpha], m >> 20);
        }
        __syncthreads();
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
            const double *nt = a.fnrm + (e * 6 + OPS::FACE(s)) * 4;
            const double n[3] = {nt[0], nt[1], nt[2]};
            double fvn[4];
            viscous_normal_flux(ph, uf, qf, n, fvn);
#pragma unroll
            for (int k = 0; k < 4; k++) a.FV[k * a.nfpt + gf0 + s] = fvn[k];
        }
        __syncthreads();
        // 6. the flux in fixed point
#pragma unroll
        for (int alpha = 0; alpha < 5; alpha++) {
            const int Ef = s_mx[5 + alpha];
#pragma unroll
            for (int d = 0; d < 3; d++) s_w[(alpha * 3 + d) * NQP + tid] = fx_from(f[d][alpha], Ef);
        }
        __syncthreads();
        // 7. projection with the corrected divergence: R~[alpha][z] = sum_d sum_q Dv_d[z][q] f~_d[alpha][q],
        //    thread (z, chunk) over its quadrature points, all variables; then the chunks' sums
        if (tid < NU * NCH) {
            const int z = tid % NU, c = tid / NU;
            const int qb = c * (NQP / 2) / NCH * 2, qn = (c + 1) * (NQP / 2) / NCH * 2;
            fxacc acc[5] = {{0, 0}, {0, 0}, {0, 0}, {0, 0}, {0, 0}};
#pragma unroll 1
            for (int d = 0; d < 3; d++)
#pragma unroll 2
                for (int q = qb; q < qn; q += 2) {
                    const fx2 m0 = op.Dvt[d][q][z], m1 = op.Dvt[d][q + 1][z];
#pragma unroll
                    for (int alpha = 0; alpha < 5; alpha++) {
                        const int4 y = *reinterpret_cast<const int4 *>(s_w + (alpha * 3 + d) * NQP + q);
                        fx_mac(acc[alpha], m0, fx2{y.x, y.y});
                        fx_mac(acc[alpha], m1, fx2{y.z, y.w});
                    }
                }
#pragma unroll
            for (int alpha = 0; alpha < 5; alpha++) s_red[(c * 5 + alpha) * NU + z] = fx_sum(acc[alpha]);
        }
        __syncthreads();
        double *R = a.R + elem_u0(a, e, NU);
        for (int it = tid; it < 5 * NU; it += NTH) {
            long long y = 0;
#pragma unroll
            for (int c = 0; c < NCH; c++) y += s_red[c * 5 * NU + it];
            const int Ef = s_mx[5 + it / NU];
            R[it] = fx_double(y, Ef - 1080 + op.kV, Ef >= 2047);
        }
        __syncthreads();
        if (tid < 10) s_mx[tid] = 0;
        if (tid == 0) s_pcnt = 0;
        __syncthreads();
    }
    fr_grid_done();
}

// -------------------------------------------------------------------------------------------------
// Phase C: interface group (common flux at every own flux point, lift and scale)
// -------------------------------------------------------------------------------------------------
// FP32: registers capped for 1280 resident threads per SM (eight tetrahedral or five pyramidal CTAs):
// the kernel waits on its partner gathers, and more warps keep more of them in flight.
template <typename T, typename OPS, int EPB>
__global__ void __launch_bounds__(OPS::NF * EPB, sizeof(T) == 4 ? 1280 / (OPS::NF * EPB) : 0) k_dense_C(HexArgs<T> a, const OPS *__restrict__ op, const FFOf<OPS> *__restrict__ opsff)
{
    constexpr int NU = OPS::NU, NF = OPS::NF, NTH = NF * EPB;
    constexpr bool F32 = sizeof(T) == 4;
    constexpr int VN = V16<T>::n;
    static_assert(NF % VN == 0 && NF % 2 == 0 && NTH % 32 == 0, "flux-point rows are whole 16-byte vectors; whole warps");
    __shared__ __align__(16) T s_d[F32 ? EPB : 1][F32 ? FR_NV * NF : 1];
    // FP64: the lift in block fixed point (fr_fx.cuh)
    __shared__ __align__(16) fx2 s_dx[F32 ? 1 : EPB][F32 ? 2 : FR_NV * NF];
    __shared__ int s_mx[F32 ? 1 : EPB][FR_NV];
    __shared__ ff s_dff[F32 ? EPB : 1][F32 ? NF : 1];    // low-Mach form: scaled common mass flux (float-float)
    __shared__ ff s_rr[F32 ? EPB : 1][F32 ? NU : 1];     // low-Mach form: R_rho (float-float)
    __shared__ ff s_idet[F32 ? EPB : 1];                 // low-Mach form: -1 / det J (float-float)
    const int el = threadIdx.x / NF, s = threadIdx.x % NF;
    fr_grid_wait();
    const long long ng = (a.ne + EPB - 1) / EPB;
    for (long long g = blockIdx.x; g < ng; g += gridDim.x) {
        const long long e0 = g * EPB;
        const int nel = (int)(a.ne - e0 < EPB ? a.ne - e0 : EPB);
        {
            bool blk_ok = true;
            for (int k = 0; k < nel; k++) blk_ok = blk_ok && fr_elem_ok(a, e0 + k, NU, NF);
            if (!blk_ok) continue;
        }
        if constexpr (!F32) {
            for (int i = threadIdx.x; i < EPB * FR_NV; i += NTH) s_mx[i / FR_NV][i % FR_NV] = 0;
            __syncthreads();
        }
        T dv[5] = {T(0), T(0), T(0), T(0), T(0)};
        bool ok = true;
        if (el < nel) {
            const long long e = e0 + el;
            const Phys<T> ph = elem_phys(a, e);
            const long long og = elem_f0(a, e, NF) + s;
            const uint32_t pc = a.partner[og];
            const bool isL = (pc & FR_LFLAG) != 0;
            const long long pg = fr_partner(a, pc, og);
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
            const T *nt = a.fnrm + (e * 6 + OPS::FACE(s)) * 4;
            const T mag = nt[3];
            const T nL[3] = {isL ? nt[0] : -nt[0], isL ? nt[1] : -nt[1], isL ? nt[2] : -nt[2]};
            T F[5];
            bool dev = false;
            if constexpr (F32) dev = ph.dev != 0;
            if (dev) {
                if constexpr (F32) {
                    float sw;
                    ok = common_flux_dev(ph, uL, uR, fvL, fvR, nL, F, sw);
                    // mass flux in float-float: 1/2 (mL - mR) + (s/2 + tau)(rho_L - rho_R), mX = own-normal n.(rho v)
                    const ff mo = a.MF[og], mp = a.MF[pg];
                    const ff mL = isL ? mo : mp, mR = isL ? mp : mo;
                    const ff Fr = ff_add(ff_mul_f(ff_sub(mL, mR), 0.5f), ff_mul_f(two_sum(uL[0], -uR[0]), 0.5f * sw + ph.tau));
                    const ff magf = a.fnrm64[(e * 6 + OPS::FACE(s)) * 4 + 3], Dr = ff_mul(magf, Fr);
                    s_dff[el][s] = isL ? Dr : ff_neg(Dr);
                    if (s == 0) s_idet[el] = a.geo64[e].idet;
                }
            } else {
                ok = common_flux(ph, uL, uR, fvL, fvR, nL, F);
            }
            const T sc = isL ? mag : -mag;
#pragma unroll
            for (int k = 0; k < 5; k++) {
                if constexpr (F32) s_d[el][k * NF + s] = sc * F[k];
                else dv[k] = sc * F[k];
            }
        }
        flag_status(a.status, ok);
        if constexpr (!F32) {
            // each variable of each element scaled by its largest magnitude (a warp holds points of up to
            // two elements)
            const unsigned mask = __match_any_sync(0xffffffffu, el);
#pragma unroll
            for (int k = 0; k < 5; k++) {
                const int m = (int)__reduce_max_sync(mask, (unsigned)fx_mag(dv[k])) >> 20;
                if ((threadIdx.x & 31) == __ffs(mask) - 1) atomicMax(&s_mx[el][k], m);
            }
            __syncthreads();
#pragma unroll
            for (int k = 0; k < 5; k++) s_dx[el][k * NF + s] = fx_from(dv[k], s_mx[el][k]);
        }
        __syncthreads();
        if constexpr (!F32) {
            const auto &fx = op->fx;
            const int kD = fx.kD;
            for (int i = threadIdx.x; i < nel * FR_NV * NU; i += NTH) {
                const int l = i / (FR_NV * NU), alpha = (i / NU) % FR_NV, z = i % NU, E = s_mx[l][alpha];
                const long long ui = elem_u0(a, e0 + l, NU) + alpha * NU + z;
                const fx2 *D = s_dx[l] + alpha * NF;
                fxacc t{0, 0};
#pragma unroll 4
                for (int s2 = 0; s2 < NF; s2 += 2) {
                    const int4 y = *reinterpret_cast<const int4 *>(D + s2);
                    fx_mac(t, fx.Lt[s2][z], fx2{y.x, y.y});
                    fx_mac(t, fx.Lt[s2 + 1][z], fx2{y.z, y.w});
                }
                const double v = (a.R[ui] + fx_double(fx_sum(t), E - 1080 + kD, E >= 2047)) * a.geo[e0 + l].nidet;
                if (a.rkstage == 0) a.R[ui] = v;
                else rk_fold(a, ui, v);
            }
        } else {
            // lift and scale: R += L D, R *= -1/det; the mass rows of low-Mach elements in float-float,
            // then the energy rows, which add H0 R_rho
            for (int pass = 0; pass < 2; pass++) {
                const int nrow = pass == 0 ? 4 : 1;
                for (int i = threadIdx.x; i < nel * nrow * NU; i += NTH) {
                    const int l = i / (nrow * NU), alpha = pass == 0 ? (i / NU) % 4 : 4, z = i % NU;
                    const long long e = e0 + l;
                    const long long ui = elem_u0(a, e, NU) + alpha * NU + z;
                    const bool dev = elem_phys(a, e).dev != 0;
                    float outf = 0.0f;
                    T out;
                    if (dev && alpha == 0) {
                        if constexpr (F32) {
                            const ff r0 = a.RL[elem_u0(a, e, NU) / FR_NV + z];
                            float sh = r0.hi, c = r0.lo;
                            const ff *d = s_dff[l];
#pragma unroll 8
                            for (int s2 = 0; s2 < NF; s2++) {
                                const float lh = op->Lt[s2][z], ll = opsff->lo.Lt[s2][z];
                                const ff ds = d[s2];
                                const float pr = lh * ds.hi;
                                const float er = __fmaf_rn(ll, ds.hi, __fmaf_rn(lh, ds.lo, __fmaf_rn(lh, ds.hi, -pr)));
                                const ff t = two_sum(sh, pr);
                                sh = t.hi;
                                c += t.lo + er;
                            }
                            const ff Rrho = ff_mul(two_sum(sh, c), s_idet[l]);
                            s_rr[l][z] = Rrho;
                            outf = Rrho.hi + Rrho.lo;
                        }
                        out = (T)outf;
                    } else {
                        const T *D = s_d[l] + alpha * NF;
                        T v = a.R[ui];
#pragma unroll 2
                        for (int s2 = 0; s2 < NF; s2 += VN) {
                            const V16<T> x = ld16(D + s2);
#pragma unroll
                            for (int j = 0; j < VN; j++) v += op->Lt[s2 + j][z] * x.v[j];
                        }
                        out = v * a.geo[e].nidet;
                        if constexpr (F32) {
                            if (dev && alpha == 4) {
                                const ff e4 = ff_fma(elem_phys(a, e).H0ff, s_rr[l][z], ff_of(out));
                                out = e4.hi + e4.lo;
                            }
                        }
                    }
                    if (a.rkstage == 0) a.R[ui] = out;
                    else rk_fold(a, ui, out);
                }
                if (pass == 0) __syncthreads();
            }
        }
        __syncthreads();
    }
    fr_grid_done();
}

// persistent grid over groups of epb elements: at most per_sm CTAs per SM, 8 waves
int grid_groups(long long ne, int epb, int per_sm)
{
    long long g = (ne + epb - 1) / epb;
    if (g > fr_sms() * per_sm * 8) g = fr_sms() * per_sm * 8;
    return (int)(g < 1 ? 1 : g);
}

int grid_elems(long long ne, int per_sm)
{
    long long g = ne;
    if (g > fr_sms() * per_sm * 8) g = fr_sms() * per_sm * 8;
    return (int)(g < 1 ? 1 : g);
}

template <typename T, typename OPS>
int dense_phase(int phase, const HexArgs<T> &a, const OPS *ops, const FFOf<OPS> *opsff, cudaStream_t s)
{
    constexpr int NU = OPS::NU, NF = OPS::NF, NUS = OPS::NUS;
    if (a.ne == 0) return 0;
    if (phase == 0) {
        if constexpr (sizeof(T) == 8) fr_launch(k_dense_disu_fx<OPS, 4>, grid_groups(a.ne, 4, 8), NF * 4, 0, s, a, ops);
        else fr_launch(k_dense_disu<OPS, 4>, grid_groups(a.ne, 4, 8), NF * 4, 0, s, a, ops, opsff);
    } else if (phase == 1) {
        constexpr int NTH = 128;
        const size_t base = (size_t)(20 * NUS + 5 * NF + 20 * NQP) * sizeof(T);
        bool tcdone = false;
        if constexpr (sizeof(T) == 4) {
            if (a.tcmode != 0) {
                tcdone = true;
                const size_t smem = base + (a.tcmode == 1 ? DenseTC<OPS, 1>::BYTES : DenseTC<OPS, 2>::BYTES);
                // persistent: as many CTAs as fit on the SMs (shared memory, registers, and the 512
                // tensor-memory columns at 32 per CTA)
                auto kern = a.tcmode == 1 ? k_dense_B<NTH, OPS, 1> : k_dense_B<NTH, OPS, 2>;
                static SmemOptIn optin[3];
                optin[a.tcmode](kern, smem);
                static int occ[3] = {-1, -1, -1};
                int &o = occ[a.tcmode];
                if (o < 0) {
                    cudaFuncAttributes fa{};
                    if (cudaFuncGetAttributes(&fa, kern) != cudaSuccess) return -1;
                    const int by_smem = (int)(232448 / (smem + fa.sharedSizeBytes + 1024));
                    const int by_regs = 65536 / (((fa.numRegs + 7) / 8 * 8) * NTH);
                    int v = by_smem < by_regs ? by_smem : by_regs;
                    if (v > 512 / 32) v = 512 / 32;
                    if (v < 1) return -4;
                    o = v;
                }
                const long long g = a.ne < fr_sms() * o ? a.ne : fr_sms() * o;
                kern<<<(int)g, NTH, smem, s>>>(a, ops, opsff);
            }
        }
        if constexpr (sizeof(T) == 8) {
            fr_launch(k_dense_B_fx<OPS, NTH>, grid_elems(a.ne, 4), NTH, 0, s, a, ops);
        } else if (!tcdone && a.ne < 8 * fr_sms()) {
            // fewer elements than resident CTAs of one element: a small handle waits for one element's chain
            // (B at 750 elements, below the line: tetrahedra 20.2 against 27.1 us with four per CTA, pyramids 26.4
            // against 36.7; at 1,296, above it: 34.8 against 30.9 and 47.3 against 42.9)
            static SmemOptIn optin;
            optin(k_dense_B<NTH, OPS, 0>, base);
            fr_launch(k_dense_B<NTH, OPS, 0>, grid_elems(a.ne, 8), NTH, base, s, a, ops, opsff);
        } else if (!tcdone) {
            using D = Dense32<OPS>;
            static SmemOptIn optin;
            optin(k_dense_B32<OPS>, D::SMEM);
            fr_launch(k_dense_B32<OPS>, grid_groups(a.ne, D::EPB, 5), D::NTH, D::SMEM, s, a, ops, opsff);
        }
    } else {
        fr_launch(k_dense_C<T, OPS, 4>, grid_groups(a.ne, 4, 8), NF * 4, 0, s, a, ops, opsff);
    }
    (void)NU;
    return cudaPeekAtLastError() == cudaSuccess ? 0 : -1;
}

}  // namespace

template <typename T>
int tet_fused_phase(int phase, const HexArgs<T> &a, const TetOps<T> *ops, const DenseOpsFF<TetOps<float>> *opsff, cudaStream_t s)
{
    return dense_phase<T, TetOps<T>>(phase, a, ops, opsff, s);
}

template <typename T>
int pyr_fused_phase(int phase, const HexArgs<T> &a, const PyrOps<T> *ops, const DenseOpsFF<PyrOps<float>> *opsff, cudaStream_t s)
{
    return dense_phase<T, PyrOps<T>>(phase, a, ops, opsff, s);
}

template int tet_fused_phase<double>(int, const HexArgs<double> &, const TetOps<double> *, const DenseOpsFF<TetOps<float>> *, cudaStream_t);
template int tet_fused_phase<float>(int, const HexArgs<float> &, const TetOps<float> *, const DenseOpsFF<TetOps<float>> *, cudaStream_t);
template int pyr_fused_phase<double>(int, const HexArgs<double> &, const PyrOps<double> *, const DenseOpsFF<PyrOps<float>> *, cudaStream_t);
template int pyr_fused_phase<float>(int, const HexArgs<float> &, const PyrOps<float> *, const DenseOpsFF<PyrOps<float>> *, cudaStream_t);
