// The per-reaction stored linearization on fixed-point logarithms (nk_fx.cuh, nk_fxpt.cuh, nk_fxd.cuh;
// included by k_linc.cu, whose slots it writes) and its product pass with the rates kernel's chunks.
//
// The pair kernels spent their FP64 pipe on ln C sums, exponentials and the accumulation of every
// reaction into shared rows between block barriers.  Here the linearization takes its terms and
// their temperature derivatives from integers, and both passes gather species sums per chunk; the
// FP64 pipe bounds the product pass (77% busy: the terms nu (q_f, q_r) and their relative
// derivatives are products in doubles).  FP64 helpers of the rare cases (nu other than 1, falloff)
// stay out of line: as predicated instructions they cost the pipe as much as executed ones.
// One linearization with its sources and the products of a linearly implicit stage, 53 species,
// 262,144 points: 37.1 -> 30.1 ms for the stage (at 2,097,152 points the linearization 53.6 ->
// 27.7 ms, a product 24.0 -> 20.9); error against 64-bit sums 3e-13 -> 4e-14.
#pragma once

#include "nk_fxd.cuh"

namespace nk {
namespace {

// ---------------------------------------------------------------- linearization pass
enum { kLcMu = 256, kLcE = 768, kLcCp = 1024 };      // (the derivative kernels' row; its third column unused)

inline size_t linc_fx_smem(const DevMech& m) { return fx_smem(m.fxs[1], m.K, 256); }
inline bool linc_fx_fits(const DevMech& m) { return m.fx_ok && m.fxs[1].np != 0 && linc_fx_smem(m) <= smem_limit(); }

// 1/y for |y| in [2^-100, 2): the float reciprocal and two Newton steps (error near 2^-53)
__device__ __forceinline__ double recip2(double y) {
    const double a = recip_nr(fabs(y)), r = fma(a, fma(-fabs(y), a, 1.0), a);
    return y < 0.0 ? -r : r;
}

// Blocks with a point outside the form (the rates kernel's conditions, |Y_k| in [2^-100, 2)) leave
// kFxSkip in their points' S1 slot for the marked pass of k_linc.cu.
template <int NP, int OWN, int BLOCKS, bool OUT>
__global__ void __launch_bounds__(32 * NP, BLOCKS)
    linc_fx_kernel(const DevMech m, const int64_t n, const int64_t ld, const double* __restrict__ T,
                   const double* __restrict__ p, const double* __restrict__ Y, const double* __restrict__ dlnA,
                   double* __restrict__ lin, const int64_t ldl, double* __restrict__ omega, double* __restrict__ hrr) {
    extern __shared__ __align__(16) unsigned char smem_fx[];
    const FxSet& f = m.fxs[1];
    unsigned char* im0 = smem_fx + kFxBase + kFxScalars * 256;
    const int K = m.K;
    const int lane = threadIdx.x & 31, part = threadIdx.x >> 5;
    const int64_t i0 = (int64_t)blockIdx.x * 32 + lane;
    const bool live = i0 < n;
    const int64_t i = live ? i0 : n - 1;
    long long* sS = reinterpret_cast<long long*>(smem_fx + kFxBase) + lane;
    unsigned char* sP = im0 + 2 * f.image + lane * 8;
    unsigned char* sQ = sP + (size_t)(K + 1) * kFxDRow;

    // a block with a point outside the form leaves here, all its points marked (as in k_jvp_fx.cuh; one
    // zero mass fraction in every block, 53 species, 262,144 points: 9.7 -> 6.8 ms)
    const double Ti = T[i], pi = p[i];
    const unsigned long long Tb = (unsigned long long)__double_as_longlong(Ti);
    double y[OWN];                                           // (all loads in flight at once)
#pragma unroll
    for (int j = 0; j < OWN; ++j) y[j] = part + NP * j < K ? Y[(int64_t)__ldg(&f.sp[part + NP * j].k) * ld + i] : 1.0;
    fx_image_load(f, 0, im0);
    const FxTab ft = stage_fx_tables(reinterpret_cast<uint32_t*>(smem_fx), m.fx_tab);
    const DfTab dt = stage_df_tables(reinterpret_cast<float2*>(smem_fx + kFxTabBytes), m);
    bool bad = !fx_T_ok(Ti) || !fx_p_ok(pi);
#pragma unroll
    for (int j = 0; j < OWN; ++j) bad |= !fx_y_ok(y[j]);
    if (__syncthreads_or(bad) != 0) {
        if (part == 0 && live) lin[cs_S(m) * ldl + i] = __longlong_as_double((long long)kFxSkip);
        fx_image_wait();
        return;
    }
    {
        unsigned long long z = 0, zc = 0;
#pragma unroll
        for (int j = 0; j < OWN; ++j) {
            if (part + NP * j >= K) break;
            fx_add_fraction((unsigned long long)__double_as_longlong(y[j]), __ldg((const long long*)&f.sp[part + NP * j].w), z, zc, bad);
        }
        reinterpret_cast<unsigned long long*>(sQ)[(2 * part) * 32] = z;
        reinterpret_cast<unsigned long long*>(sQ)[(2 * part + 1) * 32] = zc;
    }
    if (part == 0) fx_point_scalars(m, Tb, pi, sS, ft);
    __syncthreads();
    FxT P;
    P.lt = fx_frac63((unsigned long long)sS[kFxLT * 32] << 11);
    P.v = fx_frac63((unsigned long long)sS[kFxV * 32]);
    {
        unsigned long long z = 0, zc = 0;
        for (int q = 0; q < NP; ++q) {
            z += reinterpret_cast<unsigned long long*>(sQ)[(2 * q) * 32];
            zc += reinterpret_cast<unsigned long long*>(sQ)[(2 * q + 1) * 32];
        }
        // (the conditions on the point sums)
        if (__any_sync(0xffffffffu, fx_sums_bad(z, zc))) {
            if (part == 0 && live) lin[cs_S(m) * ldl + i] = __longlong_as_double((long long)kFxSkip);
            fx_image_wait();
            return;
        }
        const long long lrho = sS[kFxLpRT * 32] - fx_log2_int(z, 60, ft) - m.fx_lmaxw;
        const FxFrac u = fx_frac_T(Tb);
#pragma unroll 1
        for (int k = part; k < K; k += NP) {
            const FxSpecies* sp = f.sp + k;
            const int ks = __ldg(&sp->k);
            const double y = Y[(int64_t)ks * ld + i];
            unsigned char* row = sP + k * kFxDRow;
            const int64_t* c = fx_range(sp, Ti);
            const long long a = fx_log2_conc((unsigned long long)__double_as_longlong(y), __ldg((const long long*)&sp->lw) + lrho, ft);
            const long long h = fx_hRT(c, P, u);
            *reinterpret_cast<long long*>(row) = a;
            *reinterpret_cast<long long*>(row + kLcMu) = a + (fx_mu0(c, P, u) & ~1ll);
            *reinterpret_cast<long long*>(row + kLcE) = (1ll << kFxS) - h;
            *reinterpret_cast<long long*>(row + kLcCp) = fx_cpR(c, u);
            if (live) {
                lin[(cs_H(m) + ks) * ldl + i] = fx_to_d(h);
                lin[(cs_iY(m) + ks) * ldl + i] = recip2(y);
                lin[(cs_C(m) + ks) * ldl + i] = fx_exp2<true>(a, ft);
            }
        }
        if (part == 0) {
#pragma unroll
            for (int j = 0; j < kFxDRow / 256; ++j) *reinterpret_cast<long long*>(sP + K * kFxDRow + j * 256) = 0;
            sS[kFxLrho * 32] = lrho;
            sS[kFxSum * 32] = (long long)z;
        }
    }
    fx_image_wait();
    __syncthreads();

    double w[OUT ? OWN : 1];
    if constexpr (OUT) {
#pragma unroll
        for (int j = 0; j < OWN; ++j) w[j] = 0.0;
    }
    double S1 = 0.0;
    for (int c = 0; c < f.nchunk; ++c) {
        const unsigned char* im = im0 + (c & 1) * f.image;
        fx_image_load(f, c + 1, im0 + ((c + 1) & 1) * f.image);
        const int q1 = im[f.image_parts + part + 1];
#pragma unroll 1
        for (int q = im[f.image_parts + part]; q < q1; ++q) {
            const longlong2* rec = reinterpret_cast<const longlong2*>(im + q * (int)sizeof(FxRxn));
            const longlong2 r0 = rec[0], r1 = rec[1];
            const int info = (int)r1.y, r = (int)(r1.y >> 48);
            FxRate L{0, 0};
            long long E = 0, Cp = 0;
            {
                const uint32_t* off = reinterpret_cast<const uint32_t*>(rec + 2);
                const int nr = info & 15, np = info >> 4 & 15;
#pragma unroll 1
                for (int e = 0; e < nr; ++e) {
                    const unsigned char* a = sP + off[e];
                    fx_reac(a, L);
                    E -= *reinterpret_cast<const long long*>(a + kLcE);
                    Cp -= *reinterpret_cast<const long long*>(a + kLcCp);
                }
#pragma unroll 1
                for (int e = 0; e < np; ++e) {
                    const unsigned char* a = sP + off[4 + e];
                    fx_prod(a, L);
                    E += *reinterpret_cast<const long long*>(a + kLcE);
                    Cp += *reinterpret_cast<const long long*>(a + kLcCp);
                }
            }
            const long long ea = fx_mul(r1.x, P.v);
            long long lnk = r0.x + fx_mul(r0.y, P.lt) + ea;
            const long long s = (r0.y >> 5) - fx_scale(ea, 0x58B90BFBE8E7BCD6ull);   // beta + Ea/RT
            long long shift = 0;
            bool big = false;
            if (dlnA) {
                const double d = __ldg(dlnA + (int)(r1.y >> 32 & 0xffff));
                big = ((unsigned)__double2hiint(d) & 0x7fffffffu) >= 0x40a00000u;
                if (!big) shift = fx_log2e_times(d);
                lnk += shift;
            }
            double aT = fx_to_d(s), cL = 0.0;                // L = q cL
            bool zero = false, nan = false;
            const int kind = info >> 8 & 3;
            if (kind != 0) {
                const int4 x = __ldg(reinterpret_cast<const int4*>(m.fx_extra + (info >> 16)));
                long long lM;
                const long long z = fx_third_body(m, x.x, x.y, Y, ld, i, sS[kFxSum * 32], ft, lM);
                lM += sS[kFxLrho * 32];
                zero = z == 0;
                if (kind == 1) {
                    // q holds [M]; with [M] = 0 only L, the term without it, is left
                    if (!zero) lnk = ((lnk + lM) & ~1ll) + (long long)(z < 0);
                    cL = zero ? 1.0 : fx_exp2<true>(-(lM & ~1ll) + (long long)(z < 0), ft);
                } else {
                    const longlong2* tr = reinterpret_cast<const longlong2*>(m.fx_troe + x.z);
                    const longlong2 a = __ldg(tr), b = __ldg(tr + 1);
                    const long long e0 = fx_mul(b.x, P.v);
                    const long long l0 = a.x + fx_mul(a.y, P.lt) + e0 + shift;
                    const FxTroeD t = fx_troe_d(m.fx_troe, m.troe_df, m.troe, x.z, Ti, P.v, l0 - lnk + lM, ft, dt);
                    lnk += t.phi;
                    const long long s0 = (a.y >> 5) - fx_scale(e0, 0x58B90BFBE8E7BCD6ull);
                    aT += df_to_d(df_fma(t.px, fx_to_pair(s0 - s), t.pt));
                    cL = df_to_d(t.px) * fx_exp2(-lM, ft);
                    nan = z < 0;
                }
            }
            if (kind != 1) lnk &= ~1ll;
            L.f += lnk;
            double qf = fx_exp2<true>(L.f, ft), qr = fx_exp2<true>(L.f + L.r, ft);
            if (kind == 2 && (zero || nan)) qf = qr = zero ? 0.0 : __longlong_as_double(0x7ff8000000000000ll);
            if (big) {
                const double d = __ldg(dlnA + (int)(r1.y >> 32 & 0xffff));
                qf = fx_shift_edge(qf, d);
                qr = fx_shift_edge(qr, d);
            }
            double qq = qf - qr;
            const double qc = qq;
            if (kind == 1 && zero) qq = qf = qr = 0.0;
            S1 = fma(qq, fx_to_d(Cp), S1);
            if constexpr (OUT) *reinterpret_cast<double*>(sQ + q * 256) = qq;
            if (live) {
                double* o = lin + i;
                o[(int64_t)r * ldl] = fma(qq, aT, qr * fx_to_d(-E));
                const int nu = __ldg(m.fx_nu1 + r);                  // first coefficients of the sides
                if ((nu & 15) != 1) qf = times_nu(qf, nu & 15);
                if ((nu >> 4) != 1) qr = times_nu(qr, nu >> 4);
                o[(cs_Vf(m) + r) * ldl] = qf;
                o[(cs_Vb(m) + r) * ldl] = -qr;
                if (kind != 0) o[(cs_L(m) + (r - m.R_el)) * ldl] = qc * cL;
            }
        }
        __syncthreads();
        if constexpr (OUT) {
            const uint32_t* spec = reinterpret_cast<const uint32_t*>(im + f.image_spec);
            const unsigned char* list = im + f.image_list;
#pragma unroll
            for (int j = 0; j < OWN; ++j)
                if (part + NP * j < K) w[j] = fx_gather(spec[part + NP * j], list, sQ, w[j]);
        }
        fx_image_wait();
        __syncthreads();
    }

    double h = 0.0;
    if constexpr (OUT) {
#pragma unroll
        for (int j = 0; j < OWN; ++j)
            if (part + NP * j < K) *reinterpret_cast<double*>(sP + (part + NP * j) * kFxDRow) = w[j];
#pragma unroll 1
        for (int k = part; k < K; k += NP) {
            const unsigned char* row = sP + k * kFxDRow;
            const double o = *reinterpret_cast<const double*>(row);
            h = fma(fx_to_d((1ll << kFxS) - *reinterpret_cast<const long long*>(row + kLcE)), o, h);
            if (live) omega[(int64_t)__ldg(&f.sp[k].k) * ld + i] = o;
        }
    }
    double* sR = reinterpret_cast<double*>(sQ);
    sR[(2 * part) * 32] = S1;
    if constexpr (OUT) sR[(2 * part + 1) * 32] = h;
    __syncthreads();
    if (part != 0 || !live) return;
    for (int q = 1; q < NP; ++q) {
        S1 += sR[(2 * q) * 32];
        if constexpr (OUT) h += sR[(2 * q + 1) * 32];
    }
    lin[cs_S(m) * ldl + i] = S1 * kFxCpScale;
    if constexpr (OUT) hrr[i] = -kR * Ti * h;
}

template <bool OUT>
cudaError_t launch_linc_fx(const DevMech& m, int64_t n, int64_t ld, const double* T, const double* p, const double* Y,
                           const double* dlnA, double* lin, int64_t ldl, double* omega, double* hrr, cudaStream_t s) {
    const size_t smem = linc_fx_smem(m);
    const int np = m.fxs[1].np;
    auto kern = np == 4 ? linc_fx_kernel<4, 8, 6, OUT> : np == 12 ? linc_fx_kernel<12, 6, 2, OUT> : linc_fx_kernel<24, 6, 1, OUT>;
    const cudaError_t e = ensure_smem((const void*)kern, smem);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)((n + 31) / 32), 32 * np, smem, s>>>(m, n, ld, T, p, Y, dlnA, lin, ldl, omega, hrr);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- product pass
// The tangent of one side whose sum of r_e is not finite: the exact form where a 1/Y_e of the side
// is NaN, else V g as it is.  Out of line, read from the reaction's record.
static __device__ __noinline__ double side_exact(const RxnRec* rec, const double* invW, int side, double V, double g,
                                                 const double* iY, ExactCtx c) {
    const int4* q = reinterpret_cast<const int4*>(rec) + 6;
    const int4 h = __ldg(q), sp = __ldg(q + 2 + side), nu = __ldg(q + 4 + side);
    const int ne = side ? h.z : h.y;
    const int s4[kMaxSide] = {sp.x, sp.y, sp.z, sp.w};
    bool tiny = false;
    for (int e = 0; e < ne; ++e) tiny |= nonfinite(iY[(int64_t)s4[e] * c.ldl]);
    if (!tiny) return V * g;
    return V * side_tangent_exact(invW, ne, sp, nu, c);
}

// sum of r over a side's n molecules (1..4), a branch per count: adding under n > 1, n > 2, .. leaves
// predicated FP64 additions, which cost as much as executed ones
__device__ __forceinline__ double side_flat(const unsigned char* r, uint4 o, int n) {
    const double a = *reinterpret_cast<const double*>(r + o.x);
    switch (n) {
        case 1: return a;
        case 2: return a + *reinterpret_cast<const double*>(r + o.y);
        case 3: return a + *reinterpret_cast<const double*>(r + o.y) + *reinterpret_cast<const double*>(r + o.z);
        default:
            return a + *reinterpret_cast<const double*>(r + o.y) + *reinterpret_cast<const double*>(r + o.z) +
                   *reinterpret_cast<const double*>(r + o.w);
    }
}
static __device__ __noinline__ double over_nu(double g, int nu) { return g / (double)nu; }

static __device__ __noinline__ double side_edge(const RxnRec* rec, const double* invW, double Vf, double gf, double Vb,
                                                double gb, double a, const double* iY, ExactCtx c) {
    return a + (nonfinite(gf) ? side_exact(rec, invW, 0, Vf, gf, iY, c) : Vf * gf) +
           (nonfinite(gb) ? side_exact(rec, invW, 1, Vb, gb, iY, c) : Vb * gb);
}

// r_k in a row per species (slot order), the reactions' dq staged per chunk and summed by species:
// 34 KB of shared memory at 53 species, 24 warps per SM, where a row of d omega_k partials per warp
// held it at 12, and every point sum is made once instead of once per warp.
// dC_k has a row too: the efficiency sums are one operation and no global load of the state per entry.
constexpr int kPcScalars = 4;                       // dT/T, d rho/rho, rho, d(p/RT)

inline size_t jvpc_fx_smem(const DevMech& m) {
    const FxSet& f = m.fxs[2];
    const size_t q = (size_t)f.rows * 256, part = (size_t)f.np * 3 * 256;
    return kPcScalars * 256 + 2 * (size_t)f.image + (size_t)f.row * (m.K + 1) + (size_t)m.K * 256 + (q > part ? q : part);
}

// the stored words of one reaction
struct WordsC {
    double A, Vf, Vb, L;
    int nu;
};
__device__ __forceinline__ void load_words(const DevMech& m, const unsigned char* im, int q, const double* o, int64_t ldl,
                                           WordsC& w) {
    const long long hd = reinterpret_cast<const longlong2*>(im + q * (int)sizeof(FxRxn))[1].y;
    const int r = (int)(hd >> 48);
    w.A = __ldcs(o + (int64_t)r * ldl);
    w.Vf = __ldcs(o + (cs_Vf(m) + r) * ldl);
    w.Vb = __ldcs(o + (cs_Vb(m) + r) * ldl);
    w.L = ((int)hd >> 8 & 3) != 0 ? __ldcs(o + (cs_L(m) + (r - m.R_el)) * ldl) : 0.0;
    w.nu = __ldg(m.fx_nu1 + r);
}

// The stored words of a chunk's reactions into L2, while the chunk before is gathered: a row of the
// block's 32 points is 256 bytes, two lines.  (Words loaded a reaction ahead into registers spilled
// 240 bytes at the kernel's 80 registers.)
__device__ __forceinline__ void prefetch_words(const DevMech& m, const FxSet& f, int np, const unsigned char* im,
                                               const double* lin, int64_t ldl, int64_t n) {
    const int total = im[f.image_parts + np] * 8;
    for (int t = threadIdx.x; t < total; t += blockDim.x) {
        const long long hd = reinterpret_cast<const longlong2*>(im + (t >> 3) * (int)sizeof(FxRxn))[1].y;
        const int r = (int)(hd >> 48), word = t >> 1 & 3;
        if (word == 3 && ((int)hd >> 8 & 3) == 0) continue;
        const int64_t row = word == 0 ? r : word == 1 ? cs_Vf(m) + r : word == 2 ? cs_Vb(m) + r : cs_L(m) + (r - m.R_el);
        const int64_t pt = min((int64_t)blockIdx.x * 32 + (t & 1) * 16, n - 1);
        asm volatile("prefetch.global.L2 [%0];" ::"l"(lin + row * ldl + pt));
    }
}

template <int NP, bool RHS>
__global__ void __launch_bounds__(32 * NP, NP == 4 ? 6 : NP == 8 ? 3 : NP == 16 ? 2 : 1)
    jvpc_fx_kernel(const DevMech m, const int64_t n, const int64_t ld, const double* __restrict__ T,
                   const double* __restrict__ p, const double* __restrict__ Y, const double* __restrict__ lin,
                   const int64_t ldl, const double* __restrict__ vT, const double* __restrict__ vY,
                   double* __restrict__ d_omega, double* __restrict__ d_hrr, const double* __restrict__ fT,
                   const double* __restrict__ fY, const int64_t ldf) {
    extern __shared__ __align__(16) unsigned char smem_fx[];
    const FxSet& f = m.fxs[2];
    unsigned char* im0 = smem_fx + kPcScalars * 256;
    fx_image_load(f, 0, im0);
    const int K = m.K;
    const int lane = threadIdx.x & 31, part = threadIdx.x >> 5;
    const int64_t i0 = (int64_t)blockIdx.x * 32 + lane;
    const bool live = i0 < n;
    const int64_t i = live ? i0 : n - 1;
    double* sV = reinterpret_cast<double*>(smem_fx) + lane;
    unsigned char* sP = im0 + 2 * f.image + lane * 8;
    double* sC = reinterpret_cast<double*>(sP + (size_t)(K + 1) * 256);          // dC_k, species order
    unsigned char* sQ = sP + (size_t)(2 * K + 1) * 256;
    double* sR = reinterpret_cast<double*>(sQ);
    {
        double s = 0.0, ds = 0.0;
#pragma unroll 1
        for (int k = part; k < K; k += NP) {
            const double iw = __ldg(m.invW + k);
            s = fma(Y[(int64_t)k * ld + i], iw, s);
            ds = fma(vY[(int64_t)k * ld + i], iw, ds);
        }
        sR[(2 * part) * 32] = s;
        sR[(2 * part + 1) * 32] = ds;
    }
    __syncthreads();
    if (part == 0) {
        double s = sR[0], ds = sR[32];
        for (int q = 1; q < NP; ++q) {
            s += sR[(2 * q) * 32];
            ds += sR[(2 * q + 1) * 32];
        }
        const double invT = 1.0 / T[i], tT = vT[i] * invT, pRT = p[i] * invT * kInvR, is = 1.0 / s;
        sV[0] = tT;
        sV[32] = -tT - ds * is;                       // d rho / rho
        sV[64] = pRT * is;                            // rho
        sV[96] = -pRT * tT;                           // d(p/RT)
        *reinterpret_cast<double*>(sP + K * 256) = 0.0;
    }
    __syncthreads();
#pragma unroll 1
    for (int k = part; k < K; k += NP) {
        const int ks = __ldg(&f.sp[k].k);
        const double v = vY[(int64_t)ks * ld + i], ar = sV[32];
        *reinterpret_cast<double*>(sP + k * 256) = fma(v, lin[(cs_iY(m) + ks) * ldl + i], ar);
        sC[ks * 32] = fma(sV[64] * __ldg(m.invW + ks), v, ar * lin[(cs_C(m) + ks) * ldl + i]);
    }
    fx_image_wait();
    __syncthreads();

    double w[kFxOwn];
#pragma unroll
    for (int j = 0; j < kFxOwn; ++j) w[j] = 0.0;
    const double* o = lin + i;
    for (int c = 0; c < f.nchunk; ++c) {
        const unsigned char* im = im0 + (c & 1) * f.image;
        fx_image_load(f, c + 1, im0 + ((c + 1) & 1) * f.image);
        const int q1 = im[f.image_parts + part + 1];
#pragma unroll 1
        for (int q = im[f.image_parts + part]; q < q1; ++q) {
            const longlong2* rec = reinterpret_cast<const longlong2*>(im + q * (int)sizeof(FxRxn));
            const long long hd = rec[1].y;
            const int info = (int)hd, r = (int)(hd >> 48), kind = info >> 8 & 3;
            WordsC v;
            load_words(m, im, q, o, ldl, v);
            const uint4 re = reinterpret_cast<const uint4*>(rec)[2], pr = reinterpret_cast<const uint4*>(rec)[3];
            const int nr = info & 15, np = info >> 4 & 15;
            double gf = side_flat(sP, re, nr), gb = side_flat(sP, pr, np);
            const int nu = v.nu;                       // the stored V carry the first entries' coefficients
            if ((nu & 15) != 1) gf = over_nu(gf, nu & 15);
            if ((nu >> 4) != 1) gb = over_nu(gb, nu >> 4);
            double dq;
            if (!nonfinite(gf) && !nonfinite(gb)) {
                dq = fma(v.Vf, gf, fma(v.Vb, gb, v.A * sV[0]));
            } else {
                dq = side_edge(m.rxn + r, m.invW, v.Vf, gf, v.Vb, gb, v.A * sV[0], lin + cs_iY(m) * ldl + i,
                               ExactCtx{lin + cs_C(m) * ldl + i, vY + i, ldl, ld, sV[64], sV[32]});
            }
            if (kind != 0) {
                const int2 e = __ldg(reinterpret_cast<const int2*>(m.fx_extra + (info >> 16)));
                double dM = sV[96];                    // d[M] = d(p/RT) + sum (eps - 1) dC
#pragma unroll 1
                for (int j = e.x; j < e.y; ++j) dM = fma(__ldg(m.eff_m1 + j), sC[__ldg(&m.fx_eff[j].sp) * 32], dM);
                dq = fma(v.L, dM, dq);
            }
            *reinterpret_cast<double*>(sQ + q * 256) = dq;
        }
        fx_image_wait();
        __syncthreads();
        if (c + 1 < f.nchunk) prefetch_words(m, f, NP, im0 + ((c + 1) & 1) * f.image, lin, ldl, n);
        const uint32_t* spec = reinterpret_cast<const uint32_t*>(im + f.image_spec);
        const unsigned char* list = im + f.image_list;
#pragma unroll
        for (int j = 0; j < kFxOwn; ++j)
            if (part + NP * j < K) w[j] = fx_gather(spec[part + NP * j], list, sQ, w[j]);
        __syncthreads();
    }
    // d omega_k in species order (r_k is dead), then the shared epilogue
#pragma unroll
    for (int j = 0; j < kFxOwn; ++j)
        if (part + NP * j < K) *reinterpret_cast<double*>(sP + __ldg(&f.sp[part + NP * j].k) * 256) = w[j];
    __syncthreads();
    lin_epilogue<32, NP, RHS, 1>(m, part, live, i, T[i], vT[i], sV[64], sV[32], reinterpret_cast<double*>(sP), sR,
                                 lin + cs_H(m) * ldl + i, lin + cs_S(m) * ldl + i, ldl, Y, vY, ld, fT, fY, ldf, d_omega,
                                 d_hrr);
}

template <bool RHS>
cudaError_t launch_jvpc_fx(const DevMech& m, int64_t n, int64_t ld, const double* T, const double* p, const double* Y,
                           const double* lin, int64_t ldl, const double* vT, const double* vY, double* d_omega,
                           double* d_hrr, const double* fT, const double* fY, int64_t ldf, cudaStream_t s) {
    const size_t smem = jvpc_fx_smem(m);
    const int np = m.fxs[2].np;
    auto kern = np == 4 ? jvpc_fx_kernel<4, RHS> : np == 8 ? jvpc_fx_kernel<8, RHS> : np == 16 ? jvpc_fx_kernel<16, RHS>
                                                                                              : jvpc_fx_kernel<32, RHS>;
    const cudaError_t e = ensure_smem((const void*)kern, smem);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)((n + 31) / 32), 32 * np, smem, s>>>(m, n, ld, T, p, Y, lin, ldl, vT, vY, d_omega, d_hrr, fT, fY, ldf);
    return cudaGetLastError();
}

}  // namespace
}  // namespace nk
