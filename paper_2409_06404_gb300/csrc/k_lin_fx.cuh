// The per-entry stored linearization of the reactor on fixed-point logarithms (nk_fx.cuh, nk_fxpt.cuh, nk_fxd.cuh;
// included by k_lin.cu, whose slots and store_coef it uses): an entry's coefficient is its side's term
// divided by the concentration, nu_e q_side / C_e, one product with a row of 1/C_k, where the pair
// kernel formed exclusive products of the concentrations.  The stored words bound it together with
// the FP64 pipe (one quotient's product per entry).  53 species, states in the form: 16,384 points 0.42 ms by
// the pair kernel in four parts a point -> 0.245, 262,144 points 6.04 -> 3.10.  (Near-equilibrium states, whose
// rare species lie below 2^-100, stay with the pair kernel; a reactor step on 16,384 of them went from 9.50 to
// 8.44 ms by its launch shape, k_lin.cu, and by what the factorization gained.)
// For linearizations a solver keeps to itself; the public one and the single-precision data rounded
// from it stay with the pair kernel: two linearizations that differ by 3e-13 round some hundred
// coefficients of a field to the other float, 6e-8 of a product.
#pragma once

#include "nk_fxd.cuh"

namespace nk {
namespace {

enum { kLeMu = 256, kLeIC = 512, kLeE = 768, kLeCp = 1024 };   // (the derivative kernels' row)

inline size_t lin_fx_smem(const DevMech& m) { return fx_smem(m.fxs[1], m.K, 64); }
inline bool lin_fx_fits(const DevMech& m) { return m.fx_ok && m.fxs[1].np != 0 && lin_fx_smem(m) <= smem_limit(); }

// nu_e q / C_e of a side's entries (each a branch per count: predicated FP64 products cost as much as
// executed ones), an entry's first molecule found by adding up the coefficients before it
template <int N>
__device__ __forceinline__ void entry_coefs_n(const unsigned char* ic, const uint32_t* off, const int* nu, double q, double* B) {
    int at = 0;
#pragma unroll
    for (int e = 0; e < N; ++e) {
        double b = q * *reinterpret_cast<const double*>(ic + off[at]);
        if (nu[e] != 1) b = times_nu(b, nu[e]);
        B[e] = b;
        at += nu[e];
    }
}
__device__ __forceinline__ void entry_coefs(const unsigned char* ic, const uint32_t* off, int n, const int* nu, double q, double* B) {
    switch (n) {
        case 1: entry_coefs_n<1>(ic, off, nu, q, B); break;
        case 2: entry_coefs_n<2>(ic, off, nu, q, B); break;
        case 3: entry_coefs_n<3>(ic, off, nu, q, B); break;
        default: entry_coefs_n<4>(ic, off, nu, q, B); break;
    }
}

// Blocks with a point outside the form (as in k_linc_fx.cuh) leave kFxSkip in their points' S1 slot for
// the marked pass of k_lin.cu.
template <int NP, int OWN, int BLOCKS>
__global__ void __launch_bounds__(32 * NP, BLOCKS)
    lin_fx_kernel(const DevMech m, const int64_t n, const int64_t ld, const double* __restrict__ T,
                  const double* __restrict__ p, const double* __restrict__ Y, const double* __restrict__ dlnA,
                  double* __restrict__ lin, const int64_t ldl) {
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
    unsigned char* sQ = sP + (size_t)(K + 1) * kFxDRow;                      // the parts' sums

    // a block with a point outside the form leaves here, all its points marked (as in k_jvp_fx.cuh; one
    // zero mass fraction in every block, 53 species, 262,144 points: 9.1 -> 6.1 ms)
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
        if (part == 0 && live) lin[slot_S(m) * ldl + i] = __longlong_as_double((long long)kFxSkip);
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
            if (part == 0 && live) lin[slot_S(m) * ldl + i] = __longlong_as_double((long long)kFxSkip);
            fx_image_wait();
            return;
        }
        const long long lrho = sS[kFxLpRT * 32] - fx_log2_int(z, 60, ft) - m.fx_lmaxw;
        const FxFrac u = fx_frac_T(Tb);
#pragma unroll 1
        for (int k = part; k < K; k += NP) {
            const FxSpecies* sp = f.sp + k;
            const int ks = __ldg(&sp->k);
            unsigned char* row = sP + k * kFxDRow;
            const int64_t* c = fx_range(sp, Ti);
            const long long a = fx_log2_conc((unsigned long long)__double_as_longlong(Y[(int64_t)ks * ld + i]), __ldg((const long long*)&sp->lw) + lrho, ft);
            const long long h = fx_hRT(c, P, u);
            *reinterpret_cast<long long*>(row) = a;
            *reinterpret_cast<long long*>(row + kLeMu) = a + (fx_mu0(c, P, u) & ~1ll);
            *reinterpret_cast<double*>(row + kLeIC) = fx_exp2<true>((a & 1) - (a & ~1ll), ft);
            *reinterpret_cast<long long*>(row + kLeE) = (1ll << kFxS) - h;
            *reinterpret_cast<long long*>(row + kLeCp) = fx_cpR(c, u);
            if (live) lin[(slot_H(m) + ks) * ldl + i] = fx_to_d(h);
        }
        if (part == 0) {
            sS[kFxLrho * 32] = lrho;
            sS[kFxSum * 32] = (long long)z;
        }
    }
    fx_image_wait();
    __syncthreads();

    double S1 = 0.0;
    for (int c = 0; c < f.nchunk; ++c) {
        const unsigned char* im = im0 + (c & 1) * f.image;
        fx_image_load(f, c + 1, im0 + ((c + 1) & 1) * f.image);
        const int q1 = im[f.image_parts + part + 1];
#pragma unroll 1
        for (int q = im[f.image_parts + part]; q < q1; ++q) {
            const longlong2* rec = reinterpret_cast<const longlong2*>(im + q * (int)sizeof(FxRxn));
            const longlong2 r0 = rec[0], r1 = rec[1];
            const uint32_t* off = reinterpret_cast<const uint32_t*>(rec + 2);
            const int info = (int)r1.y, r = (int)(r1.y >> 48);
            FxRate L{0, 0};
            long long E = 0, Cp = 0;
            {
                const int nr = info & 15, np = info >> 4 & 15;
#pragma unroll 1
                for (int e = 0; e < nr; ++e) {
                    const unsigned char* a = sP + off[e];
                    fx_reac(a, L);
                    E -= *reinterpret_cast<const long long*>(a + kLeE);
                    Cp -= *reinterpret_cast<const long long*>(a + kLeCp);
                }
#pragma unroll 1
                for (int e = 0; e < np; ++e) {
                    const unsigned char* a = sP + off[4 + e];
                    fx_prod(a, L);
                    E += *reinterpret_cast<const long long*>(a + kLeE);
                    Cp += *reinterpret_cast<const long long*>(a + kLeCp);
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
            if (live) {
                const int4* xr = reinterpret_cast<const int4*>(m.rxn + r) + 6;
                const int4 h = __ldg(xr), s0 = __ldg(xr + 2), s1 = __ldg(xr + 3), u0 = __ldg(xr + 4), u1 = __ldg(xr + 5);
                const int sp[2 * kMaxSide] = {s0.x, s0.y, s0.z, s0.w, s1.x, s1.y, s1.z, s1.w};
                const int nu[2 * kMaxSide] = {u0.x, u0.y, u0.z, u0.w, u1.x, u1.y, u1.z, u1.w};
                double Bv[2 * kMaxSide] = {};
                entry_coefs(sP + kLeIC, off, h.y, nu, qf, Bv);
                entry_coefs(sP + kLeIC, off + 4, h.z, nu + kMaxSide, -qr, Bv + kMaxSide);
                const double A = fma(qq, aT, qr * fx_to_d(-E));
                if (kind == 0)
                    store_coef<32, 0>(m, r, lin, ldl, i, h.y, h.z, sp, nullptr, A, Bv, 0.0);
                else
                    store_coef<32, 1>(m, r, lin, ldl, i, h.y, h.z, sp, nullptr, A, Bv, qc * cL);
            }
        }
        fx_image_wait();
        __syncthreads();
    }

    double* sR = reinterpret_cast<double*>(sQ);
    sR[part * 32] = S1;
    __syncthreads();
    if (part != 0 || !live) return;
    for (int q = 1; q < NP; ++q) S1 += sR[q * 32];
    lin[slot_S(m) * ldl + i] = S1 * kFxCpScale;
}

inline cudaError_t launch_lin_fx(const DevMech& m, int64_t n, int64_t ld, const double* T, const double* p, const double* Y,
                          const double* dlnA, double* lin, int64_t ldl, cudaStream_t s) {
    const size_t smem = lin_fx_smem(m);
    const int np = m.fxs[1].np;
    auto kern = np == 4 ? lin_fx_kernel<4, 8, 6> : np == 12 ? lin_fx_kernel<12, 6, 2> : lin_fx_kernel<24, 6, 1>;
    const cudaError_t e = ensure_smem((const void*)kern, smem);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)((n + 31) / 32), 32 * np, smem, s>>>(m, n, ld, T, p, Y, dlnA, lin, ldl);
    return cudaGetLastError();
}

}  // namespace
}  // namespace nk
