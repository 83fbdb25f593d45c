// Rates kernel of the FP64 form on fixed-point logarithms (nk_fx.cuh, nk_fxpt.cuh): the path of
// every mechanism whose numbers fit the format (DevMech::fx_ok: at most four molecules per side,
// rate constants and reaction Gibbs energies below 2^2900 over the temperature window).
//
// The kernel it takes the place of (k_rates.cuh, pairs) spent about 720 instructions and 11.4 FP64
// operations per reaction and point at 53 species / 325 reactions: the reaction's Gibbs polynomials
// in pairs, ln C sums in pairs, one FP64 operation per exponential, a block barrier per round.
// Here a reaction takes about 320 instructions and 6.7 FP64 operations (the difference of the two
// terms and one addition per molecule), and issue slots and the FP64 pipe bound it about equally
// (61% and 56% busy).  Accumulators in registers, loops over species not unrolled and the falloff
// out of line: the unrolled form of the same kernel measured 18 ms, waiting for instructions.
// 53 species, 2,097,152 points: 22.0 -> 13.9 ms; its error against 64-bit sums fell from 3e-13 to
// 3e-14 (2-norm).
#pragma once

#include "nk_fxpt.cuh"

namespace nk {
namespace {

// the float of ln T from log2 T
__device__ __forceinline__ float fx_lnT_float(long long lT) {
    const dfl a = df_mul(fx_to_pair(lT), dfl{0.693147182464599609375f, -1.9046542121259336e-09f});
    return a.h + a.l;
}
// q times a float (out of line: the product would be predicated for every reaction)
static __device__ __noinline__ double fx_times_float(double q, float f) { return q * widen(f); }
// the mixed form's falloff factor F P_r/(1 + P_r), all in single precision
static __device__ __noinline__ float fx_troe_float(const TroeRecF* t, float Mf, float lnkf, float shf, float Tf, float lnTf,
                                                   float invTf) {
    const float4 t0 = __ldg(reinterpret_cast<const float4*>(t));       // lnA0, beta0, Ea0R, a
    const float4 t1 = __ldg(reinterpret_cast<const float4*>(t) + 1);   // 1/T3, 1/T1, T2, has
    if (Mf == 0.0f) return 0.0f;
    const float lnk0 = fmaf(-t0.z, invTf, fmaf(t0.y, lnTf, t0.x + shf));
    const float lnPr = lnk0 - lnkf + logf(Mf);
    float Fc = (1.0f - t0.w) * expf(-Tf * t1.x) + t0.w * expf(-Tf * t1.y);
    if (t1.w != 0.0f) Fc += expf(-t1.z * invTf);
    const float lFc = log10f(Fc);
    const float c = fmaf(-0.67f, lFc, -0.4f);
    const float nn = fmaf(-1.27f, lFc, 0.75f);
    const float u = fmaf(lnPr, (float)kInvLn10, c);
    const float f1 = u / fmaf(-0.14f, u, nn);
    const float lF = lFc / fmaf(f1, f1, 1.0f);
    return exp10f(lF) / (1.0f + expf(-lnPr));
}

// NP parts per point, 32 points per block.  RHS: the implicit-stage sources instead (omega ->
// W_k omega_k / rho, hrr -> hrr/(rho c_p)).  A point outside the fixed-point form (fx_T_ok, fx_p_ok,
// fx_add_fraction, fx_sums_bad) leaves kFxSkip in its hrr: the fallback pass
// (k_rates.cuh) takes it.
// MIXED (NK_MIXED): ln k_f and the whole falloff in single precision, operation by operation as the
// pair kernel's mixed form has them (so its results stay, to some 1e-13); concentrations, K_c, the
// difference and the sums as in the FP64 form.  Rates and transport at 120 species / 700
// reactions, 110,592 points: 7.05 -> 5.21 ms (all of it the rates').
template <int NP, bool RHS, bool MIXED>
__global__ void __launch_bounds__(32 * NP, NP <= 32 ? 32 / NP : 1)
    rates_fx_kernel(const DevMech m, const int64_t n, const int64_t ld, const double* __restrict__ T,
                    const double* __restrict__ p, const double* __restrict__ Y, const double* __restrict__ dlnA,
                    double* __restrict__ omega, double* __restrict__ hrr) {
    extern __shared__ __align__(16) unsigned char smem_fx[];
    unsigned char* im0 = smem_fx + kFxBase + kFxScalars * 256;
    const FxSet& f = m.fxs[0];
    const int K = m.K;
    const int lane = threadIdx.x & 31, part = threadIdx.x >> 5;
    const int64_t i0 = (int64_t)blockIdx.x * 32 + lane;
    const bool live = i0 < n;
    const int64_t i = live ? i0 : n - 1;                 // idle lanes of the last block repeat point n-1
    double Ti = T[i];
    const double pi = p[i];
    bool bad = !fx_T_ok(Ti) || !fx_p_ok(pi);
    // A block with no point in T's and p's ranges leaves before its set-up (every part holds the same
    // points).  Among others single points are left to the fallback pass alone: a point's result does
    // not depend on its neighbours.
    if (__all_sync(0xffffffffu, bad)) {
        if (part == 0 && live) hrr[i] = __longlong_as_double((long long)kFxSkip);
        return;
    }
    fx_image_load(f, 0, im0);
    const FxTab ft = stage_fx_tables(reinterpret_cast<uint32_t*>(smem_fx), m.fx_tab);
    const DfTab dt = stage_df_tables(reinterpret_cast<float2*>(smem_fx + kFxTabBytes), m);   // (Troe)
    __syncthreads();
    long long* sS = reinterpret_cast<long long*>(smem_fx + kFxBase) + lane;
    unsigned char* sP = im0 + 2 * f.image + lane * 8;                         // species rows
    unsigned char* sQ = sP + (size_t)(K + 1) * kFxRow;                           // rates of progress

    if (bad) Ti = 1000.0;                                // the lane goes on with any state, its results are not stored
    const unsigned long long Tb = (unsigned long long)__double_as_longlong(Ti);
    {
        unsigned long long z = 0, zc = 0;
#pragma unroll 1
        for (int k = part; k < K; k += NP) {
            const FxSpecies* sp = f.sp + k;
            fx_add_fraction((unsigned long long)__double_as_longlong(Y[(int64_t)__ldg(&sp->k) * ld + i]),
                            __ldg((const long long*)&sp->w), z, zc, bad);
        }
        if (part == 0) fx_point_scalars(m, Tb, pi, sS, ft);
        reinterpret_cast<unsigned long long*>(sQ)[(2 * part) * 32] = z;
        reinterpret_cast<unsigned long long*>(sQ)[(2 * part + 1) * 32] = bad ? kFxPoison : zc;
    }
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
        bad = fx_sums_bad(z, zc);
        const long long lrho = bad ? 0 : sS[kFxLpRT * 32] - fx_log2_int(z, 60, ft) - m.fx_lmaxw;
        const FxFrac u = fx_frac_T(Tb);
#pragma unroll 1
        for (int k = part; k < K; k += NP) {
            const FxSpecies* sp = f.sp + k;
            const unsigned long long yb = (unsigned long long)__double_as_longlong(Y[(int64_t)__ldg(&sp->k) * ld + i]);
            const long long a = bad ? 0 : fx_log2_conc(yb, __ldg((const long long*)&sp->lw) + lrho, ft);
            *reinterpret_cast<long long*>(sP + k * kFxRow) = a;
            *reinterpret_cast<long long*>(sP + k * kFxRow + 256) = a + (fx_mu0(fx_range(sp, Ti), P, u) & ~1ll);
        }
        if (part == 0) {
            if constexpr (MIXED) {
                // T, ln T and 1/T in single precision, as the pair kernel rounds them
                const float lnT = fx_lnT_float(sS[kFxLT * 32]);
                sS[kFxTf * 32] = (long long)((unsigned long long)__float_as_uint(lnT) << 32 | __float_as_uint(narrow(1.0 / Ti)));
            }
            *reinterpret_cast<long long*>(sP + K * kFxRow) = 0;
            *reinterpret_cast<long long*>(sP + K * kFxRow + 256) = 0;
            sS[kFxLrho * 32] = lrho;
            sS[kFxSum * 32] = bad ? 0 : (long long)z;
        }
    }
    fx_image_wait();
    __syncthreads();

    double w[kFxOwn];
#pragma unroll
    for (int j = 0; j < kFxOwn; ++j) w[j] = 0.0;
    for (int c = 0; c < f.nchunk; ++c) {
        const unsigned char* im = im0 + (c & 1) * f.image;
        fx_image_load(f, c + 1, im0 + ((c + 1) & 1) * f.image);
        const int q1 = im[f.image_parts + part + 1];
        for (int q = im[f.image_parts + part]; q < q1; ++q) {
            const longlong2* rec = reinterpret_cast<const longlong2*>(im + q * (int)sizeof(FxRxn));
            const longlong2 r0 = rec[0], r1 = rec[1];       // lnA, beta; Ea, (info, orig)
            const int info = (int)r1.y;
            FxRate L = fx_sides(sP, info, reinterpret_cast<const uint4*>(rec)[2], reinterpret_cast<const uint4*>(rec)[3]);
            long long lnk = 0;
            float lnkf = 0.0f, lnTf = 0.0f, invTf = 0.0f, shf = 0.0f;
            if constexpr (MIXED) {
                const unsigned long long tf = (unsigned long long)sS[kFxTf * 32];
                lnTf = __uint_as_float((unsigned)(tf >> 32));
                invTf = __uint_as_float((unsigned)tf);
                const int orig = (int)(r1.y >> 32 & 0xffff), dev = (int)((unsigned long long)r1.y >> 48);
                if (dlnA) shf = (float)__ldg(dlnA + orig);
                const float4 xf = __ldg(reinterpret_cast<const float4*>(m.rxnf + dev));   // lnA, beta, EaR
                lnkf = fmaf(-xf.z, invTf, fmaf(xf.y, lnTf, xf.x + shf));
                lnk = fx_log2e_times(lnkf);
            } else {
                lnk = r0.x + fx_mul(r0.y, P.lt) + fx_mul(r1.x, P.v);
            }
            long long shift = 0;
            bool big = false;                               // a shift of ln A outside +-2048 (or NaN)
            if (MIXED) {
                big = !(fabsf(lnkf) < 2000.0f);
                if (big) lnk = 0;
            }
            if (!MIXED && dlnA) {
                const double d = __ldg(dlnA + (int)(r1.y >> 32 & 0xffff));
                big = ((unsigned)__double2hiint(d) & 0x7fffffffu) >= 0x40a00000u;
                if (!big) shift = fx_log2e_times(d);
                lnk += shift;
            }
            long long z = 1;                                // [M]/rho' of third-body and Troe reactions
            [[maybe_unused]] float Ff = 1.0f;
            const int kind = info >> 8 & 3;
            if (kind != 0) {
                const int4 x = __ldg(reinterpret_cast<const int4*>(m.fx_extra + (info >> 16)));
                long long lM;
                z = fx_third_body(m, x.x, x.y, Y, ld, i, sS[kFxSum * 32], ft, lM);
                lM += sS[kFxLrho * 32];
                if (kind == 1) {
                    lnk = ((lnk + lM) & ~1ll) + (long long)(z < 0);
                } else if constexpr (MIXED) {
                    Ff = fx_troe_float(m.troef + x.z, z == 0 ? 0.0f : z < 0 ? -narrow(fx_exp2(lM, ft)) : narrow(fx_exp2(lM, ft)), lnkf, shf, narrow(Ti), lnTf, invTf);
                } else {
                    const longlong2* tr = reinterpret_cast<const longlong2*>(m.fx_troe + x.z);
                    const longlong2 a = __ldg(tr), b = __ldg(tr + 1);
                    const long long l0 = a.x + fx_mul(a.y, P.lt) + fx_mul(b.x, P.v) + shift;
                    lnk += fx_troe(m.fx_troe, m.troe_df, m.troe, x.z, Ti, P.v, l0 - lnk + lM, ft, dt);
                }
            }
            if (kind != 1) lnk &= ~1ll;                     // bit 0 is the sign of the products
            L.f += lnk;
            double qq = fx_exp2<true>(L.f, ft) - fx_exp2<true>(L.f + L.r, ft);
            if (z <= 0 && (z == 0 || (kind == 2 && !MIXED))) qq = z == 0 ? 0.0 : __longlong_as_double(0x7ff8000000000000ll);
            if constexpr (MIXED) {
                if (kind == 2) qq = fx_times_float(qq, Ff);
                if (big) qq = fx_shift_edge(qq, (double)lnkf);
            } else if (big) {
                qq = fx_shift_edge(qq, __ldg(dlnA + (int)(r1.y >> 32 & 0xffff)));
            }
            *reinterpret_cast<double*>(sQ + q * 256) = qq;
        }
        __syncthreads();
        const uint32_t* spec = reinterpret_cast<const uint32_t*>(im + f.image_spec);
        const unsigned char* list = im + f.image_list;
#pragma unroll
        for (int j = 0; j < kFxOwn; ++j) {
            const int k = part + NP * j;
            if (k < K) w[j] = fx_gather(spec[k], list, sQ, w[j]);
        }
        fx_image_wait();
        __syncthreads();
    }

    // omega_k (or the source W_k omega_k / rho), sum_k h_k/RT omega_k and, for the sources,
    // c_p/R = sum_k Y_k/W_k c_p,k/R of this part's species
    const bool store = live && sS[kFxSum * 32] != 0;
    double h = 0.0, cpm = 0.0, inv_rho = 0.0;
    if constexpr (RHS) inv_rho = fx_exp2(-sS[kFxLrho * 32], ft);
    // (each part reads and writes its own species' rows, which the reactions are done with)
#pragma unroll
    for (int j = 0; j < kFxOwn; ++j)
        if (part + NP * j < K) *reinterpret_cast<double*>(sP + (part + NP * j) * kFxRow) = w[j];
    {
        const FxFrac u = fx_frac_T(Tb);
#pragma unroll 1
        for (int k = part; k < K; k += NP) {
            double o = *reinterpret_cast<const double*>(sP + k * kFxRow);
            const FxSpecies* sp = f.sp + k;
            const int64_t* c = fx_range(sp, Ti);
            const int ks = __ldg(&sp->k);
            h = fma(fx_to_d(fx_hRT(c, P, u)), o, h);
            if constexpr (RHS) {
                cpm = fma(Y[(int64_t)ks * ld + i] * __ldg(m.invW + ks), fx_to_d(fx_cpR(c, u)), cpm);
                o *= __ldg(m.W + ks) * inv_rho;
            }
            if (store) omega[(int64_t)ks * ld + i] = o;
        }
    }
    double* sR = reinterpret_cast<double*>(sQ);            // (the last chunk is done with)
    sR[(2 * part) * 32] = h;
    if constexpr (RHS) sR[(2 * part + 1) * 32] = cpm;
    __syncthreads();
    if (part != 0 || !live) return;
    for (int q = 1; q < NP; ++q) {
        h += sR[(2 * q) * 32];
        if constexpr (RHS) cpm += sR[(2 * q + 1) * 32];
    }
    const double hr = -kR * Ti * h;                        // heat release -sum_k h_k omega_k
    if (!store)
        hrr[i] = __longlong_as_double((long long)kFxSkip);
    else if constexpr (RHS)
        hrr[i] = hr * inv_rho / (kR * kFxCpScale * cpm);                // dT/dt = hrr / (rho c_p)
    else
        hrr[i] = hr;
}

template <int NP, bool RHS, bool MIXED>
cudaError_t launch_rates_fx_np(const DevMech& m, int64_t n, int64_t ld, const double* T, const double* p,
                               const double* Y, const double* dlnA, double* omega, double* hrr, cudaStream_t s) {
    auto kern = rates_fx_kernel<NP, RHS, MIXED>;
    const size_t smem = fx_smem(m.fxs[0], m.K, 256);
    const cudaError_t e = ensure_smem((const void*)kern, smem);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)((n + 31) / 32), 32 * NP, smem, s>>>(m, n, ld, T, p, Y, dlnA, omega, hrr);
    return cudaGetLastError();
}

template <bool RHS, bool MIXED>
cudaError_t launch_rates_fx(const DevMech& m, int64_t n, int64_t ld, const double* T, const double* p,
                            const double* Y, const double* dlnA, double* omega, double* hrr, cudaStream_t s) {
    switch (fx_parts(m.K)) {
        case 4: return launch_rates_fx_np<4, RHS, MIXED>(m, n, ld, T, p, Y, dlnA, omega, hrr, s);
        case 8: return launch_rates_fx_np<8, RHS, MIXED>(m, n, ld, T, p, Y, dlnA, omega, hrr, s);
        case 16: return launch_rates_fx_np<16, RHS, MIXED>(m, n, ld, T, p, Y, dlnA, omega, hrr, s);
        default: return launch_rates_fx_np<32, RHS, MIXED>(m, n, ld, T, p, Y, dlnA, omega, hrr, s);
    }
}

}  // namespace
}  // namespace nk
