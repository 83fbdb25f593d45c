// Jacobian-vector product kernel on fixed-point logarithms (nk_fx.cuh, nk_fxpt.cuh, nk_fxd.cuh), with
// the rates kernel's layout.
//
// Per species a row holds log2 C_k, mu_k (as the rates kernel), r_k = d ln C_k = d rho/rho +
// dY_k/Y_k (a float pair), e_k = 1 - h_k/RT = T d mu_k/dT (natural units) and c_p,k/R, the last two
// as integers: a reaction's temperature derivatives are integer sums over its molecules where the
// pair kernel (k_jvp.cuh) evaluated three reaction polynomials.  With theta = dT/T,
// s = T d ln k/dT (53 species / 325 reactions, 512,000 points: 10.9 -> 7.1 ms; error against 64-bit
// sums 3e-13 -> 4e-14):
//   dq = q_f (theta s + sum_reactants r) - q_r (theta (s + sum nu e) + sum_products r).
#pragma once

#include "nk_fxd.cuh"

namespace nk {
namespace {

enum { kJvMu = 256, kJvR = 512, kJvE = 768, kJvCp = 1024 };
constexpr int kJvScalars = kFxScalars + 5;       // then theta, d rho/rho, rho as doubles, theta and d rho/rho as pairs

// Shared memory of a block; the form takes mechanisms for which it fits.
inline size_t jvp_fx_smem(const DevMech& m, bool omega) {
    const FxSet& f = m.fxs[1];
    const size_t red = (size_t)f.np * 5 * 256;             // the parts' sums at the end
    const size_t b = fx_smem(f, m.K, omega ? 512 : 256), q = (size_t)f.rows * (omega ? 512 : 256);
    return b + (kJvScalars - kFxScalars) * 256 + (red > q ? red - q : 0);
}
inline bool jvp_fx_fits(const DevMech& m, bool omega) {
    return m.fx_ok && m.fxs[1].np != 0 && jvp_fx_smem(m, omega) <= smem_limit();
}

// own: species per part at most.  Blocks with a point outside the form (the rates kernel's
// conditions, |Y_k| in [2^-100, 2), and the direction's values and quotients by Y_k in the pairs'
// range) leave kFxSkip in their points' d_hrr for the marked pass of k_jvp.cuh.
template <int NP, int OWN, int BLOCKS, bool OMEGA, bool RHS>
__global__ void __launch_bounds__(32 * NP, BLOCKS)
    jvp_fx_kernel(const DevMech m, const int64_t n, const int64_t ld, const double* __restrict__ T,
                  const double* __restrict__ p, const double* __restrict__ Y, const double* __restrict__ dlnA,
                  const double* __restrict__ vT, const double* __restrict__ vY, double* __restrict__ omega,
                  double* __restrict__ hrr, double* __restrict__ d_omega, double* __restrict__ d_hrr) {
    extern __shared__ __align__(16) unsigned char smem_fx[];
    const FxSet& f = m.fxs[1];
    unsigned char* im0 = smem_fx + kFxBase + kJvScalars * 256;
    const int K = m.K;
    const int lane = threadIdx.x & 31, part = threadIdx.x >> 5;
    const int64_t i0 = (int64_t)blockIdx.x * 32 + lane;
    const bool live = i0 < n;
    const int64_t i = live ? i0 : n - 1;
    long long* sS = reinterpret_cast<long long*>(smem_fx + kFxBase) + lane;
    double* sV = reinterpret_cast<double*>(sS) + kFxScalars * 32;                // theta, d rho/rho, rho
    float2* sVp = reinterpret_cast<float2*>(sV + 3 * 32);                        // theta, d rho/rho
    unsigned char* sP = im0 + 2 * f.image + lane * 8;
    unsigned char* sQ = sP + (size_t)(K + 1) * kFxDRow;
    constexpr int kQ = OMEGA ? 512 : 256;                                        // dq (and q) of a reaction

    // A block with a point outside the form leaves before its set-up, all its points marked: the marked
    // pass works by whole blocks, so it takes the others at no cost, where they would cost this pass
    // (one zero mass fraction in every block, 53 species, 262,144 points: 12.4 -> 9.0 ms, 8.7 of them the
    // marked pass).
    const double Ti = T[i], pi = p[i];
    const unsigned long long Tb = (unsigned long long)__double_as_longlong(Ti);
    {
        double y[OWN], v[OWN];                               // (all loads in flight at once)
#pragma unroll
        for (int j = 0; j < OWN; ++j) {
            y[j] = v[j] = 0.0;
            if (part + NP * j >= K) continue;
            const int64_t at = (int64_t)__ldg(&f.sp[part + NP * j].k) * ld + i;
            y[j] = Y[at];
            v[j] = vY[at];
        }
        bool bad = !fx_T_ok(Ti) || !fx_p_ok(pi);
        unsigned long long z = 0, zc = 0;
        double ds = 0.0;
#pragma unroll
        for (int j = 0; j < OWN; ++j) {
            if (part + NP * j >= K) break;
            const FxSpecies* sp = f.sp + part + NP * j;
            fx_add_fraction((unsigned long long)__double_as_longlong(y[j]), __ldg((const long long*)&sp->w), z, zc, bad);
            bad |= !(fx_y_ok(y[j]) && pair_range_ok(v[j]) && quot_range_ok(v[j], y[j]));
            ds = fma(v[j], __ldg(m.invW + __ldg(&sp->k)), ds);
        }
        reinterpret_cast<unsigned long long*>(sQ)[(3 * part) * 32] = z;
        reinterpret_cast<unsigned long long*>(sQ)[(3 * part + 1) * 32] = zc;
        reinterpret_cast<double*>(sQ)[(3 * part + 2) * 32] = ds;
        if (__syncthreads_or(bad) != 0) {
            if (part == 0 && live) d_hrr[i] = __longlong_as_double((long long)kFxSkip);
            return;
        }
    }
    fx_image_load(f, 0, im0);
    const FxTab ft = stage_fx_tables(reinterpret_cast<uint32_t*>(smem_fx), m.fx_tab);
    const DfTab dt = stage_df_tables(reinterpret_cast<float2*>(smem_fx + kFxTabBytes), m);
    __syncthreads();
    if (part == 0) {
        fx_point_scalars(m, Tb, pi, sS, ft);
        unsigned long long z = 0, zc = 0;
        double ds = 0.0;
        for (int q = 0; q < NP; ++q) {
            z += reinterpret_cast<unsigned long long*>(sQ)[(3 * q) * 32];
            zc += reinterpret_cast<unsigned long long*>(sQ)[(3 * q + 1) * 32];
            ds += reinterpret_cast<double*>(sQ)[(3 * q + 2) * 32];
        }
        bool bad = fx_sums_bad(z, zc);
        const long long ls = fx_log2_int(bad ? 1ull << 60 : z, 60, ft) + m.fx_lmaxw;
        const double theta = vT[i] / Ti, arho = -theta - ds * fx_exp2(-ls, ft);
        bad |= !(pair_range_ok(theta) && pair_range_ok(arho));
        const dfl th = bad ? dfl{0.0f, 0.0f} : split_pair(theta), ar = bad ? dfl{0.0f, 0.0f} : split_pair(arho);
        sV[0] = theta;
        sV[32] = arho;
        sV[64] = fx_exp2(bad ? 0 : sS[kFxLpRT * 32] - ls, ft);
        sVp[0] = make_float2(th.h, th.l);
        sVp[32] = make_float2(ar.h, ar.l);
        sS[kFxLrho * 32] = bad ? 0 : sS[kFxLpRT * 32] - ls;
        sS[kFxSum * 32] = bad ? 0 : (long long)z;
#pragma unroll
        for (int j = 0; j < kFxDRow / 256; ++j) *reinterpret_cast<long long*>(sP + K * kFxDRow + j * 256) = 0;
    }
    __syncthreads();
    // (the conditions on the point sums)
    if (__any_sync(0xffffffffu, sS[kFxSum * 32] == 0)) {
        if (part == 0 && live) d_hrr[i] = __longlong_as_double((long long)kFxSkip);
        fx_image_wait();
        return;
    }
    FxT P;
    P.lt = fx_frac63((unsigned long long)sS[kFxLT * 32] << 11);
    P.v = fx_frac63((unsigned long long)sS[kFxV * 32]);
    {
        const long long lrho = sS[kFxLrho * 32];
        const dfl ar = dfl_of(sVp[32]);
        const FxFrac u = fx_frac_T(Tb);
#pragma unroll 1
        for (int k = part; k < K; k += NP) {
            const FxSpecies* sp = f.sp + k;
            const int64_t at = (int64_t)__ldg(&sp->k) * ld + i;
            const double y = Y[at];
            unsigned char* row = sP + k * kFxDRow;
            const int64_t* c = fx_range(sp, Ti);
            const long long a = fx_log2_conc((unsigned long long)__double_as_longlong(y), __ldg((const long long*)&sp->lw) + lrho, ft);
            const dfl r = df_add(ar, quot_pair(vY[at], y));
            *reinterpret_cast<long long*>(row) = a;
            *reinterpret_cast<long long*>(row + kJvMu) = a + (fx_mu0(c, P, u) & ~1ll);
            *reinterpret_cast<float2*>(row + kJvR) = make_float2(r.h, r.l);
            *reinterpret_cast<long long*>(row + kJvE) = (1ll << kFxS) - fx_hRT(c, P, u);
            *reinterpret_cast<long long*>(row + kJvCp) = fx_cpR(c, u);
        }
    }
    fx_image_wait();
    __syncthreads();

    double w[OWN], wq[OMEGA ? OWN : 1];
#pragma unroll
    for (int j = 0; j < OWN; ++j) w[j] = 0.0;
    if constexpr (OMEGA) {
#pragma unroll
        for (int j = 0; j < OWN; ++j) wq[j] = 0.0;
    }
    double acc_h = 0.0, acc_cp = 0.0, acc_dh = 0.0;      // sums over reactions of q dH/RT, q dCp/R, dq dH/RT
    for (int c = 0; c < f.nchunk; ++c) {
        const unsigned char* im = im0 + (c & 1) * f.image;
        fx_image_load(f, c + 1, im0 + ((c + 1) & 1) * f.image);
        const int q1 = im[f.image_parts + part + 1];
#pragma unroll 1
        for (int q = im[f.image_parts + part]; q < q1; ++q) {
            const longlong2* rec = reinterpret_cast<const longlong2*>(im + q * (int)sizeof(FxRxn));
            const longlong2 r0 = rec[0], r1 = rec[1];
            const int info = (int)r1.y;
            FxRate L{0, 0};
            long long E = 0, Cp = 0;                     // sum nu e, sum nu c_p/R
            dfl gf, gr;                                  // sum over reactants, products of r
            {
                const uint32_t* off = reinterpret_cast<const uint32_t*>(rec + 2);
                const int nr = info & 15, np = info >> 4 & 15;
                const unsigned char* a = sP + off[0];
                fx_reac(a, L);
                E -= *reinterpret_cast<const long long*>(a + kJvE);
                Cp -= *reinterpret_cast<const long long*>(a + kJvCp);
                gf = dfl_of(*reinterpret_cast<const float2*>(a + kJvR));
#pragma unroll 1
                for (int e = 1; e < nr; ++e) {
                    a = sP + off[e];
                    fx_reac(a, L);
                    E -= *reinterpret_cast<const long long*>(a + kJvE);
                    Cp -= *reinterpret_cast<const long long*>(a + kJvCp);
                    gf = df_add(gf, dfl_of(*reinterpret_cast<const float2*>(a + kJvR)));
                }
                a = sP + off[4];
                fx_prod(a, L);
                E += *reinterpret_cast<const long long*>(a + kJvE);
                Cp += *reinterpret_cast<const long long*>(a + kJvCp);
                gr = dfl_of(*reinterpret_cast<const float2*>(a + kJvR));
#pragma unroll 1
                for (int e = 1; e < np; ++e) {
                    a = sP + off[4 + e];
                    fx_prod(a, L);
                    E += *reinterpret_cast<const long long*>(a + kJvE);
                    Cp += *reinterpret_cast<const long long*>(a + kJvCp);
                    gr = df_add(gr, dfl_of(*reinterpret_cast<const float2*>(a + kJvR)));
                }
            }
            const long long ea = fx_mul(r1.x, P.v);      // -log2(e) Ea/RT
            long long lnk = r0.x + fx_mul(r0.y, P.lt) + ea;
            const long long s = (r0.y >> 5) - fx_scale(ea, 0x58B90BFBE8E7BCD6ull);   // beta + Ea/RT (ln2 2^63)
            const dfl th = dfl_of(sVp[0]);
            long long shift = 0;
            bool big = false;
            if (dlnA) {
                const double d = __ldg(dlnA + (int)(r1.y >> 32 & 0xffff));
                big = ((unsigned)__double2hiint(d) & 0x7fffffffu) >= 0x40a00000u;
                if (!big) shift = fx_log2e_times(d);
                lnk += shift;
            }
            long long z = 1;
            const int kind = info >> 8 & 3;
            if (kind != 0) {
                const int4 x = __ldg(reinterpret_cast<const int4*>(m.fx_extra + (info >> 16)));
                long long lM;
                dfl dM;
                z = fx_third_body_d(m, x.x, x.y, Y, vY, ld, i, sS[kFxSum * 32], th, dfl_of(sVp[32]), ft, lM, dM);
                lM += sS[kFxLrho * 32];
                if (kind == 1) {
                    lnk = ((lnk + lM) & ~1ll) + (long long)(z < 0);
                    gf = df_add(gf, dM);
                    gr = df_add(gr, dM);
                } else {
                    const longlong2* tr = reinterpret_cast<const longlong2*>(m.fx_troe + x.z);
                    const longlong2 a = __ldg(tr), b = __ldg(tr + 1);
                    const long long e0 = fx_mul(b.x, P.v);
                    const long long l0 = a.x + fx_mul(a.y, P.lt) + e0 + shift;
                    const FxTroeD t = fx_troe_d(m.fx_troe, m.troe_df, m.troe, x.z, Ti, P.v, l0 - lnk + lM, ft, dt);
                    lnk += t.phi;
                    // d ln F = px d ln P_r + pt theta, d ln P_r = (s_0 - s) theta + d ln[M]
                    const long long s0 = (a.y >> 5) - fx_scale(e0, 0x58B90BFBE8E7BCD6ull);
                    const dfl g = df_fma(t.px, df_fma(fx_to_pair(s0 - s), th, dM), df_mul(t.pt, th));
                    gf = df_add(gf, g);
                    gr = df_add(gr, g);
                }
            }
            if (kind != 1) lnk &= ~1ll;
            L.f += lnk;
            double qf = fx_exp2<true>(L.f, ft), qr = fx_exp2<true>(L.f + L.r, ft);
            if (z <= 0 && (z == 0 || kind == 2)) qf = qr = z == 0 ? 0.0 : __longlong_as_double(0x7ff8000000000000ll);
            if (big) {
                const double d = __ldg(dlnA + (int)(r1.y >> 32 & 0xffff));
                qf = fx_shift_edge(qf, d);
                qr = fx_shift_edge(qr, d);
            }
            const double Gf = df_to_d(df_fma(fx_to_pair(s), th, gf)), Gr = df_to_d(df_fma(fx_to_pair(s + E), th, gr));
            const double qq = qf - qr;
            const double dq = fma(qf, Gf, -qr * Gr);
            acc_cp = fma(qq, fx_to_d(Cp), acc_cp);
            if constexpr (OMEGA || RHS) acc_h = fma(qq, fx_to_d(-E + ((long long)(((info >> 4) & 15) - (info & 15)) << kFxS)), acc_h);
            *reinterpret_cast<double*>(sQ + q * kQ) = RHS ? fma(-sV[32], qq, dq) : dq;
            if constexpr (OMEGA) *reinterpret_cast<double*>(sQ + q * kQ + 256) = qq;
        }
        __syncthreads();
        const uint32_t* spec = reinterpret_cast<const uint32_t*>(im + f.image_spec);
        const unsigned char* list = im + f.image_list;
#pragma unroll
        for (int j = 0; j < OWN; ++j) {
            const int k = part + NP * j;
            if (k < K) {
                w[j] = fx_gather<kQ / 256>(spec[k], list, sQ, w[j]);
                if constexpr (OMEGA) wq[j] = fx_gather<2>(spec[k], list, sQ + 256, wq[j]);
            }
        }
        fx_image_wait();
        __syncthreads();
    }

    // d omega_k (sources: W_k (d omega_k - omega_k d rho/rho)/rho) and sum_k h_k/RT of it
    const double arho = sV[32], rho = sV[64];
    double cpm = 0.0, dcpm = 0.0, inv_rho = 0.0;
    if constexpr (RHS) inv_rho = 1.0 / rho;
#pragma unroll
    for (int j = 0; j < OWN; ++j)
        if (part + NP * j < K) {
            *reinterpret_cast<double*>(sP + (part + NP * j) * kFxDRow) = w[j];
            if constexpr (OMEGA) *reinterpret_cast<double*>(sP + (part + NP * j) * kFxDRow + kJvMu) = wq[j];
        }
#pragma unroll 1
    for (int k = part; k < K; k += NP) {
        const FxSpecies* sp = f.sp + k;
        const int ks = __ldg(&sp->k);
        const unsigned char* row = sP + k * kFxDRow;
        double dw = *reinterpret_cast<const double*>(row);
        double o = 0.0;
        if constexpr (OMEGA) o = *reinterpret_cast<const double*>(row + kJvMu);
        acc_dh = fma(fx_to_d((1ll << kFxS) - *reinterpret_cast<const long long*>(row + kJvE)), dw, acc_dh);
        if constexpr (RHS) {
            const double cpk = fx_to_d(*reinterpret_cast<const long long*>(row + kJvCp));      // (over kFxCpScale)
            const double iw = __ldg(m.invW + ks);
            const double yk = Y[(int64_t)ks * ld + i] * iw, vk = vY[(int64_t)ks * ld + i] * iw;
            cpm = fma(yk, cpk, cpm);
            dcpm = fma(vk, cpk, fma(yk * (nasa_dcpR_dT(nasa_range(m, ks, Ti), Ti) * (1.0 / kFxCpScale)), vT[i], dcpm));
            const double wr = __ldg(m.W + ks) * inv_rho;
            dw *= wr;
            o *= wr;
        }
        if (live) {
            d_omega[(int64_t)ks * ld + i] = dw;
            if (OMEGA && omega) omega[(int64_t)ks * ld + i] = o;
        }
    }
    double* sR = reinterpret_cast<double*>(sQ);
    sR[(5 * part) * 32] = acc_h;
    sR[(5 * part + 1) * 32] = acc_cp;
    sR[(5 * part + 2) * 32] = acc_dh;
    if constexpr (RHS) {
        sR[(5 * part + 3) * 32] = cpm;
        sR[(5 * part + 4) * 32] = dcpm;
    }
    __syncthreads();
    if (part != 0 || !live) return;
    for (int q = 1; q < NP; ++q) {
        acc_h += sR[(5 * q) * 32];
        acc_cp += sR[(5 * q + 1) * 32];
        acc_dh += sR[(5 * q + 2) * 32];
        if constexpr (RHS) {
            cpm += sR[(5 * q + 3) * 32];
            dcpm += sR[(5 * q + 4) * 32];
        }
    }
    // d hrr = -R (dT sum_k c_p,k/R omega_k + T sum_k h_k/RT d omega_k)
    const double hr = -kR * Ti * acc_h;
    if constexpr (RHS) acc_dh = fma(arho, acc_h, acc_dh);        // (the sums hold d omega - omega d rho/rho)
    const double dhr = -kR * fma(vT[i], acc_cp * kFxCpScale, Ti * acc_dh);
    if constexpr (RHS) {
        const double irc = inv_rho / (kR * kFxCpScale * cpm);    // 1 / (rho c_p)
        d_hrr[i] = irc * fma(-hr, arho + dcpm / cpm, dhr);
        if (hrr) hrr[i] = hr * irc;
    } else {
        d_hrr[i] = dhr;
        if (hrr) hrr[i] = hr;
    }
}

template <int NP, int OWN, int BLOCKS, bool OMEGA, bool RHS>
cudaError_t launch_jvp_fx_np(const DevMech& m, int64_t n, int64_t ld, const double* T, const double* p, const double* Y,
                             const double* dlnA, const double* vT, const double* vY, double* omega, double* hrr,
                             double* d_omega, double* d_hrr, cudaStream_t s) {
    auto kern = jvp_fx_kernel<NP, OWN, BLOCKS, OMEGA, RHS>;
    const size_t smem = jvp_fx_smem(m, OMEGA);
    const cudaError_t e = ensure_smem((const void*)kern, smem);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)((n + 31) / 32), 32 * NP, smem, s>>>(m, n, ld, T, p, Y, dlnA, vT, vY, omega, hrr, d_omega, d_hrr);
    return cudaGetLastError();
}

template <bool OMEGA, bool RHS>
cudaError_t launch_jvp_fx(const DevMech& m, int64_t n, int64_t ld, const double* T, const double* p, const double* Y,
                          const double* dlnA, const double* vT, const double* vY, double* omega, double* hrr,
                          double* d_omega, double* d_hrr, cudaStream_t s) {
    switch (m.fxs[1].np) {
        case 4: return launch_jvp_fx_np<4, 8, 6, OMEGA, RHS>(m, n, ld, T, p, Y, dlnA, vT, vY, omega, hrr, d_omega, d_hrr, s);
        case 12: return launch_jvp_fx_np<12, 6, 2, OMEGA, RHS>(m, n, ld, T, p, Y, dlnA, vT, vY, omega, hrr, d_omega, d_hrr, s);
        default: return launch_jvp_fx_np<24, 6, 1, OMEGA, RHS>(m, n, ld, T, p, Y, dlnA, vT, vY, omega, hrr, d_omega, d_hrr, s);
    }
}

}  // namespace
}  // namespace nk
