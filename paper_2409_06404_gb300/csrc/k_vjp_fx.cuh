// Vector-Jacobian product kernel on fixed-point logarithms (nk_fx.cuh, nk_fxpt.cuh, nk_fxd.cuh): the
// transpose of k_jvp_fx.cuh, with the same rows (bar_omega_k as a pair in place of r_k).
//
// A reaction's cotangent qbar_r = sum nu bar_omega - bar_hrr R T sum nu h/RT gives its two terms
// F_r = qbar_r q_f and B_r = -qbar_r q_r (cotangents of ln q_f and ln q_r), which are staged per chunk;
// a species then sums S_k = Cbar_k C_k = sum over its reactant molecules F_r + over its product
// molecules B_r + Y_k sum over its efficiencies w X_r, X_r = (F_r + B_r) px/([M]/rho') (px = 1 for
// third-body reactions), and the ln A gradient of a reaction is the sum of F + B over the block's
// points, each lane summing one reaction's row.  A persistent grid walks the tiles of 32 points.
// Rates and their gradients through autograd, 53 species / 325 reactions, 200,003 points: 8.8 -> 5.3
// ms (of which the rates 2.1 -> 1.3); error against 64-bit sums 3e-13 -> 6e-14.
#pragma once

#include "nk_fxd.cuh"

namespace nk {
namespace {

enum { kVjMu = 256, kVjW = 512, kVjE = 768, kVjCp = 1024 };
constexpr int kVjScalars = kFxScalars;

inline size_t vjp_fx_smem(const DevMech& m, bool want_g) {
    const FxSet& f = m.fxs[1];
    return fx_smem(f, m.K, 512) + (size_t)f.xrows * 256 + (want_g ? (size_t)((m.R + 1) & ~1) * 8 : 0);
}
inline bool vjp_fx_fits(const DevMech& m) { return m.fx_ok && m.fxs[1].np != 0 && vjp_fx_smem(m, true) <= smem_limit(); }

// Tiles with a point outside the form (the rates kernel's conditions, |Y_k| in [2^-100, 2),
// bar_omega_k in the pairs' range) leave kFxSkip in their points' gT for the marked passes of k_vjp.cu
// and add nothing to the ln A sums.
template <int NP, int OWN, int BLOCKS, bool WANT_G, bool HB>
__global__ void __launch_bounds__(32 * NP, BLOCKS)
    vjp_fx_kernel(const DevMech m, const int64_t n, const int64_t ld, const double* __restrict__ T,
                  const double* __restrict__ p, const double* __restrict__ Y, const double* __restrict__ dlnA,
                  const double* __restrict__ bar_omega, const double* __restrict__ bar_hrr, double* __restrict__ gT,
                  double* __restrict__ gY, double* __restrict__ ws) {
    extern __shared__ __align__(16) unsigned char smem_fx[];
    const FxSet& f = m.fxs[1];
    unsigned char* im0 = smem_fx + kFxBase + kVjScalars * 256;
    const FxTab ft = stage_fx_tables(reinterpret_cast<uint32_t*>(smem_fx), m.fx_tab);
    const DfTab dt = stage_df_tables(reinterpret_cast<float2*>(smem_fx + kFxTabBytes), m);
    const int K = m.K, R = m.R;
    const int lane = threadIdx.x & 31, part = threadIdx.x >> 5;
    long long* sS = reinterpret_cast<long long*>(smem_fx + kFxBase) + lane;
    unsigned char* sP = im0 + 2 * f.image + lane * 8;
    unsigned char* sQ = sP + (size_t)(K + 1) * kFxDRow;                          // F, B of a reaction
    const size_t qb = (size_t)f.rows * 512, pb = (size_t)f.np * 3 * 256;
    unsigned char* sX = sQ + (qb > pb ? qb : pb);                                // X of third-body and Troe
    double* gw = reinterpret_cast<double*>(sX - lane * 8 + (size_t)f.xrows * 256);   // ln A sums, device order
    if (WANT_G)
        for (int r = threadIdx.x; r < R; r += 32 * NP) gw[r] = 0.0;

    for (int64_t tile = blockIdx.x; tile * 32 < n; tile += gridDim.x) {
        const int64_t i0 = tile * 32 + lane;
        const bool live = i0 < n;
        const int64_t i = live ? i0 : n - 1;
        __syncthreads();                                  // the tables; the last tile's sums are read
        fx_image_load(f, 0, im0);
        const double Ti = T[i], pi = p[i];
        const unsigned long long Tb = (unsigned long long)__double_as_longlong(Ti);
        {
            bool bad = !fx_T_ok(Ti) || !fx_p_ok(pi);
            unsigned long long z = 0, zc = 0;
#pragma unroll 1
            for (int k = part; k < K; k += NP) {
                const FxSpecies* sp = f.sp + k;
                const int64_t at = (int64_t)__ldg(&sp->k) * ld + i;
                const double y = Y[at];
                fx_add_fraction((unsigned long long)__double_as_longlong(y), __ldg((const long long*)&sp->w), z, zc, bad);
                bad |= !(fx_y_ok(y) && pair_range_ok(bar_omega[at]));
            }
            if (part == 0) fx_point_scalars(m, Tb, pi, sS, ft);
            reinterpret_cast<unsigned long long*>(sQ)[(2 * part) * 32] = z;
            reinterpret_cast<unsigned long long*>(sQ)[(2 * part + 1) * 32] = zc;
            // a tile with a point outside the form is left to the marked passes, all its points marked
            // (as in k_jvp_fx.cuh)
            if (__syncthreads_or(bad) != 0) {
                if (live && part == 0) gT[i] = __longlong_as_double((long long)kFxSkip);
                fx_image_wait();
                continue;
            }
        }
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
                if (live && part == 0) gT[i] = __longlong_as_double((long long)kFxSkip);
                fx_image_wait();
                continue;
            }
            const long long lrho = sS[kFxLpRT * 32] - fx_log2_int(z, 60, ft) - m.fx_lmaxw;
            const FxFrac u = fx_frac_T(Tb);
#pragma unroll 1
            for (int k = part; k < K; k += NP) {
                const FxSpecies* sp = f.sp + k;
                const int64_t at = (int64_t)__ldg(&sp->k) * ld + i;
                unsigned char* row = sP + k * kFxDRow;
                const int64_t* c = fx_range(sp, Ti);
                const long long a = fx_log2_conc((unsigned long long)__double_as_longlong(Y[at]), __ldg((const long long*)&sp->lw) + lrho, ft);
                const dfl w = split_pair(bar_omega[at]);
                *reinterpret_cast<long long*>(row) = a;
                *reinterpret_cast<long long*>(row + kVjMu) = a + (fx_mu0(c, P, u) & ~1ll);
                *reinterpret_cast<float2*>(row + kVjW) = make_float2(w.h, w.l);
                *reinterpret_cast<long long*>(row + kVjE) = (1ll << kFxS) - fx_hRT(c, P, u);
                if constexpr (HB) *reinterpret_cast<long long*>(row + kVjCp) = fx_cpR(c, u);
            }
            if (part == 0) {
                sS[kFxLrho * 32] = lrho;
                sS[kFxSum * 32] = (long long)z;
            }
        }
        const double hbRT = HB ? bar_hrr[i] * (kR * Ti) : 0.0, hbCp = -hbRT * kFxCpScale;
        fx_image_wait();
        __syncthreads();

        double w[OWN];
#pragma unroll
        for (int j = 0; j < OWN; ++j) w[j] = 0.0;
        double Tbar = 0.0;                               // T times the temperature cotangent at fixed C_k
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
                long long E = 0, Cp = 0;                 // sum nu e, sum nu c_p/R
                dfl ws_;                                 // sum nu bar_omega
                {
                    const uint32_t* off = reinterpret_cast<const uint32_t*>(rec + 2);
                    const int nr = info & 15, np = info >> 4 & 15;
                    const unsigned char* a = sP + off[4];
                    fx_prod(a, L);
                    E += *reinterpret_cast<const long long*>(a + kVjE);
                    if constexpr (HB) Cp += *reinterpret_cast<const long long*>(a + kVjCp);
                    ws_ = dfl_of(*reinterpret_cast<const float2*>(a + kVjW));
#pragma unroll 1
                    for (int e = 1; e < np; ++e) {
                        a = sP + off[4 + e];
                        fx_prod(a, L);
                        E += *reinterpret_cast<const long long*>(a + kVjE);
                        if constexpr (HB) Cp += *reinterpret_cast<const long long*>(a + kVjCp);
                        ws_ = df_add(ws_, dfl_of(*reinterpret_cast<const float2*>(a + kVjW)));
                    }
#pragma unroll 1
                    for (int e = 0; e < nr; ++e) {
                        a = sP + off[e];
                        fx_reac(a, L);
                        E -= *reinterpret_cast<const long long*>(a + kVjE);
                        if constexpr (HB) Cp -= *reinterpret_cast<const long long*>(a + kVjCp);
                        ws_ = df_add(ws_, df_neg(dfl_of(*reinterpret_cast<const float2*>(a + kVjW))));
                    }
                }
                double qbar = live ? df_to_d(ws_) : 0.0;
                if constexpr (HB) {
                    const long long dH = ((long long)((info >> 4 & 15) - (info & 15)) << kFxS) - E;
                    if (live) qbar = fma(-hbRT, fx_to_d(dH), qbar);
                }
                const long long ea = fx_mul(r1.x, P.v);  // -log2(e) Ea/RT
                long long lnk = r0.x + fx_mul(r0.y, P.lt) + ea;
                long long s = (r0.y >> 5) - fx_scale(ea, 0x58B90BFBE8E7BCD6ull);     // beta + Ea/RT
                long long shift = 0;
                bool big = false;
                if (dlnA) {
                    const double d = __ldg(dlnA + (int)(r1.y >> 32 & 0xffff));
                    big = ((unsigned)__double2hiint(d) & 0x7fffffffu) >= 0x40a00000u;
                    if (!big) shift = fx_log2e_times(d);
                    lnk += shift;
                }
                long long z = 1;
                dfl px{1.0f, 0.0f};
                const int kind = info >> 8 & 3;
                if (kind != 0) {
                    const int4 x = __ldg(reinterpret_cast<const int4*>(m.fx_extra + (info >> 16)));
                    long long lM;
                    z = fx_third_body(m, x.x, x.y, Y, ld, i, sS[kFxSum * 32], ft, lM);
                    lM += sS[kFxLrho * 32];
                    if (kind == 1) {
                        lnk = ((lnk + lM) & ~1ll) + (long long)(z < 0);
                    } else {
                        const longlong2* tr = reinterpret_cast<const longlong2*>(m.fx_troe + x.z);
                        const longlong2 a = __ldg(tr), b = __ldg(tr + 1);
                        const long long e0 = fx_mul(b.x, P.v);
                        const long long l0 = a.x + fx_mul(a.y, P.lt) + e0 + shift;
                        const FxTroeD t = fx_troe_d(m.fx_troe, m.troe_df, m.troe, x.z, Ti, P.v, l0 - lnk + lM, ft, dt);
                        lnk += t.phi;
                        const long long s0 = (a.y >> 5) - fx_scale(e0, 0x58B90BFBE8E7BCD6ull);
                        px = t.px;
                        s += fx_of_pair(df_fma(px, fx_to_pair(s0 - s), t.pt));   // with T d ln F/dT
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
                if (!live) qf = qr = 0.0;
                const double F = qbar * qf, B = -qbar * qr;
                const double G = F + B;
                Tbar = fma(G, fx_to_d(s), Tbar);
                Tbar = fma(B, fx_to_d(E), Tbar);
                if constexpr (HB) Tbar = fma(hbCp * (qf - qr), fx_to_d(Cp), Tbar);
                if (kind != 0) {
                    // X = G px rho'/[M] (z in units 2^(eff_shift - 60)); the p/(RT) part of [M]
                    double X = 0.0;
                    if (z != 0 && live) {
                        const dfl iz = df_div(px, fx_to_pair(z < 0 ? -z : z));
                        X = G * (z < 0 ? -df_to_d(iz) : df_to_d(iz));                // times 2^-48 of z's unit
                    }
                    Tbar = fma(-X, fx_to_d(sS[kFxSum * 32] >> m.fx_eff_shift), Tbar);
                    // times 2^(60 - 48 - eff_shift): the efficiency terms' Y w come in units of 1
                    *reinterpret_cast<double*>(sX + (info >> 10 & 63) * 256) =
                        X * __hiloint2double((1023 + 12 - m.fx_eff_shift) << 20, 0);
                }
                *reinterpret_cast<double*>(sQ + q * 512) = F;
                *reinterpret_cast<double*>(sQ + q * 512 + 256) = B;
            }
            __syncthreads();
            const uint32_t* spec = reinterpret_cast<const uint32_t*>(im + f.image_spec);
            const unsigned char* list = im + f.image_list;
            const uint32_t* eff = reinterpret_cast<const uint32_t*>(im + f.image_eff);
#pragma unroll
            for (int j = 0; j < OWN; ++j) {
                const int k = part + NP * j;
                if (k < K) {
                    const uint32_t wd = spec[k];
                    const unsigned char* l = list + (wd >> 15 & ~1u);
                    const unsigned char* e = l + (wd >> 7 & 510u);
                    double a = w[j];
#pragma unroll 1
                    for (; l != e; l += 2) a += *reinterpret_cast<const double*>(sQ + 256 + 2 * *reinterpret_cast<const uint16_t*>(l));
                    e += (wd & 255u) * 2;
#pragma unroll 1
                    for (; l != e; l += 2) a += *reinterpret_cast<const double*>(sQ + 2 * *reinterpret_cast<const uint16_t*>(l));
                    const uint32_t we = eff[k];
                    if ((we & 255u) != 0) {
                        const FxEffTerm* t = reinterpret_cast<const FxEffTerm*>(im + f.image_effl) + (we >> 8);
                        double b = 0.0;
#pragma unroll 1
                        for (int e2 = 0; e2 < (int)(we & 255u); ++e2)
                            b = fma(t[e2].w, *reinterpret_cast<const double*>(sX + t[e2].x * 256), b);
                        a = fma(b, Y[(int64_t)__ldg(&f.sp[k].k) * ld + i], a);
                    }
                    w[j] = a;
                }
            }
            if (WANT_G) {
                // four lanes sum a row over the points, eight columns each (the rows, 512 bytes apart, start
                // at different columns: two lanes a bank at most), then over the four
                const int rows = im[f.image_parts + NP], g = lane >> 2, h = lane & 3;
                for (int r8 = part * 8; r8 < rows; r8 += NP * 8) {
                    const int row = min(r8 + g, rows - 1);
                    const double* q = reinterpret_cast<const double*>(sQ - lane * 8 + row * 512);
                    double a = 0.0;
#pragma unroll 4
                    for (int c2 = 0; c2 < 8; ++c2) {
                        const int col = h * 8 + ((c2 + g) & 7);
                        a += q[col] + q[32 + col];
                    }
                    a += __shfl_xor_sync(0xffffffffu, a, 1);
                    a += __shfl_xor_sync(0xffffffffu, a, 2);
                    if (h == 0 && r8 + g < rows) gw[reinterpret_cast<const FxRxn*>(im)[row].orig >> 16] += a;
                }
            }
            fx_image_wait();
            __syncthreads();
        }

        // sum_k S_k and T Tbar over the parts
        double cc = 0.0;
#pragma unroll
        for (int j = 0; j < OWN; ++j)
            if (part + NP * j < K) {
                cc += w[j];
                *reinterpret_cast<double*>(sP + (part + NP * j) * kFxDRow) = w[j];
            }
        double* sR = reinterpret_cast<double*>(sQ);
        sR[(2 * part) * 32] = cc;
        sR[(2 * part + 1) * 32] = Tbar;
        __syncthreads();
        cc = sR[0];
        Tbar = sR[32];
        for (int q = 1; q < NP; ++q) {
            cc += sR[(2 * q) * 32];
            Tbar += sR[(2 * q + 1) * 32];
        }
        // C_k = rho y_k, rho = p/(R T s), s = sum y_k: rho's cotangent through T and every Y_k
        if (live && part == 0) gT[i] = (Tbar - cc) / Ti;
        if (live) {
            const double sbar = -cc * fx_exp2(sS[kFxLrho * 32] - sS[kFxLpRT * 32], ft);      // -cc/s
#pragma unroll 1
            for (int k = part; k < K; k += NP) {
                const int ks = __ldg(&f.sp[k].k);
                const int64_t at = (int64_t)ks * ld + i;
                const double y = Y[at], S = *reinterpret_cast<const double*>(sP + k * kFxDRow);
                gY[at] = fma(S, y < 0.0 ? -recip_nr(-y) : recip_nr(y), __ldg(m.invW + ks) * sbar);
            }
        }
    }
    if (WANT_G) {
        __syncthreads();
        for (int r = threadIdx.x; r < R; r += 32 * NP) ws[(size_t)blockIdx.x * R + r] = gw[r];
    }
}

// Blocks of the persistent grid per SM, and the kernel, for the mechanism's parts.
inline int vjp_fx_blocks(const DevMech& m) { return m.fxs[1].np == 4 ? 6 : m.fxs[1].np == 12 ? 2 : 1; }

template <bool WANT_G, bool HB>
cudaError_t launch_vjp_fx(const DevMech& m, int64_t grid, int64_t n, int64_t ld, const double* T, const double* p,
                          const double* Y, const double* dlnA, const double* bar_omega, const double* bar_hrr,
                          double* gT, double* gY, double* ws, cudaStream_t s) {
    const size_t smem = vjp_fx_smem(m, WANT_G);
    const int np = m.fxs[1].np;
    auto kern = np == 4 ? vjp_fx_kernel<4, 8, 6, WANT_G, HB> : np == 12 ? vjp_fx_kernel<12, 6, 2, WANT_G, HB>
                                                                       : vjp_fx_kernel<24, 6, 1, WANT_G, HB>;
    const cudaError_t e = ensure_smem((const void*)kern, smem);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)grid, 32 * np, smem, s>>>(m, n, ld, T, p, Y, dlnA, bar_omega, bar_hrr, gT, gY, ws);
    return cudaGetLastError();
}

}  // namespace
}  // namespace nk
