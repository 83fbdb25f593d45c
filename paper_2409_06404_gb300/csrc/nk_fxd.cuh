// Derivative pieces of the fixed-point reaction kernels (JVP, VJP): tangent quantities are float
// pairs (they range over 2^+-120, where fixed point would lose the small ones), the state's
// logarithms and the temperature derivatives' coefficients 64-bit integers (nk_fx.cuh).
#pragma once

#include "nk_fxpt.cuh"

namespace nk {

// a double within 2^+-120 (or zero) as mantissa pair in +-[1, 2) and exponent, by integer operations
struct MantPair {
    dfl m;
    int e;
};
__device__ __forceinline__ MantPair mant_pair(double x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    MantPair r;
    r.e = (int)(b >> 52 & 0x7ff) - 1023;
    const unsigned sign = (unsigned)(b >> 32) & 0x80000000u;
    if ((b << 1) == 0) return {dfl{0.0f, 0.0f}, 0};
    // h: the mantissa rounded to 24 bits; l: the 29 bits left over, signed (at most half h's last place)
    const unsigned long long m = b & 0x000fffffffffffffull, t = (m + (1ull << 28)) >> 29;
    const float h = __uint_as_float((0x3f800000u + (unsigned)t) | sign);
    const float l = __fmul_rn((float)((int)(unsigned)m - (int)((unsigned)t << 29)), 0x1p-52f);
    r.m = dfl{h, __uint_as_float(__float_as_uint(l) ^ sign)};
    return r;
}
// v / y for doubles whose exponents differ by at most 120 (v may be zero), as a pair
__device__ __forceinline__ dfl quot_pair(double v, double y) {
    const MantPair a = mant_pair(v), b = mant_pair(y);
    const float s = b.m.h < 0.0f ? -1.0f : 1.0f;
    const dfl q = df_div(dfl{a.m.h * s, a.m.l * s}, dfl{b.m.h * s, b.m.l * s});
    return df_ldexp(q, a.e - b.e);
}
// a double within 2^+-100 (or zero) as a pair
__device__ __forceinline__ dfl split_pair(double v) {
    const MantPair a = mant_pair(v);
    return df_ldexp(a.m, a.e);
}
// v 2^s as a pair, for a double of any size below 2^100: what a pair cannot carry (below 2^-126)
// goes to zero
__device__ __forceinline__ dfl split_pair_scaled(double v, int s) {
    const MantPair a = mant_pair(v);
    return a.e + s < -126 ? dfl{0.0f, 0.0f} : df_ldexp(a.m, a.e + s);
}
// |y| in [2^-100, 2): a mass fraction the derivative kernels take
__device__ __forceinline__ bool fx_y_ok(double y) {
    const unsigned e = (unsigned)((unsigned long long)__double_as_longlong(y) >> 52) & 0x7ffu;
    return e - 923u <= 100u;
}
__device__ __forceinline__ dfl fxc_ln2() { return {0.693147182464599609375f, -1.9046542121259336e-09f}; }

// As fx_third_body, and d ln[M]: with [M] = rho' z, z = s + sum (eps - 1) Y/W, s = sum Y/W, at
// d rho/rho = arho and d(p/RT) = -theta p/RT it is
//   (arho (z - s) - theta s + sum (eps - 1) dY/W) / z,
// the sum in double (its terms are in the pairs' range, but where they cancel it may be of any size
// below that), the rest in pairs of z's unit.
__device__ __forceinline__ long long fx_third_body_d(const DevMech& m, int eff0, int eff1, const double* Y,
                                                     const double* vY, int64_t ld, int64_t i, long long sum, dfl theta,
                                                     dfl arho, const FxTab& t, long long& lM, dfl& dlnM) {
    const long long s = sum >> m.fx_eff_shift;
    long long z = s;
    double dz = 0.0;
    for (int j = eff0; j < eff1; ++j) {
        const FxEff* p = m.fx_eff + j;
        const longlong2 e = __ldg(reinterpret_cast<const longlong2*>(p));
        const int64_t at = (int64_t)(int)e.y * ld + i;
        const unsigned long long yb = (unsigned long long)__double_as_longlong(__ldg(Y + at));
        dz = fma(__ldg(&p->wd), __ldg(vY + at), dz);
        if ((yb << 1) != 0) {
            const long long g = fx_mul(e.x, fx_frac63(fx_half63(yb & 0x7fffffffffffffffull)));
            z += (long long)yb < 0 ? -g : g;
        }
    }
    lM = fx_log2_int((unsigned long long)(z > 0 ? z : z < 0 ? -z : 1ll), 60 - m.fx_eff_shift, t) + m.fx_lmaxw;
    dfl d = split_pair_scaled(dz, 12 - m.fx_eff_shift);
    d = df_fma(arho, fx_to_pair(z - s), d);
    d = df_add(d, df_neg(df_mul(theta, fx_to_pair(s))));
    dlnM = df_div(z < 0 ? df_neg(d) : d, fx_to_pair(z < 0 ? -z : z != 0 ? z : 1ll));
    return z;
}

// The Troe factor's logarithm and derivatives: phi = log2 of F P_r/(1 + P_r) as fx_troe forms it,
// px = d ln F/d ln P_r (with the P_r/(1 + P_r) part), pt = T d ln F/dT at constant P_r.  With
// D = u^2 + v^2 and rho = v^2/D: d rho = 2 u v (u dv - v du)/D^2, where
//   for d log2 P_r: u dv - v du = -log10(2) (0.14 u + v),
//   for d Lc:       u dv - v du = log10(2) (0.67 v - 1.1762 u)      (1.1762 = 1.27 - 0.14 0.67),
// and T d ln F_cent/dT = ln2 (sum of F_cent's terms times their exponents' T d/dT)/F_cent.
struct FxTroeD {
    long long phi;
    dfl px, pt;
};
static __device__ __noinline__ FxTroeD fx_troe_d(const FxTroe* fx, const float4* df, const TroeRec* d, int aux, double T,
                                                 FxFrac v, long long X, FxTab t, DfTab dt) {
    const long long* r = reinterpret_cast<const long long*>(fx + aux);
    const FxFrac u = fx_frac_T((unsigned long long)__double_as_longlong(T));
    long long Lc = 0;
    dfl cT{0.0f, 0.0f};                                   // T d ln F_cent/dT
    const int flags = (int)__ldg(r + 8);
    bool edge = !(flags & 1);
    const dfl one{1.0f, 0.0f};
    if (!edge) {
        const long long t3 = fx_mul(__ldg(r + 4), u), t1 = fx_mul(__ldg(r + 6), u);
        const unsigned long long e3 = fx_exp2_int(__ldg(r + 3) + t3, t), e1 = fx_exp2_int(__ldg(r + 5) + t1, t);
        unsigned long long Fc = e3 + e1;
        long long FT = fx_mul(2 * t3, fx_frac63(e3 << 3)) + fx_mul(2 * t1, fx_frac63(e1 << 3));
        if (flags & 2) {
            const long long t2 = fx_mul(__ldg(r + 7), v);
            const unsigned long long e2 = fx_exp2_int(t2, t);
            Fc += e2;
            FT -= fx_mul(2 * t2, fx_frac63(e2 << 3));
        }
        edge = Fc < 1ull << 48;
        if (edge) Fc = 1ull << 60;
        Lc = fx_log2_int(Fc, 60, t);
        const dfl f = fx_to_pair((long long)Fc);          // F_cent 2^12
        cT = df_mul(df_ldexp(df_div(fx_to_pair(FT), f), 12), fxc_ln2());
    }
    if (edge) {
        TPairs tp;
        tp.T = T;
        tp.Td = fx_T_pair(T);
        tp.invTd = fx_invT_pair(v);
        const TroeCent c = troe_cent(df, d, aux, tp, dt);
        Lc = fx_of_pair(df_mul(c.L, dfl{3.321928024291992f, 7.0595369580300144e-08f}));
        cT = df_mul(c.LT, dfc_ln10());
    }
    constexpr unsigned long long kLog10_2 = 0x268826A13EF3FDE6ull;
    constexpr unsigned long long k067 = 0x55C28F5C28F5C28Full, k027 = 0x228F5C28F5C28F5Cull, k014 = 0x11EB851EB851EB85ull;
    const dfl lam{0.3010300099849701f, -1.4320989122586137e-08f};                          // log10(2)
    const long long L10 = fx_scale(Lc, kLog10_2);
    const long long uu = fx_scale(X, kLog10_2) - (long long)(0.4 * 281474976710656.0) - fx_scale(L10, k067);
    const long long vv = (long long)(0.75 * 281474976710656.0) - L10 - fx_scale(L10, k027) - fx_scale(uu, k014);
    const dfl pu = fx_to_pair(uu), pv = fx_to_pair(vv), Lp = fx_to_pair(Lc);
    const dfl v2 = df_mul(pv, pv);
    const dfl iD = df_div(one, df_fma(pu, pu, v2));
    const dfl rho = df_mul(v2, iD);
    dfl w = df_mul(df_mul(df_mul(pu, iD), df_mul(pv, iD)), Lp);
    w = df_mul(dfl{2.0f * w.h, 2.0f * w.l}, lam);
    const unsigned long long zi = fx_exp2_int(X < 0 ? X : -X, t);
    const dfl z = df_ldexp(fx_to_pair((long long)zi), -12);
    const long long s = fx_log2_int((1ull << 60) + zi, 60, t);
    FxTroeD o;
    o.phi = fx_of_pair(df_mul(Lp, rho)) + (X < 0 ? X : 0ll) - s;
    // d ln F/d ln P_r: the broadening's part and 1/(1 + P_r)
    const dfl a = df_neg(df_fma(pu, df_neg(dfc_m0_14()), pv));
    o.px = df_fma(w, a, df_div(X < 0 ? one : z, df_add(one, z)));
    const dfl b = df_fma(pv, df_neg(dfc_m0_67()), df_neg(df_mul(pu, dfl{1.17620003223419189453125f, -3.2234190427971043e-08f})));
    o.pt = df_mul(df_fma(w, b, rho), cT);
    return o;
}

}  // namespace nk
