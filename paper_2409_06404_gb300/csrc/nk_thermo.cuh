// NASA-7 species properties from 64-bit integer polynomials (FxThermo), for kernels the FP64 pipe
// would bound: c_p, h and g of a species take 15 multiply-adds, which cost 64 issue slots each as
// FP64 operations on GB300 and about 8 as integer ones (fx_mul: three 32-bit multiplications).  The
// integers are finer than a double's last bit, so the rounded results are at least as accurate.
#pragma once

#include "nk_fx.cuh"
#include "nk_internal.cuh"

namespace nk {

// T's fractions for the two ranges (64 <= T < 4096, else ok is false) and ln(T)/16
struct ThT {
    FxFrac lo, hi, ln;
    bool ok;
};
__device__ __forceinline__ ThT th_fractions(const DevMech& m, double T, double lnT) {
    ThT t;
    const unsigned long long b = (unsigned long long)__double_as_longlong(T), l = (unsigned long long)__double_as_longlong(lnT);
    t.ok = m.th_lo != 0 && (long long)b >= 0x4050000000000000ll && (long long)b < 0x40afffffffc00000ll;
    const unsigned long long mt = (b & 0x000fffffffffffffull) | 0x0010000000000000ull;
    const int e = (int)(b >> 52) - 1023;                        // T = mt 2^(e - 52), e in 6..11
    t.hi = fx_frac63(mt << ((e - 1) & 63));                     // T/2^12 = mt 2^(e - 64): times 2^63
    t.lo = fx_frac63(mt << ((e + 11 - m.th_lo) & 63));          // T/2^th_lo (used for T <= T_mid < 2^th_lo)
    const int el = (int)(l >> 52) - 1023;                       // ln T in [4, 8.4)
    t.ln = fx_frac63(((l & 0x000fffffffffffffull) | 0x0010000000000000ull) << ((el + 7) & 63));
    return t;
}
__device__ __forceinline__ long long th_c(const int64_t* c, int j) { return __ldg((const long long*)c + j); }

__device__ __forceinline__ double th_cp(const int64_t* c, FxFrac u, int s) {
    long long t = th_c(c, 4);
    t = th_c(c, 3) + fx_mul(t, u);
    t = th_c(c, 2) + fx_mul(t, u);
    t = th_c(c, 1) + fx_mul(t, u);
    return fx_round_d(th_c(c, 0) + fx_mul(t, u), s);
}
__device__ __forceinline__ double th_h(const int64_t* c, FxFrac u, int s) {
    long long t = th_c(c, 10);
    t = th_c(c, 9) + fx_mul(t, u);
    t = th_c(c, 8) + fx_mul(t, u);
    t = th_c(c, 7) + fx_mul(t, u);
    t = th_c(c, 6) + fx_mul(t, u);
    return fx_round_d(th_c(c, 5) + fx_mul(t, u), s);
}
__device__ __forceinline__ double th_g(const int64_t* c, FxFrac u, FxFrac ln, int s) {
    long long t = th_c(c, 17);
    t = th_c(c, 16) + fx_mul(t, u);
    t = th_c(c, 15) + fx_mul(t, u);
    t = th_c(c, 14) + fx_mul(t, u);
    t = th_c(c, 12) + fx_mul(th_c(c, 13), ln) + fx_mul(t, u);
    return fx_round_d(th_c(c, 11) + fx_mul(t, u), s);
}

}  // namespace nk
