// Base-2 logarithms in 64-bit fixed point ("fx"), the exponent arithmetic of the FP64 reaction
// kernels.
//
// A rate term is one exponential of a sum of logarithms (ln k_f, chemical potentials, ln C).  The
// sums used to run in double-float pairs: ~11 FP32 operations per addition, 14 per multiply-add,
// and each exponential ended in one FP64 addition, on a pipe that takes 64 issue slots per warp
// instruction on GB300 (1.67 FP64 operations per clock and SM against 128 for integer additions
// and FFMA, measured).  As 64-bit integers in units of 2^-48 of log2 the additions take two
// instructions, are exact and associative, and the result's double is put together from the
// integer exponent and two floats without the FP64 pipe.  Range +-32768 (the kernels' bounds are
// checked at mechanism load and per block of points), rounding 2^-49 absolute per product: a rate
// term carries about 5e-15 relative, against 1e-13 of the pairs.
//
// Products of a coefficient and a per-point temperature variable (log2 T, 128/T, T/4096, all in
// [0, 1) as 63-bit fractions) take three 32-bit multiplications (fx_mul); the variables are split
// so that all partial products are single IMAD.WIDE/IMAD.HI instructions.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "nk_df.cuh"

namespace nk {

constexpr int kFxS = 48;                       // fraction bits
constexpr int kFxExpTab = 128, kFxLogTab = 128;
constexpr double kFxTmin = 128.0, kFxTmax = 4096.0;  // open interval of temperatures the fractions cover
constexpr long long kFxZero = -(5000LL << kFxS);     // log2 of a zero concentration: any rate term
                                                     // holding it (up to four per side) underflows
// Tables in device memory and, staged, in shared memory: exp entries {T_j (float), d_j}, then log
// entries {L_j (64 bits)}, then the 16-bit reciprocals.
struct FxTab {
    const uint2* e;      // [128] T_j = 2^(j/128) cut to a float (bits) and (j/128 - log2 T_j) 2^48
    const long long* l;  // [128] -log2(c_j / 1024) 2^48
    const uint32_t* c;   // [128] c_j, about 1024/(1 + (j + 1/2)/128)
};
constexpr int kFxTabBytes = kFxExpTab * 8 + kFxLogTab * 8 + kFxLogTab * 4;

__device__ __forceinline__ FxTab stage_fx_tables(uint32_t* s, const uint32_t* g) {
    for (int j = threadIdx.x; j < kFxTabBytes / 4; j += blockDim.x) s[j] = __ldg(g + j);
    return FxTab{reinterpret_cast<const uint2*>(s), reinterpret_cast<const long long*>(s + 2 * kFxExpTab),
                 s + 2 * kFxExpTab + 2 * kFxLogTab};
}

// A fraction in [0, 1): h 2^-31 + l 2^-63 with 0 <= h < 2^31 and l signed.
struct FxFrac {
    int32_t h, l;
};
__device__ __forceinline__ FxFrac fx_frac63(unsigned long long w) {   // w 2^-63, w < 2^63 - 2^31
    return {(int32_t)((w + 0x80000000ull) >> 32), (int32_t)(uint32_t)w};
}

// c w / 2 for a 64-bit c and a fraction w, cut by 1.25 units on average (the tables add it back)
__device__ __forceinline__ long long fx_mul(long long c, FxFrac w) {
    const int32_t ch = (int32_t)(c >> 32);
    const uint32_t cl = (uint32_t)c;
    long long r = (long long)ch * w.h;
    r += (unsigned long long)__umulhi(cl, (uint32_t)w.h);
    return r + (long long)__mulhi(ch, w.l);
}

// log2 of m 2^(e - 52) for a 53-bit m with the leading bit set, as fx.  Table of 128 ten-bit
// reciprocals c_j: r = m c_j 2^-62 - 1 is exact in 64 bits (|r| < 0.0045), log(1 + r) by its
// series with r and r^2/2 carried in two floats, degree 6 (error below 2^-49).
__device__ __forceinline__ long long fx_log2_core(unsigned long long m, int e, const FxTab& t) {
    const int j = (int)(m >> 45) & 127;
    const uint32_t c = t.c[j];
    const unsigned long long P = (unsigned long long)(uint32_t)m * c + ((unsigned long long)((uint32_t)(m >> 32) * c) << 32);
    const long long R = (long long)(P - (1ull << 62));                                // r 2^62
    const float p = __fmul_rn(__fsub_rn(__int_as_float(0x4B400000 + (int)(R >> 33)), 12582912.0f), 0x1p-29f);
    const float l = __fmul_rn(__fsub_rn(__int_as_float(0x4B000000 | ((int)(R >> 10) & 0x7fffff)), 8388608.0f), 0x1p-52f);
    const float q = __fmul_rn(p, p);
    const float qe = __fmaf_rn(p, p, -q);
    const float s = __fmaf_rn(-0.5f, q, p);
    float lo = __fmaf_rn(-0.5f, q, __fsub_rn(p, s));
    lo = __fmaf_rn(-0.5f, qe, lo);
    lo = __fadd_rn(lo, l);
    lo = __fmaf_rn(l, __fsub_rn(q, p), lo);
    const float tl = __fmaf_rn(p, __fmaf_rn(p, __fmaf_rn(p, -1.0f / 6.0f, 0.2f), -0.25f), 1.0f / 3.0f);
    lo = __fmaf_rn(__fmul_rn(q, p), tl, lo);
    constexpr float L2EH = 1.4426950216293335f, L2EL = 1.9259629911266175e-08f;
    const float y = __fmul_rn(s, L2EH);
    float ye = __fmaf_rn(s, L2EH, -y);
    ye = __fmaf_rn(s, L2EL, ye);
    ye = __fmaf_rn(lo, L2EH, ye);
    constexpr float M1 = 1.5f * 0x1p-6f, M2 = 1.5f * 0x1p-25f;                        // ulps 2^-29, 2^-48
    const float k1 = __fadd_rn(__fadd_rn(y, ye), M1);
    const float k2 = __fadd_rn(__fadd_rn(__fsub_rn(y, __fsub_rn(k1, M1)), ye), M2);
    constexpr int B1 = 0x3CC00000, B2 = 0x33400000;                                   // bits of M1, M2
    return ((long long)e << kFxS) + t.l[j] + ((long long)(__float_as_int(k1) - B1) << 19) +
           (long long)(__float_as_int(k2) - B2);
}
// of a positive normal double (bits)
__device__ __forceinline__ long long fx_log2_bits(unsigned long long b, const FxTab& t) {
    return fx_log2_core((b & 0x000fffffffffffffull) | 0x0010000000000000ull, (int)(b >> 52) - 1023, t);
}
// of v 2^-s for a positive 64-bit integer v (its top 53 bits)
__device__ __forceinline__ long long fx_log2_int(unsigned long long v, int s, const FxTab& t) {
    const int z = __clzll((long long)v);
    return fx_log2_core((v << z) >> 11, 63 - z - s, t);
}

// 2^x: v = T_j (1 + (2^r' - 1)) with x = m + j/128 + r, r' = r + d_j in [0, 2^-7 + 2^-22) exact in
// 42 bits as two floats; 2^r' - 1 by the exponential series to degree 5, r' ln2 and its square in
// two floats; the double's bits are T_j's plus the two floats rounded to integers, plus m in the
// exponent.  Relative error about 1e-15.  x >= 1024 gives inf, x < -1022 gives 0.  SIGNED: bit 0 of
// x is the sign of the result.
template <bool SIGNED = false>
__device__ __forceinline__ double fx_exp2(long long x, const FxTab& t) {
    const int xh = (int)(x >> 32);
    const uint2 en = t.e[(xh >> 9) & 127];
    const unsigned long long R = (((unsigned long long)((uint32_t)xh & 0x1ffu) << 32) | (uint32_t)x) + en.y;
    const float fh = __fsub_rn(__int_as_float(0x4B000000 | (int)(R >> 19)), 8388608.0f);          // unit 2^-29
    const float fl = __fsub_rn(__int_as_float(0x4B000000 | (int)((uint32_t)R & 0x7ffffu)), 8388608.0f);   // unit 2^-48
    constexpr float c1 = 0.693147182464599609375f * 0x1p-29f, c2 = -1.9046542121259336e-09f * 0x1p-29f;
    constexpr float c3 = 0.693147182464599609375f * 0x1p-48f;
    const float p = __fmul_rn(fh, c1);
    float e = __fmaf_rn(fh, c1, -p);
    e = __fmaf_rn(fh, c2, e);
    e = __fmaf_rn(fl, c3, e);
    const float q = __fmul_rn(p, p);
    const float qe = __fmaf_rn(p, p, -q);
    const float s = __fmaf_rn(0.5f, q, p);
    float lo = __fmaf_rn(0.5f, q, -__fsub_rn(s, p));
    const float tl = __fmaf_rn(p, __fmaf_rn(p, 1.0f / 120.0f, 1.0f / 24.0f), 1.0f / 6.0f);
    float w = __fmaf_rn(__fmul_rn(q, p), tl, e);
    w = __fmaf_rn(0.5f, qe, w);
    w = __fmaf_rn(s, e, w);                                                           // e (p + p^2/2)
    lo = __fadd_rn(lo, w);
    const float T = __uint_as_float(en.x);
    const float v = __fmul_rn(T, s);
    float ve = __fmaf_rn(T, s, -v);
    ve = __fmaf_rn(T, lo, ve);
    constexpr float M1 = 0x1p-6f, M2 = 1.5f * 0x1p-28f;                               // ulps 2^-29, 2^-51
    const float k1 = __fadd_rn(__fadd_rn(v, ve), M1);
    const float k2 = __fadd_rn(__fadd_rn(__fsub_rn(v, __fsub_rn(k1, M1)), ve), M2);
    // bits in units of 2^-52: T 2^29, k1 2^23, k2 2; the constants are the bits of 1.0f, M1, M2
    constexpr unsigned long long K0 = 0x3ff0000000000000ull - ((unsigned long long)0x3f800000u << 29) -
                                      ((unsigned long long)0x3C800000u << 23) - ((unsigned long long)0x31C00000u << 1);
    unsigned long long b = (unsigned long long)en.x * (1u << 29) + K0;
    b = (unsigned long long)__float_as_uint(k1) * (1u << 23) + b;
    b = (unsigned long long)__float_as_uint(k2) * 2u + b;
    const int m = xh >> 16;
    uint32_t hi = (uint32_t)(b >> 32) + ((uint32_t)m << 20), lo32 = (uint32_t)b;
    if ((unsigned)(m + 1022) > 2045u) {
        hi = m < 0 ? 0u : 0x7ff00000u;
        lo32 = 0u;
    }
    if (SIGNED) hi |= (uint32_t)x << 31;
    return __hiloint2double((int)hi, (int)lo32);
}

// x 2^-48 as a double, by integer operations
__device__ __forceinline__ double fx_to_d(long long x) {
    const unsigned long long a = (unsigned long long)(x < 0 ? -x : x);
    const int z = __clzll((long long)a);
    if (a == 0) return 0.0;
    const unsigned long long m = (a << z) >> 11;                                      // 53 bits, cut
    const unsigned long long b = m + ((unsigned long long)(1023 + 63 - kFxS - z - 1) << 52);
    return __longlong_as_double((long long)(b | ((unsigned long long)x & 0x8000000000000000ull)));
}
// x 2^-s as a double (to nearest, ties up in magnitude), by integer operations
__device__ __forceinline__ double fx_round_d(long long x, int s) {
    const unsigned long long a = (unsigned long long)(x < 0 ? -x : x);
    if (a == 0) return 0.0;
    const int z = __clzll((long long)a);
    const unsigned long long n = a << z;
    const unsigned long long m = (n >> 11) + ((n >> 10) & 1ull);                      // 53 bits (a carry raises the exponent)
    const unsigned long long b = m + ((unsigned long long)(1023 + 63 - s - z - 1) << 52);
    return __longlong_as_double((long long)(b | ((unsigned long long)x & 0x8000000000000000ull)));
}
// x 2^-48 as a float pair (pieces of 22 bits, exact but for the last rounding)
__device__ __forceinline__ dfl fx_to_pair(long long x) {
    const float a = __fmul_rn(__fsub_rn(__int_as_float(0x4B400000 + (int)(x >> 44)), 12582912.0f), 0x1p-4f);
    const float b = __fmul_rn(__fsub_rn(__int_as_float(0x4B000000 | ((int)(x >> 22) & 0x3fffff)), 8388608.0f), 0x1p-26f);
    const float c = __fmul_rn(__fsub_rn(__int_as_float(0x4B000000 | ((int)x & 0x3fffff)), 8388608.0f), 0x1p-48f);
    dfl s = two_sum(a, b);
    s.l = __fadd_rn(s.l, c);
    return fast_two_sum(s.h, s.l);
}
// a pair (|x| < 8192) as fx
__device__ __forceinline__ long long fx_of_pair(dfl x) {
    constexpr float M1 = 1.5f * 0x1p14f, M2 = 1.5f * 0x1p-8f, M3 = 1.5f * 0x1p-25f;   // ulps 2^-9, 2^-31, 2^-48
    const float k1 = __fadd_rn(x.h, M1);
    const dfl r = two_sum(__fsub_rn(x.h, __fsub_rn(k1, M1)), x.l);
    const float k2 = __fadd_rn(r.h, M2);
    const float k3 = __fadd_rn(__fadd_rn(__fsub_rn(r.h, __fsub_rn(k2, M2)), r.l), M3);
    return ((long long)(__float_as_int(k1) - 0x46C00000) << 39) + ((long long)(__float_as_int(k2) - 0x3BC00000) << 17) +
           (long long)(__float_as_int(k3) - 0x33400000);
}
// a double of magnitude below 2048 (a shift of ln A) times log2(e), as fx
__device__ __forceinline__ long long fx_log2e_times(double d) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(d);
    const int e = (int)(b >> 52 & 0x7ff) - 1023;
    const unsigned long long m = (b & 0x000fffffffffffffull) | 0x0010000000000000ull;
    const int sh = e - 4;                                                             // m 2^(e - 52 + 48)
    long long v = (long long)(sh >= 0 ? m << sh : (sh > -54 ? m >> -sh : 0ull));
    if ((long long)b < 0) v = -v;
    // log2 e = 1 + 0.4426950408889634...: fx_mul halves, so the fraction is twice 0.4427
    constexpr unsigned long long F = 0x71547652B82FE177ull;                           // 0.88539008177792681... 2^63
    return v + fx_mul(v, FxFrac{(int32_t)((F + 0x80000000ull) >> 32), (int32_t)(uint32_t)F});
}

// a float of magnitude below 4096 times log2(e), as fx
__device__ __forceinline__ long long fx_log2e_times(float f) {
    const uint32_t b = __float_as_uint(f);
    const int sh = (int)(b >> 23 & 0xffu) - 127 + kFxS - 23;                          // m 2^sh units
    const long long m = (long long)((b & 0x7fffffu) | 0x800000u);
    long long v = sh >= 0 ? m << (sh & 63) : (sh > -24 ? m >> -sh : 0);
    if ((int)b < 0) v = -v;
    constexpr unsigned long long F = 0x71547652B82FE177ull;                           // 0.88539008177792681... 2^63
    return v + fx_mul(v, FxFrac{(int32_t)((F + 0x80000000ull) >> 32), (int32_t)(uint32_t)F});
}

}  // namespace nk
