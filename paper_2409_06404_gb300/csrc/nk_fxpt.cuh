// Per-point set-up and reaction terms of the fixed-point reaction kernels (nk_fx.cuh), shared by
// the rates and their derivatives.
//
// A block takes 32 points, one lane each, and NP warps ("parts") share a point.  Species k belongs
// to part k % NP (at most kFxOwn species per part); the parts take the reactions of a chunk in
// turn and leave their rates of progress in shared memory, and each part then sums its own
// species over the chunk's list (FxTables): two barriers per chunk of up to 48 reactions, where adding
// into the species' rows directly took one per round of reactions without a common species (84
// rounds at 325 reactions), and no reaction waits for another.  The order of every sum is fixed by
// the mechanism.
//
// A negative concentration (a negative mass fraction) enters by its magnitude with its sign in bit 0
// of a_k and mu_k: the low bit of a sum is then the parity of its negative factors, so the sign of
// each side's product comes out of the same additions.
//
// Reverse rates come from chemical potentials: with a_k = log2 C_k and
// mu_k = a_k + log2(e) g_k/RT + log2(R T/p0), log2 q_f = log2 k_f + sum_reactants a and
// log2 q_r = log2 q_f + sum_products mu - sum_reactants mu.  So the NASA-7 polynomials are evaluated
// once per species instead of once per reaction, and a reaction's sums are integer additions.
#pragma once

#include "nk_fx.cuh"
#include "nk_rxn.cuh"

namespace nk {

// Marks a point whose state is outside the fixed-point form in an output the fallback pass reads
// (a quiet NaN no arithmetic returns).
constexpr unsigned long long kFxSkip = 0x7ff80f15ca1cedull << 8 | 0x5aull;

// fraction y/2 of a double in [0, 2) (bits; below 2^-60 cut off)
__device__ __forceinline__ unsigned long long fx_half63(unsigned long long b) {
    const int e = (int)(b >> 52) - 1023;
    const unsigned long long m = (b & 0x000fffffffffffffull) | 0x0010000000000000ull;
    const int sh = e + 10;
    return sh >= 0 ? m << sh : (sh > -54 ? m >> -sh : 0ull);
}

// temperature fractions: T/4096 from T's bits (128 < T < 4096)
__device__ __forceinline__ FxFrac fx_frac_T(unsigned long long b) {
    const int e = (int)(b >> 52) - 1023;
    return fx_frac63(((b & 0x000fffffffffffffull) | 0x0010000000000000ull) << ((e - 1) & 63));
}

struct FxT {
    FxFrac lt, v;          // log2(T)/16 and 128/T
};

// log2(e) g/RT + log2(R T/p0) of a species (c: its range's coefficients)
__device__ __forceinline__ long long fx_mu0(const int64_t* c, const FxT& P, FxFrac u) {
    long long t = __ldg((const long long*)c + 5);
    t = __ldg((const long long*)c + 4) + fx_mul(t, u);
    t = __ldg((const long long*)c + 3) + fx_mul(t, u);
    t = __ldg((const long long*)c + 2) + fx_mul(t, u);
    t = __ldg((const long long*)c + 0) + fx_mul(t, u);
    t += fx_mul(__ldg((const long long*)c + 1), P.lt);
    return t + fx_mul(__ldg((const long long*)c + 6), P.v);
}
// h/RT and c_p/R (over kFxCpScale) of a species
__device__ __forceinline__ long long fx_hRT(const int64_t* c, const FxT& P, FxFrac u) {
    long long t = __ldg((const long long*)c + 12);
    t = __ldg((const long long*)c + 11) + fx_mul(t, u);
    t = __ldg((const long long*)c + 10) + fx_mul(t, u);
    t = __ldg((const long long*)c + 9) + fx_mul(t, u);
    t = __ldg((const long long*)c + 8) + fx_mul(t, u);
    return t + fx_mul(__ldg((const long long*)c + 13), P.v);
}
__device__ __forceinline__ long long fx_cpR(const int64_t* c, FxFrac u) {
    long long t = __ldg((const long long*)c + 17);
    t = __ldg((const long long*)c + 16) + fx_mul(t, u);
    t = __ldg((const long long*)c + 15) + fx_mul(t, u);
    t = __ldg((const long long*)c + 14) + fx_mul(t, u);
    return __ldg((const long long*)c + 7) + fx_mul(t, u);
}
__device__ __forceinline__ const int64_t* fx_range(const FxSpecies* s, double T) {
    // T <= T_mid on the bit patterns (both positive)
    const bool lo = __double_as_longlong(T) <= __ldg(reinterpret_cast<const long long*>(&s->Tmid));
    return lo ? s->c[0] : s->c[1];
}

// Shared memory of a block (after the fixed-point and the pair tables): the scalars of its points, log2 C_k, mu_k and the
// rates of progress of one chunk, each as rows of 32 lanes.
constexpr int kFxScalars = 6;      // log2 T, 128/T (63 bits), log2(p/(R T)), log2 rho', sum Y/W, floats of ln T and 1/T
enum { kFxLT = 0, kFxV = 1, kFxLpRT = 2, kFxLrho = 3, kFxSum = 4, kFxTf = 5 };
constexpr size_t kFxBase = kFxTabBytes + kDfTabBytes;
// The row after the last species is zero; two chunk images are double buffered; row_bytes per
// reaction of a chunk.
inline size_t fx_smem(const FxSet& f, int K, int row_bytes) {
    const size_t q = (size_t)f.rows * row_bytes, part = (size_t)f.np * 3 * 256;   // the parts' sums come first
    return kFxBase + kFxScalars * 256 + 2 * (size_t)f.image + (size_t)f.row * (K + 1) + (q > part ? q : part);
}
// Starts the copy of chunk c's image into shared memory (cp.async; waited for by fx_image_wait and
// a barrier).
__device__ __forceinline__ void fx_image_load(const FxSet& f, int c, unsigned char* dst) {
    if (c < f.nchunk) {
        const unsigned char* src = f.chunks + (size_t)c * f.image;
        const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
        for (int o = threadIdx.x * 16; o < f.image; o += blockDim.x * 16)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d + o), "l"(src + o) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}
__device__ __forceinline__ void fx_image_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// ---- the state a point needs for the fixed-point form, and its scalars
constexpr unsigned long long kFxPoison = 1ull << 55;      // (added by up to 32 parts without wrapping)
__device__ __forceinline__ bool fx_T_ok(double T) {      // 128 (1 + 2^-31) < T < 4096 (1 - 2^-30)
    const long long b = __double_as_longlong(T);
    return b > 0x4060000000200000ll && b < 0x40afffffffc00000ll;
}
__device__ __forceinline__ bool fx_p_ok(double p) {      // [2^-100, 2^101)
    return (unsigned)((unsigned long long)__double_as_longlong(p) >> 52) - 923u <= 200u;
}
// adds |y|'s part of sum |Y| (units 2^-40) and y/W's of sum Y/W (units 2^-60, relative to the
// largest 1/W); bad: y is subnormal, 2 or more in magnitude, or not finite
__device__ __forceinline__ void fx_add_fraction(unsigned long long yb, long long w, unsigned long long& z,
                                                unsigned long long& zc, bool& bad) {
    if ((yb << 1) == 0) return;
    const unsigned long long a = yb & 0x7fffffffffffffffull;
    bad |= (unsigned)(a >> 52) - 1u >= 1023u;
    const unsigned long long f = fx_half63(a);
    const unsigned long long t = (unsigned long long)fx_mul(w, fx_frac63(f));
    z += (long long)yb < 0 ? 0ull - t : t;
    zc += f >> 22;
}
// sum |Y| above 1.5 (or poisoned), or sum Y/W not positive or not resolved
__device__ __forceinline__ bool fx_sums_bad(unsigned long long z, unsigned long long zc) {
    return zc > (3ull << 39) || z < (1ull << 50) || z > (1ull << 62);
}
// log2 T, 128/T and log2(p/(R T)) of a point into its scalars
__device__ __forceinline__ void fx_point_scalars(const DevMech& m, unsigned long long Tb, double p, long long* sS,
                                                 const FxTab& t) {
    const unsigned long long pb = (unsigned long long)__double_as_longlong(p);
    const unsigned long long vb = (unsigned long long)__double_as_longlong(128.0 / __longlong_as_double((long long)Tb));
    const long long lT = fx_log2_bits(Tb, t);
    sS[kFxLT * 32] = lT;
    sS[kFxV * 32] = (long long)(((vb & 0x000fffffffffffffull) | 0x0010000000000000ull) << (((int)(vb >> 52) - 1012) & 63));
    sS[kFxLpRT * 32] = fx_log2_bits(pb, t) - m.fx_lR - lT;
}
// log2 |C_k| with the sign in bit 0, from the mass fraction's bits and log2(rho/W_k)
__device__ __forceinline__ long long fx_log2_conc(unsigned long long yb, long long lr, const FxTab& t) {
    if ((yb << 1) == 0) return kFxZero;
    return ((fx_log2_bits(yb & 0x7fffffffffffffffull, t) + lr) & ~1ll) | (long long)(yb >> 63);
}
// z = [M]/rho' and log2 |z| from the third-body efficiencies, [M] = rho' (sum Y/W + sum (eps - 1)
// Y/W).  Y is read again (it is in L1 or L2).
__device__ __forceinline__ long long fx_third_body(const DevMech& m, int eff0, int eff1, const double* Y, int64_t ld,
                                                   int64_t i, long long sum, const FxTab& t, long long& lM) {
    long long z = sum >> m.fx_eff_shift;
    for (int j = eff0; j < eff1; ++j) {
        const longlong2 e = __ldg(reinterpret_cast<const longlong2*>(m.fx_eff + j));
        const unsigned long long yb = (unsigned long long)__double_as_longlong(__ldg(Y + (int64_t)(int)e.y * ld + i));
        if ((yb << 1) != 0) {
            const long long d = fx_mul(e.x, fx_frac63(fx_half63(yb & 0x7fffffffffffffffull)));
            z += (long long)yb < 0 ? -d : d;
        }
    }
    lM = fx_log2_int((unsigned long long)(z > 0 ? z : z < 0 ? -z : 1ll), 60 - m.fx_eff_shift, t) + m.fx_lmaxw;
    return z;
}

// 1/T as a pair from its fraction 128/T, T as a pair from its bits
__device__ __forceinline__ dfl fx_invT_pair(FxFrac v) {
    const float a = __fmul_rn((float)(v.h >> 9), 0x1p-29f);                    // 2^-22/128
    const float b = __fmul_rn((float)(v.h & 511), 0x1p-38f), c = __fmul_rn((float)v.l, 0x1p-70f);
    const dfl s = two_sum(a, b);
    return fast_two_sum(s.h, __fadd_rn(s.l, c));
}
__device__ __forceinline__ dfl fx_T_pair(double T) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(T);
    const unsigned long long w = ((b & 0x000fffffffffffffull) | 0x0010000000000000ull) << (((int)(b >> 52) - 1024) & 63);
    const float h = __fmul_rn((float)(int)(w >> 41), 0x1p-10f), c = __fmul_rn((float)((int)(w >> 19) & 0x3fffff), 0x1p-32f);
    const dfl s = two_sum(h, c);
    return fast_two_sum(s.h, __fadd_rn(s.l, __fmul_rn((float)((int)w & 0x7ffff), 0x1p-51f)));
}

// 2^x as an integer in units of 2^-60, for x <= 1 (cut below 2^-60)
__device__ __forceinline__ unsigned long long fx_exp2_int(long long x, const FxTab& t) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(fx_exp2(x, t));
    const int e = (int)(b >> 52) - 1023;
    const unsigned long long m = (b & 0x000fffffffffffffull) | 0x0010000000000000ull;
    const int sh = e + 8;                                // m 2^(e - 52 + 60)
    return sh >= 0 ? m << sh : (sh > -54 ? m >> -sh : 0ull);
}
// c w for a constant fraction F 2^-63 of magnitude below 1 (fx_mul halves: c doubled)
__device__ __forceinline__ long long fx_scale(long long c, unsigned long long F) {
    return fx_mul(2 * c, FxFrac{(int32_t)((F + 0x80000000ull) >> 32), (int32_t)(uint32_t)F});
}

// log2 of the Troe factor F P_r/(1 + P_r) from X = log2 P_r.  With Lc = log2 F_cent,
// u = X log10(2) - 0.4 - 0.67 log10(2) Lc and v = 0.75 - 1.27 log10(2) Lc - 0.14 u it is
// Lc v^2/(u^2 + v^2) + log2(P_r/(1 + P_r)): exponentials and logarithms in fixed point, the one
// quotient in pairs.  F_cent from its three terms as integers; where they do not fit (a outside
// (0, 1), F_cent below 2^-12) it comes from troe_cent.  Out of line: its hundreds of instructions
// would push the reaction loop out of the instruction cache.
static __device__ __noinline__ long long fx_troe_cent_edge(const float4* df, const TroeRec* d, int aux, double T, FxFrac v,
                                                           DfTab dt) {
    TPairs tp;
    tp.T = T;
    tp.Td = fx_T_pair(T);
    tp.invTd = fx_invT_pair(v);
    constexpr dfl LOG2_10{3.321928024291992f, 7.0595369580300144e-08f};
    return fx_of_pair(df_mul(troe_cent(df, d, aux, tp, dt).L, LOG2_10));
}
static __device__ __noinline__ long long fx_troe(const FxTroe* fx, const float4* df, const TroeRec* d, int aux, double T,
                                                 FxFrac v, long long X, FxTab t, DfTab dt) {
    const long long* r = reinterpret_cast<const long long*>(fx + aux);
    const FxFrac u = fx_frac_T((unsigned long long)__double_as_longlong(T));
    long long Lc = 0;
    const int flags = (int)__ldg(r + 8);
    bool edge = !(flags & 1);
    if (!edge) {
        unsigned long long Fc = fx_exp2_int(__ldg(r + 3) + fx_mul(__ldg(r + 4), u), t) +
                                fx_exp2_int(__ldg(r + 5) + fx_mul(__ldg(r + 6), u), t);
        if (flags & 2) Fc += fx_exp2_int(fx_mul(__ldg(r + 7), v), t);
        edge = Fc < 1ull << 48;
        Lc = fx_log2_int(edge ? 1ull << 60 : Fc, 60, t);
    }
    if (edge) Lc = fx_troe_cent_edge(df, d, aux, T, v, dt);
    constexpr unsigned long long kLog10_2 = 0x268826A13EF3FDE6ull;                  // log10(2) 2^63
    constexpr unsigned long long k067 = 0x55C28F5C28F5C28Full, k027 = 0x228F5C28F5C28F5Cull, k014 = 0x11EB851EB851EB85ull;
    const long long L10 = fx_scale(Lc, kLog10_2);
    const long long uu = fx_scale(X, kLog10_2) - (long long)(0.4 * 281474976710656.0) - fx_scale(L10, k067);
    const long long vv = (long long)(0.75 * 281474976710656.0) - L10 - fx_scale(L10, k027) - fx_scale(uu, k014);
    const dfl pu = fx_to_pair(uu), pv = fx_to_pair(vv);
    const dfl v2 = df_mul(pv, pv);
    const dfl ratio = df_div(v2, df_fma(pu, pu, v2));
    // log2(P_r/(1 + P_r)) = min(X, 0) - log2(1 + 2^-|X|)
    const unsigned long long z = fx_exp2_int(X < 0 ? X : -X, t);
    const long long s = fx_log2_int((1ull << 60) + z, 60, t);
    return fx_of_pair(df_mul(fx_to_pair(Lc), ratio)) + (X < 0 ? X : 0ll) - s;
}

// log2 q_f less log2 k_f and log2 q_r less log2 q_f of a reaction record: sums over its molecules
// (sp: the species rows, mu_k 256 bytes after log2 C_k).
struct FxRate {
    long long f, r;
};
__device__ __forceinline__ void fx_reac(const unsigned char* a, FxRate& x) {
    x.f += *reinterpret_cast<const long long*>(a);
    x.r -= *reinterpret_cast<const long long*>(a + 256);
}
__device__ __forceinline__ void fx_prod(const unsigned char* a, FxRate& x) {
    x.r += *reinterpret_cast<const long long*>(a + 256);
}
__device__ __forceinline__ FxRate fx_sides(const unsigned char* sp, int info, uint4 re, uint4 pr) {
    FxRate x{0, 0};
    fx_reac(sp + re.x, x);
    fx_reac(sp + re.y, x);
    fx_prod(sp + pr.x, x);
    fx_prod(sp + pr.y, x);
    if ((info & 15) > 2) {
        fx_reac(sp + re.z, x);
        if ((info & 15) > 3) fx_reac(sp + re.w, x);
    }
    if ((info >> 4 & 15) > 2) {
        fx_prod(sp + pr.z, x);
        if ((info >> 4 & 15) > 3) fx_prod(sp + pr.w, x);
    }
    return x;
}

// a rate of progress times e^d for a shift of ln A outside the fixed-point form
static __device__ __noinline__ double fx_shift_edge(double q, double d) { return q * exp(d); }

// Sum over one species' rows of a chunk, the rows MUL 256 bytes apart (w: its word in the image,
// list: the image's row list, q: the rows, this lane's column), added to s in list order.  (Two rows
// per step left predicated FP64 additions behind, which cost as much as executed ones.)
template <int MUL = 1>
__device__ __forceinline__ double fx_gather(uint32_t w, const unsigned char* list, const unsigned char* q, double s) {
    const unsigned char* l = list + (w >> 15 & ~1u);
    const unsigned char* e = l + (w >> 7 & 510u);
#pragma unroll 1
    for (; l != e; l += 2) s += *reinterpret_cast<const double*>(q + MUL * *reinterpret_cast<const uint16_t*>(l));
    e += (w & 255u) * 2;
#pragma unroll 1
    for (; l != e; l += 2) s -= *reinterpret_cast<const double*>(q + MUL * *reinterpret_cast<const uint16_t*>(l));
    return s;
}

// q times a stoichiometric coefficient other than 1.  Out of line: inline it becomes a predicated
// conversion and product on the FP64 pipe for every reaction.
static __device__ __noinline__ double times_nu(double q, int nu) { return q * (double)nu; }

}  // namespace nk
