// Product pass in single precision with the rates kernel's chunks (included by k_lin.cu, whose
// arithmetic it keeps operation by operation): a part takes reactions of a chunk without waiting for
// the others, so all its warps' loads are in flight at once, where the rounds of jvp_lin32_kernel
// let one reaction per warp load between barriers (1.7 TB/s of the stored words at 2,097,152
// points).  A species' terms are summed in the order of those rounds (FxTerm32) and the point sums
// by the same parts, so the results are the same bits.  Load latency bounds it (waits on stored words
// 4.2 cycles per issue, issue slots 51% busy), so a reaction's words are loaded while the one before
// is summed, and all parts load the state.  53 species, 2,097,152 points: 12.6 -> 9.0 ms per product
// (2.3 TB/s of the stored words); the single-precision stage of 175,616 points with its ten
// products: 21.7 -> 15.7 ms.
#pragma once

#include "nk_fxpt.cuh"

namespace nk {
namespace {

inline size_t lin32_fx_smem(const FxSet& f, int K, int old_np) {
    return (size_t)3 * old_np * 256 + 5 * 128 + 128 + 2 * (size_t)f.image + (size_t)K * 384 + (size_t)f.rows * 256;
}
inline const FxSet& lin32_set(const DevMech& m, int old_np) { return m.fx32[old_np == 1 ? 0 : old_np == 2 ? 1 : 2]; }
inline bool lin32_fx_fits(const DevMech& m, int old_np) {
    return m.fx_ok && lin32_fx_smem(lin32_set(m, old_np), m.K, old_np) <= smem_limit();
}

// the stored words of one reaction
struct Words32 {
    float A, br[kMaxSide], bp[kMaxSide], L;
    int er;
};
__device__ __forceinline__ void load_words32(const DevMech& m, const unsigned char* im, int q, const float* a, int64_t ldl,
                                             Words32& w) {
    const int4 h = reinterpret_cast<const int4*>(im + q * (int)sizeof(FxRxn32))[1];      // info, r, boff, eff0
    const int nr = h.x & 15, np = h.x >> 4 & 15;
    w.A = __ldcs(a + (int64_t)h.y * ldl);
    const float* B = a + ((int64_t)m.R + h.z) * ldl;
#pragma unroll
    for (int e = 0; e < kMaxSide; ++e) {
        w.br[e] = e < nr ? __ldcs(B + (int64_t)e * ldl) : 0.0f;
        w.bp[e] = e < np ? __ldcs(B + (int64_t)(nr + e) * ldl) : 0.0f;
    }
    w.er = __ldcs(reinterpret_cast<const int32_t*>(a) + (slot_E32(m) + h.y) * ldl);
    w.L = h.x >> 8 != 0 ? __ldcs(a + (slot_M(m) + (h.y - m.R_el)) * ldl) : 0.0f;
}

// OLD: the parts of jvp_lin32_kernel's shape for this mechanism.
template <int NP, int OLD, bool RHS>
__global__ void __launch_bounds__(32 * NP, NP == 4 ? 8 : NP == 8 ? 4 : NP == 16 ? 2 : 1)
    jvp_lin32_fx_kernel(const DevMech m, const int64_t n, const int64_t ld, const double* __restrict__ T,
                        const double* __restrict__ p, const double* __restrict__ Y, const float* __restrict__ lin,
                        const int64_t ldl, const double* __restrict__ vT, const double* __restrict__ vY,
                        double* __restrict__ d_omega, double* __restrict__ d_hrr, const double* __restrict__ fT,
                        const double* __restrict__ fY, const int64_t ldf) {
    extern __shared__ __align__(16) unsigned char smem_fx[];
    const FxSet& f = m.fx32[OLD == 1 ? 0 : OLD == 2 ? 1 : 2];
    const int K = m.K;
    const int lane = threadIdx.x & 31, part = threadIdx.x >> 5;
    const int64_t i0 = (int64_t)blockIdx.x * 32 + lane;
    const bool live = i0 < n;
    const int64_t i = live ? i0 : n - 1;
    unsigned char* im0 = smem_fx;
    fx_image_load(f, 0, im0);
    double* sR = reinterpret_cast<double*>(smem_fx + 2 * f.image) + lane;        // part sums
    float* sV = reinterpret_cast<float*>(smem_fx + 2 * f.image + 3 * OLD * 256) + lane;   // tT, rho, arho, d(p/RT)
    unsigned char* sdC = smem_fx + 2 * f.image + 3 * OLD * 256 + 6 * 128 + lane * 4;      // dC_k, slot order
    float* sW = reinterpret_cast<float*>(sdC + (size_t)K * 128);                 // d omega_k sums, species order
    int* sE = reinterpret_cast<int*>(sW + (size_t)K * 32);                       // E_k, species order
    unsigned char* sQ = reinterpret_cast<unsigned char*>(sE + (size_t)K * 32) + lane * 4;   // dq and exponent, 8 bytes a lane
    const int32_t* linE = reinterpret_cast<const int32_t*>(lin) + slot_EK32(m) * ldl + i;
    // (Y and vY go through the rows of the sums and of E_k, so that all parts load; summed in species order)
#pragma unroll 4
    for (int k = part; k < K; k += NP) {
        sW[k * 32] = narrow(Y[(int64_t)k * ld + i]);
        sE[k * 32] = __float_as_int(narrow(vY[(int64_t)k * ld + i]));
    }
    __syncthreads();
    if (part == 0) {
        const float Ti = narrow(T[i]), dT = narrow(vT[i]);
        const float invT = 1.0f / Ti, tT = dT * invT;
        const float pRT = narrow(p[i]) * invT * kInvRf;
        float s = 0.0f, ds = 0.0f;
#pragma unroll 4
        for (int k = 0; k < K; ++k) {
            const float iw = __ldg(m.f_invW + k);
            s = fmaf(sW[k * 32], iw, s);
            ds = fmaf(__int_as_float(sE[k * 32]), iw, ds);
        }
        const float rho = pRT / s;
        sV[0] = tT;
        sV[32] = rho;
        sV[64] = -tT - ds / s;                                   // d rho / rho
        sV[96] = -pRT * tT;
    }
    __syncthreads();
    {
        const float rho = sV[32], arho = sV[64];
#pragma unroll 4
        for (int k = part; k < K; k += NP) {
            const float iw = __ldg(m.f_invW + k);
            const int ek = linE[(int64_t)k * ldl];
            *reinterpret_cast<float*>(sdC + (size_t)__ldg(m.fx32_slot + k) * 128) =
                fmaf(sW[k * 32] * iw * rho, arho, rho * __int_as_float(sE[k * 32]) * iw);
            sE[k * 32] = ek;
        }
    }
    fx_image_wait();
    __syncthreads();

    float w[kFxOwn];
    int ek[kFxOwn];
#pragma unroll
    for (int j = 0; j < kFxOwn; ++j) {
        w[j] = 0.0f;
        ek[j] = part + NP * j < K ? sE[__ldg(&f.sp[part + NP * j].k) * 32] : 0;
    }
    // each part's next reaction is loaded while this one is summed, also across the chunks
    const float* a = lin + i;
    Words32 x;
    if (im0[f.image_parts + part] < im0[f.image_parts + part + 1]) load_words32(m, im0, im0[f.image_parts + part], a, ldl, x);
    for (int c = 0; c < f.nchunk; ++c) {
        const unsigned char* im = im0 + (c & 1) * f.image;
        const unsigned char* in = im0 + ((c + 1) & 1) * f.image;
        fx_image_load(f, c + 1, im0 + ((c + 1) & 1) * f.image);
        const int q1 = im[f.image_parts + part + 1];
#pragma unroll 1
        for (int q = im[f.image_parts + part]; q < q1; ++q) {
            const int4* rec = reinterpret_cast<const int4*>(im + q * (int)sizeof(FxRxn32));
            const int4 o4 = rec[0], h = rec[1];                  // offsets; info, r, boff, eff0
            const int nr = h.x & 15, np = h.x >> 4 & 15, kind = h.x >> 8;
            const Words32 v = x;
            if (q + 1 < q1) load_words32(m, im, q + 1, a, ldl, x);
            const unsigned of[8] = {(unsigned)o4.x & 0xffffu, (unsigned)o4.x >> 16, (unsigned)o4.y & 0xffffu, (unsigned)o4.y >> 16,
                                    (unsigned)o4.z & 0xffffu, (unsigned)o4.z >> 16, (unsigned)o4.w & 0xffffu, (unsigned)o4.w >> 16};
            float dq = v.A * sV[0];
#pragma unroll
            for (int e = 0; e < kMaxSide; ++e)
                if (e < nr) dq = fmaf(v.br[e], *reinterpret_cast<const float*>(sdC + of[e]), dq);
#pragma unroll
            for (int e = 0; e < kMaxSide; ++e)
                if (e < np) dq = fmaf(v.bp[e], *reinterpret_cast<const float*>(sdC + of[4 + e]), dq);
            if (kind != 0) {
                float dM = sV[96];
                const int e1 = rec[2].x;
                for (int j = h.w; j < e1; ++j)
                    dM = fmaf(__ldg(m.f_eff_m1 + j),
                              *reinterpret_cast<const float*>(sdC + (size_t)__ldg(m.fx32_slot + __ldg(m.eff_sp + j)) * 128), dM);
                dq = fmaf(v.L, dM, dq);
            }
            *reinterpret_cast<int2*>(sQ + q * 256) = make_int2(__float_as_int(dq), v.er);
        }
        fx_image_wait();
        __syncthreads();
        if (c + 1 < f.nchunk && in[f.image_parts + part] < in[f.image_parts + part + 1])
            load_words32(m, in, in[f.image_parts + part], a, ldl, x);
        const uint32_t* spec = reinterpret_cast<const uint32_t*>(im + f.image_spec);
#pragma unroll
        for (int j = 0; j < kFxOwn; ++j)
            if (part + NP * j < K) {
                const uint32_t wd = spec[part + NP * j];
                const uint2* t = reinterpret_cast<const uint2*>(im + f.image_list) + (wd >> 8);
                float acc = w[j];
#pragma unroll 1
                for (int e = 0; e < (int)(wd & 255u); ++e) {
                    const uint2 x = t[e];
                    const int2 v = *reinterpret_cast<const int2*>(sQ + x.x);
                    acc = fmaf(__uint_as_float(x.y) * pow2f(v.y - ek[j]), __int_as_float(v.x), acc);
                }
                w[j] = acc;
            }
        __syncthreads();
    }
#pragma unroll
    for (int j = 0; j < kFxOwn; ++j)
        if (part + NP * j < K) sW[__ldg(&f.sp[part + NP * j].k) * 32] = w[j];
    __syncthreads();

    // The epilogue of jvp_lin32_kernel: the outputs by all parts, which leave what the point sums take in
    // shared memory (h_k/RT in the rows of dC_k, the sources' y_k and v_k in the reactions' rows where they
    // fit); the sums by the old number of parts.  (All of it by one part of four: 9 species / 21
    // reactions, 1,000,000 points, sources' product 763 us instead of 613.)
    const double Td = T[i], dTd = vT[i];
    const float Ti = narrow(Td), dT = narrow(dTd), rho = sV[32], arho = sV[64];
    const float inv_rho = RHS ? 1.0f / rho : 0.0f;
    const double arho_d = widen(arho);
    float* sH = reinterpret_cast<float*>(sdC);
    const bool stash = RHS && K <= f.rows;
#pragma unroll 2
    for (int k = part; k < K; k += NP) {
        double dw = scale2(widen(sW[k * 32]), sE[k * 32]);
        sH[k * 32] = lin[(slot_H32(m) + k) * ldl + i];
        if constexpr (RHS) {
            const float iw = __ldg(m.f_invW + k);
            if (stash)
                *reinterpret_cast<float2*>(sQ + k * 256) =
                    make_float2(narrow(Y[(int64_t)k * ld + i]) * iw, narrow(vY[(int64_t)k * ld + i]) * iw);
            dw = fma(widen(inv_rho / iw), dw, -fY[(int64_t)k * ldf + i] * arho_d);
        }
        if (live) d_omega[(int64_t)k * ld + i] = dw;
    }
    __syncthreads();
    if (part >= OLD) return;
    double hsum = 0.0;
    float cpm = 0.0f, dcpm = 0.0f;
#pragma unroll 2
    for (int k = part; k < K; k += OLD) {
        hsum = fma(widen(sH[k * 32]), scale2(widen(sW[k * 32]), sE[k * 32]), hsum);
        if constexpr (RHS) {
            const bool lo = __double_as_longlong(Td) <= __ldg(reinterpret_cast<const long long*>(m.Tmid) + k);
            const float* cf = m.f_cp + ((size_t)k * 2 + (lo ? 0 : 1)) * 8;
            const float4 c = __ldg(reinterpret_cast<const float4*>(cf));
            const float a5 = __ldg(cf + 4);
            const float cpk = fmaf(Ti, fmaf(Ti, fmaf(Ti, fmaf(Ti, a5, c.w), c.z), c.y), c.x);
            const float dcpk = fmaf(Ti, fmaf(Ti, fmaf(Ti, 4.0f * a5, 3.0f * c.w), 2.0f * c.z), c.y);
            float2 yv;
            if (stash) {
                yv = *reinterpret_cast<const float2*>(sQ + k * 256);
            } else {
                const float iw = __ldg(m.f_invW + k);
                yv = make_float2(narrow(Y[(int64_t)k * ld + i]) * iw, narrow(vY[(int64_t)k * ld + i]) * iw);
            }
            cpm = fmaf(yv.x, cpk, cpm);
            dcpm = fmaf(yv.y, cpk, fmaf(yv.x * dcpk, dT, dcpm));
        }
    }
    if constexpr (OLD > 1) {
        sR[part * 32] = hsum;
        if constexpr (RHS) {
            sR[(OLD + part) * 32] = widen(cpm);
            sR[(2 * OLD + part) * 32] = widen(dcpm);
        }
        asm volatile("bar.sync 1, %0;" ::"n"(32 * OLD) : "memory");
        if (part != 0) return;
        hsum = sR[0];
        double cpd = RHS ? sR[OLD * 32] : 0.0, dcpd = RHS ? sR[2 * OLD * 32] : 0.0;
#pragma unroll
        for (int q = 1; q < OLD; ++q) {
            hsum += sR[q * 32];
            if constexpr (RHS) {
                cpd += sR[(OLD + q) * 32];
                dcpd += sR[(2 * OLD + q) * 32];
            }
        }
        cpm = narrow(cpd);
        dcpm = narrow(dcpd);
    }
    if (live) {
        const uint32_t lo = reinterpret_cast<const uint32_t*>(lin)[slot_S(m) * ldl + i];
        const uint32_t hi = reinterpret_cast<const uint32_t*>(lin)[(slot_S(m) + 1) * ldl + i];
        const double S1 = __hiloint2double((int)hi, (int)lo);
        const double dhr = -kR * fma(dTd, S1, Td * hsum);
        if constexpr (RHS)
            d_hrr[i] = fma(dhr, widen(inv_rho / (8.314462618f * cpm)), -fT[i] * widen(arho + dcpm / cpm));
        else
            d_hrr[i] = dhr;
    }
}

template <int OLD, bool RHS>
cudaError_t launch_lin32_fx(const DevMech& m, int64_t n, int64_t ld, const double* T, const double* p, const double* Y,
                            const float* lin, int64_t ldl, const double* vT, const double* vY, double* d_omega,
                            double* d_hrr, const double* fT, const double* fY, int64_t ldf, cudaStream_t s) {
    const FxSet& f = lin32_set(m, OLD);
    const size_t smem = lin32_fx_smem(f, m.K, OLD);
    auto kern = f.np == 4 ? jvp_lin32_fx_kernel<4, OLD, RHS> : f.np == 8 ? jvp_lin32_fx_kernel<8, OLD, RHS>
              : f.np == 16 ? jvp_lin32_fx_kernel<16, OLD, RHS> : jvp_lin32_fx_kernel<32, OLD, RHS>;
    const cudaError_t e = ensure_smem((const void*)kern, smem);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)((n + 31) / 32), 32 * f.np, smem, s>>>(m, n, ld, T, p, Y, lin, ldl, vT, vY, d_omega, d_hrr, fT, fY, ldf);
    return cudaGetLastError();
}

template <bool RHS>
cudaError_t launch_lin32_fx(int old_np, const DevMech& m, int64_t n, int64_t ld, const double* T, const double* p,
                            const double* Y, const float* lin, int64_t ldl, const double* vT, const double* vY,
                            double* d_omega, double* d_hrr, const double* fT, const double* fY, int64_t ldf, cudaStream_t s) {
    if (old_np == 1) return launch_lin32_fx<1, RHS>(m, n, ld, T, p, Y, lin, ldl, vT, vY, d_omega, d_hrr, fT, fY, ldf, s);
    if (old_np == 2) return launch_lin32_fx<2, RHS>(m, n, ld, T, p, Y, lin, ldl, vT, vY, d_omega, d_hrr, fT, fY, ldf, s);
    return launch_lin32_fx<4, RHS>(m, n, ld, T, p, Y, lin, ldl, vT, vY, d_omega, d_hrr, fT, fY, ldf, s);
}

}  // namespace
}  // namespace nk
