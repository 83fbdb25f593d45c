// Thermodynamic properties per point: NASA-7 species c_p, h, g and the mass-based mixture
// c_p and h, mean molar mass and ideal-gas density (Eq. 1b-1d of the paper).
// One thread per point; species rows are read coalesced across the warp (SoA layout).  The species
// polynomials are integer ones (nk_thermo.cuh) for 64 K <= T < 4096 K, doubles elsewhere: in
// doubles alone the FP64 pipe bounded the kernel (25 operations per species and point, 1.04 of its
// measured rate); four per species are left.  Unrolled, so that a few points, which wait for each species'
// coefficients, wait less often (53 species, 5,000 points: 66.8 -> 57 us).
#include "nk_thermo.cuh"

namespace nk {
namespace {

constexpr int kBlk = 128;

__global__ void __launch_bounds__(kBlk) thermo_kernel(DevMech m, int64_t n, int64_t ld,
                                                      const double* __restrict__ T, const double* __restrict__ p,
                                                      const double* __restrict__ Y, double* __restrict__ cp_mix,
                                                      double* __restrict__ h_mix, double* __restrict__ Wbar,
                                                      double* __restrict__ rho, double* __restrict__ cp_k,
                                                      double* __restrict__ h_k, double* __restrict__ g_k) {
    const int64_t i = (int64_t)blockIdx.x * kBlk + threadIdx.x;
    if (i >= n) return;
    const double Ti = T[i];
    const double lnT = log(Ti), invT = 1.0 / Ti, RT = kR * Ti;
    double s = 0.0, cp = 0.0, h = 0.0;
    const ThT t = th_fractions(m, Ti, lnT);
    if (t.ok) {
#pragma unroll 3
        for (int k = 0; k < m.K; ++k) {
            const FxThermo* x = m.th + k;
            const double2 head = __ldg(reinterpret_cast<const double2*>(x));             // T_mid; sh[0], sh[1]
            const bool lo = __double_as_longlong(Ti) <= __double_as_longlong(head.x);    // (both positive)
            const int64_t* c = lo ? x->c[0] : x->c[1];
            const FxFrac u = lo ? t.lo : t.hi;
            const double yw = Y[(int64_t)k * ld + i] * __ldg(m.invW + k);
            const double cpk = th_cp(c, u, __double2loint(head.y)), hk = th_h(c, u, __double2hiint(head.y));
            s += yw;
            cp = fma(yw, cpk, cp);
            h = fma(yw, hk, h);
            if (cp_k) cp_k[(int64_t)k * ld + i] = cpk;
            if (h_k) h_k[(int64_t)k * ld + i] = hk;
            if (g_k) g_k[(int64_t)k * ld + i] = th_g(c, u, t.ln, __ldg(&x->sh[2]));
        }
        const double wb = 1.0 / s;
        if (cp_mix) cp_mix[i] = cp;
        if (h_mix) h_mix[i] = h;
        if (Wbar) Wbar[i] = wb;
        if (rho) rho[i] = p[i] * wb * invT * kInvR;
        return;
    }
#pragma unroll 2
    for (int k = 0; k < m.K; ++k) {
        const double yw = Y[(int64_t)k * ld + i] * __ldg(m.invW + k);
        const double* c = nasa_range(m, k, Ti);
        const double cpR = nasa_cpR(c, Ti);
        const double hRT = nasa_hRT(c, Ti, invT);
        s += yw;
        cp = fma(yw, cpR, cp);
        h = fma(yw, hRT, h);
        if (cp_k) cp_k[(int64_t)k * ld + i] = kR * cpR;
        if (h_k) h_k[(int64_t)k * ld + i] = RT * hRT;
        if (g_k) g_k[(int64_t)k * ld + i] = RT * nasa_gRT(c, Ti, lnT, invT);
    }
    const double wb = 1.0 / s;
    if (cp_mix) cp_mix[i] = kR * cp;
    if (h_mix) h_mix[i] = RT * h;
    if (Wbar) Wbar[i] = wb;
    if (rho) rho[i] = p[i] * wb * invT * kInvR;
}

}  // namespace

cudaError_t launch_thermo(const DevMech& m, int64_t n, int64_t ld, const double* T, const double* p,
                          const double* Y, double* cp_mix, double* h_mix, double* Wbar, double* rho,
                          double* cp_k, double* h_k, double* g_k, cudaStream_t s) {
    const int64_t grid = (n + kBlk - 1) / kBlk;
    thermo_kernel<<<(unsigned)grid, kBlk, 0, s>>>(m, n, ld, T, p, Y, cp_mix, h_mix, Wbar, rho, cp_k, h_k, g_k);
    return cudaGetLastError();
}

}  // namespace nk
