// LU factorization with partial pivoting of one N x N block in shared memory by one warp, the
// step shared by the block-Jacobi kernels (k_lu.cu, k_jac.cu).
//
// The block a has row stride S.  At step k the warp picks the largest |a_rk| over the rows
// r >= k not yet eliminated (lowest position on ties, NaN counted as +inf so that the order is
// total), swaps that row into position k, and updates the remaining (N - 1 - k)^2 entries against
// it.  On return row k holds L_k,0..k-1 (unit lower part) and U_k,k.. of the k-th pivot row with
// 1/U_kk in place of U_kk, and perm[k] the original index of that row.  A zero pivot (a singular
// block) is replaced by 1: the factors stay finite and GMRES, which only uses them as a
// preconditioner, still converges, more slowly.
//
// The FP64 pipe bounds it (16 cycles per warp instruction whatever the active lanes), so
// - the pivot search compares bit patterns as integers and reduces them with three warp
//   reductions (as double comparisons and shuffles it took about 20 FP64 warp instructions a
//   step, a fifth of the factorization's);
// - the lanes take the remaining square in tiles of 4 rows x 8 columns: ceil(m/4) ceil(m/8) warp
//   instructions for m remaining rows instead of m ceil(m/32) with a row per lane (1,960 against
//   2,410 over the 53 steps at N = 54; 1,620 if no lane were ever idle).  Every entry still takes
//   its updates in the order of the steps, so the factors are the same bits.
#pragma once
#include "nk_internal.cuh"

namespace nk {

__device__ __forceinline__ void warp_lu(double* a, const int N, const int S, const int lane, int32_t* perm) {
    constexpr unsigned kAll = 0xffffffffu;
    for (int r = lane; r < N; r += 32) perm[r] = r;
    __syncwarp();
    const int tr = lane >> 3, tc = lane & 7;
    for (int k = 0; k < N; ++k) {
        unsigned hi = 0, lo = 0, best = (unsigned)N;
        for (int r = k + lane; r < N; r += 32) {
            const unsigned long long b = (unsigned long long)__double_as_longlong(a[r * S + k]);
            unsigned h = (unsigned)(b >> 32) & 0x7fffffffu, l = (unsigned)b;
            if (h > 0x7ff00000u || (h == 0x7ff00000u && l != 0)) {              // NaN as +inf
                h = 0x7ff00000u;
                l = 0;
            }
            if (best == (unsigned)N || h > hi || (h == hi && l > lo)) {
                hi = h;
                lo = l;
                best = (unsigned)r;
            }
        }
        const unsigned mh = __reduce_max_sync(kAll, hi);
        const unsigned ml = __reduce_max_sync(kAll, hi == mh ? lo : 0u);
        const int pr = (int)__reduce_min_sync(kAll, hi == mh && lo == ml ? best : (unsigned)N);
        if (pr != k) {
            for (int j = lane; j < N; j += 32) {
                const double t = a[k * S + j];
                a[k * S + j] = a[pr * S + j];
                a[pr * S + j] = t;
            }
            if (lane == 0) {
                const int32_t t = perm[k];
                perm[k] = perm[pr];
                perm[pr] = t;
            }
            __syncwarp();
        }
        double pv = a[k * S + k];
        if ((__double_as_longlong(pv) << 1) == 0) pv = 1.0;
        const double inv = 1.0 / pv;
        const double* ap = a + k * S;
        for (int r = k + 1 + lane; r < N; r += 32) a[r * S + k] *= inv;
        __syncwarp();
        for (int r = k + 1 + tr; r < N; r += 4) {
            double* ar = a + r * S;
            const double l = ar[k];
#pragma unroll 4
            for (int j = k + 1 + tc; j < N; j += 8) ar[j] = fma(-l, ap[j], ar[j]);
        }
        if (lane == 0) a[k * S + k] = inv;
        __syncwarp();
    }
}

}  // namespace nk
