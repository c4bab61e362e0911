// Device side of the Sec. III-C stopping test, shared by every engine.
#pragma once

#include <cmath>

#include "opf_internal.h"

namespace opf {

// Stopping test of Sec. III-C (plus the absolute gate on pres) from the six
// sums and the square roots of the first five.
__device__ __forceinline__ void apply_roots(DevStatus *st, const double s[6], const double root[5], double rho,
                                            long long add_iters) {
    const double pres = root[0];
    const double dres = rho * root[1];
    const double eprim = fmax(root[2], root[3]);
    const double edual = root[4];
    st->iter += add_iters;
    st->pres = pres;
    st->dres = dres;
    st->eprim = eprim;
    st->edual = edual;
    st->obj = s[5];
    bool finite = true;
    for (int q = 0; q < 6; ++q) finite = finite && isfinite(s[q]);
    st->numeric = finite ? 0 : 1;
    st->converged = (finite && pres <= st->eps_rel * eprim && dres <= st->eps_rel * edual &&
                     pres <= st->eps_abs_pres) ? 1 : 0;
    if (st->converged || st->numeric || st->iter >= st->max_iter) st->done = 1;
}

__device__ __forceinline__ void apply_test(DevStatus *st, const double s[6], double rho, long long add_iters) {
    double root[5];
    for (int q = 0; q < 5; ++q) root[q] = sqrt(s[q]);
    apply_roots(st, s, root, rho, add_iters);
}

// The same by a whole warp: s in shared memory, one square root per lane (an
// FP64 square root is some 20 instructions of 64 cycles each on this part's
// FP64 pipe, so the five run side by side); lane 0 updates *st.
__device__ __forceinline__ void apply_test_warp(DevStatus *st, const double *s, double rho, long long add_iters) {
    const int lane = threadIdx.x & 31;
    const double mine = lane < 5 ? sqrt(s[lane]) : 0.0;
    double root[5];
#pragma unroll
    for (int q = 0; q < 5; ++q) root[q] = __shfl_sync(0xffffffffu, mine, q);
    if (lane == 0) apply_roots(st, s, root, rho, add_iters);
}

// Sums of six quantities over the lanes of a warp, the quantities spread over
// the lanes as they are added: 9 FP64 adds per lane instead of the 30 of six
// butterflies (a warp's FP64 add occupies its sub-partition's FP64 pipe for
// about 64 cycles).  Lane l returns the sum of quantity l >> 2 (0 for 6, 7).
__device__ __forceinline__ double warp_sum6(const double a[6]) {
    const unsigned lane = threadIdx.x & 31u;
    const bool b4 = lane & 16u, b3 = lane & 8u, b2 = lane & 4u;
    double t[4], u[2];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const double hi = i < 2 ? a[4 + i] : 0.0;
        t[i] = (b4 ? hi : a[i]) + __shfl_xor_sync(0xffffffffu, b4 ? a[i] : hi, 16);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) u[i] = (b3 ? t[2 + i] : t[i]) + __shfl_xor_sync(0xffffffffu, b3 ? t[i] : t[2 + i], 8);
    double v = (b2 ? u[1] : u[0]) + __shfl_xor_sync(0xffffffffu, b2 ? u[0] : u[1], 4);
    v += __shfl_xor_sync(0xffffffffu, v, 2);
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    return v;
}

// Sums of six quantities over a CTA, red[w][q] per warp: thread q < 6 returns
// the sum of quantity q (in warp order).  Ends without a barrier after the sum.
__device__ __forceinline__ double cta_sum6(const double acc[6], double (*red)[6]) {
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const double v = warp_sum6(acc);
    if ((lane & 3) == 0 && lane < 24) red[w][lane >> 2] = v;
    __syncthreads();
    double t = 0.0;
    if (tid < 6)
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t += red[i][tid];
    return t;
}

}  // namespace opf
