// An upper bound of the kernel P along a row of an event's window, for the fixed-point
// scatter (tsp_rec.cuh): no sum can overflow when every event's largest term is known.
#pragma once

#include <math.h>

#ifdef __CUDACC__
#define TSP_HD __host__ __device__ __forceinline__
#else
#define TSP_HD inline
#endif

namespace tsp {

// Along the row, u in [ulo, uhi] from the chord's centre,
//   Q = Qc + gam2 u,  aCb = alpha u + beta,
//   log2 P = C0 - log2(Q) / 2 + (log2(e) / 2) (aCb^2 / Q - 2 iz u^2).
// With the row's least Q, which is at an end, in both places the rest is a quadratic in
// u, largest at an end or, if it is concave, at its vertex.  For the events whose bound over the
// whole window (window_bound) is more than four times too large: their terms then found
// no room (130 mm, 5 sigma, 2e5 events at 4 mm: 2060 us an update, 252 with this, the general
// passes 412).  For all events it would take an upload 15% longer.
// On the GPU with the approximate functions, far within the 1% that the bound is widened by.
TSP_HD float bound_rsqrt(float x)
{
#ifdef __CUDA_ARCH__
    return rsqrtf(x);
#else
    return 1.0f / sqrtf(x);
#endif
}

TSP_HD float bound_div(float a, float b)
{
#ifdef __CUDA_ARCH__
    return __fdividef(a, b);
#else
    return a / b;
#endif
}

TSP_HD float row_p_bound(float Qc, float gam2, float alpha, float beta, float ulo, float uhi,
                         float C0, float iz, float half_log2e)
{
    const float q = fminf(fmaf(gam2, ulo, Qc), fmaf(gam2, uhi, Qc));
    if (!(q > 0.0f)) return INFINITY;
    const float rs = bound_rsqrt(q), i = rs * rs;
    const float a2 = alpha * alpha * i - 2.0f * iz, a1 = alpha * beta * i;
    const float top = a2 < 0.0f ? fminf(fmaxf(bound_div(-a1, a2), ulo), uhi) : ulo;
    const float f0 = fmaf(fmaf(a2, ulo, 2.0f * a1), ulo, beta * beta * i);
    const float f1 = fmaf(fmaf(a2, uhi, 2.0f * a1), uhi, beta * beta * i);
    const float f2 = fmaf(fmaf(a2, top, 2.0f * a1), top, beta * beta * i);
    return 1.01f * exp2f(fmaf(half_log2e, fmaxf(fmaxf(f0, f1), f2), C0)) * rs;
}

}  // namespace tsp
