// The rotation of a one-sided Jacobi step, in few FP64 instructions.
#pragma once

#include <cuda_runtime.h>

namespace pne {

__device__ __forceinline__ int double_exponent(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// x 2^(1023 - e) truncated to FP32 (0 below FP32's range), and back, by bits
__device__ __forceinline__ float scaled_float(double x, int e)
{
    const int hi = __double2hiint(x), ex = ((hi >> 20) & 0x7ff) - e + 127;
    if (ex <= 0) return 0.f;
    return __int_as_float((hi & 0x80000000) | (min(ex, 254) << 23) | ((hi & 0xfffff) << 3) |
                          (int)((unsigned)__double2loint(x) >> 29));
}
__device__ __forceinline__ double widen(float x)        // normal x
{
    const int b = __float_as_int(x);
    return __hiloint2double((b & 0x80000000) | ((((b >> 23) & 0xff) + 896) << 20) | ((b & 0x7fffff) >> 3), b << 29);
}

// Cosine and sine of the rotation (x, y) -> (c x - s y, s x + c y) that makes two
// columns with squared norms a, b and inner product g != 0 orthogonal: tangent
// t = sign(z) / (|z| + sqrt(1 + z^2)), z = h / (2 g), h = b - a.  An FP64 division
// or square root is a dozen FP64 instructions, each 64 clocks of a warp's
// scheduler on this GPU, so t starts in FP32 (off by about 2^-22) and two Newton
// steps on g t^2 + h t - g, residual in FP64 and slope in FP32, take it to FP64:
// the error left is t^2 / (1 + t^2) times its square each time, 2^-45 and below
// FP64's rounding.  The second step matters although the first leaves columns
// that the next sweep would still rotate: an inner product just above the bound
// is rotated once and never again, and a small entry of V is a few such t (2.1e-14
// of its own size with one step, 4.1e-16 with two, as with division and root).
__device__ __forceinline__ void jacobi_rotation(double a, double b, double g, double &cs, double &sn)
{
    const double h = b - a;
    const int eh = max(double_exponent(h), double_exponent(g));
    const float hf = scaled_float(h, eh), g2 = 2.f * scaled_float(g, eh);
    const float t = (hf < 0.f ? -g2 : g2) / (fabsf(hf) + sqrtf(fmaf(hf, hf, g2 * g2)));
    if (fabsf(t) >= 1e-18f && fabsf(t) <= 1.5f) {
        const float slope = 1.f / fmaf(g2, t, hf);
        double td = widen(t);
#pragma unroll
        for (int step = 0; step < 2; ++step) {
            const float dt = -scaled_float(fma(fma(g, td, h), td, -g), eh) * slope;
            td += fabsf(dt) >= 1e-36f ? widen(dt) : 0.0;
        }
        // c = rsqrt(1 + t^2) in FP32 and s = t c miss c^2 + s^2 = 1 by r = O(1e-7), which
        // (1 + r)^(-1/2) to second order corrects
        const double c = widen(rsqrtf(fmaf(t, t, 1.f))), s = td * c;
        const double r = fma(s, s, fma(c, c, -1.0));
        const double k = fma(r, fma(r, 0.375, -0.5), 1.0);
        cs = c * k;
        sn = s * k;
    } else {                                 // graded beyond FP32: t = g / h to rounding
        cs = 1.0;
        sn = g / h;
    }
}

}  // namespace pne
