// One-sided Jacobi of small matrices, in few FP64 instructions.
#pragma once

#include <cuda_runtime.h>

#include <cmath>

namespace pne {

constexpr int kJacobiDim = 16;               // most columns and rows
constexpr int kJacobiThreads = 128;          // of the block
constexpr int kJacobiLd = kJacobiDim + 1;    // column stride in shared memory

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
// is rotated once and never again, and a small entry of V is a few such t (a sine is
// off by up to 1.5e-14 of its own size with one step, 3.9e-16 with two, 4.3e-16 with
// division and root).  Weight passing of eight 3 x 3 networks of chi = 16 takes 99 ms
// with two steps, 95 with one.
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

// ---- one-sided Jacobi (Hestenes) of the columns of a matrix in shared memory
// (entry (row, c) at c * kJacobiLd + row).  A round of the tournament rotates up to
// eight disjoint pairs at once, sixteen threads to a pair and a row each: the
// four warps of the block.  An FP64 instruction takes a warp's scheduler about
// 64 clocks on this GPU (two lanes per clock and SM), an FP32 or integer one
// two, so a round is as long as the FP64 instructions of one warp: the sums
// halve their list at each exchange (5 additions for the three inner products,
// not 12), and the rotation takes ten (jacobi_rotation).  At n = 16 a round on
// one warp, four rows to a lane, took 5.2 k clocks (two thirds of a bond update:
// 1.03 M of 1.5 M clocks).
struct JacobiPair {
    int c0, c1;
    bool on;
};

// Pair `pr` of round rd among n columns (n2 = n rounded up to even): the circle
// method; an odd n leaves one column out.
__device__ __forceinline__ JacobiPair jacobi_pair(int pr, int rd, int n, int n2)
{
    const int m = n2 - 1;
    int c0 = rd + pr, c1 = rd + m - pr;
    c0 = pr == 0 ? m : (c0 >= m ? c0 - m : c0);
    c1 = pr == 0 ? rd : (c1 >= m ? c1 - m : c1);
    const int lo = c0 < c1 ? c0 : c1, hi = c0 < c1 ? c1 : c0;
    return {lo, hi, pr < n2 / 2 && hi < n};
}

// On return the columns of W are orthogonal, sorted by their norms (sig)
// descending; the rotations are accumulated on V (identity on entry, the same
// layout), whose columns move along.  The whole block.
__device__ inline void jacobi_columns(double *W, double *V, double *sig, int n)
{
    const int lane = threadIdx.x & 31, pr = threadIdx.x >> 4, row = threadIdx.x & 15, base = lane & 16;
    const int n2 = n + (n & 1), rounds = n2 - 1;
    for (int sweep = 0; sweep < 60 && n > 1; ++sweep) {
        int rotated = 0;
        for (int rd = 0; rd < rounds; ++rd) {
            const JacobiPair p = jacobi_pair(pr, rd, n, n2);
            const bool in = p.on && row < n;
            double *wp = W + p.c0 * kJacobiLd + row, *wq = W + p.c1 * kJacobiLd + row;
            const double x = in ? *wp : 0.0, y = in ? *wq : 0.0;
            // sums over the 16 rows of x^2, y^2 and x y
            double s0 = x * x, s1 = y * y;
            const double s2 = x * y;
            const bool u8 = lane & 8, u4 = lane & 4;
            double g0 = __shfl_xor_sync(0xffffffffu, u8 ? s0 : s2, 8), g1 = __shfl_xor_sync(0xffffffffu, s1, 8);
            s0 = (u8 ? s2 : s0) + g0;
            s1 = s1 + g1;
            g0 = __shfl_xor_sync(0xffffffffu, u4 ? s0 : s1, 4);
            s0 = (u4 ? s1 : s0) + g0;                 // lanes 0: x^2, 4: y^2, 8: x y
            s0 += __shfl_xor_sync(0xffffffffu, s0, 2);
            s0 += __shfl_xor_sync(0xffffffffu, s0, 1);
            const double a = __shfl_sync(0xffffffffu, s0, base), b = __shfl_sync(0xffffffffu, s0, base + 4),
                         g = __shfl_sync(0xffffffffu, s0, base + 8);
            // |g| <= 1e-15 sqrt(a b)
            const int e = max(double_exponent(a), double_exponent(b));
            const float af = scaled_float(a, e), bf = scaled_float(b, e), gf = scaled_float(g, e);
            bool small = fabsf(gf) <= 1e-15f * sqrtf(af) * sqrtf(bf);
            if (af == 0.f || bf == 0.f) small = fabs(g) <= 1e-15 * sqrt(a) * sqrt(b);   // norms 2^63 apart
            const bool turn = p.on && !(small || g == 0.0);
            if (turn) {
                double cs, sn;
                jacobi_rotation(a, b, g, cs, sn);
                if (row < n) {
                    *wp = cs * x - sn * y;
                    *wq = sn * x + cs * y;
                    {
                        double *vp = V + p.c0 * kJacobiLd + row, *vq = V + p.c1 * kJacobiLd + row;
                        const double vx = *vp, vy = *vq;
                        *vp = cs * vx - sn * vy;
                        *vq = sn * vx + cs * vy;
                    }
                }
            }
            rotated |= __syncthreads_or(turn);
        }
        if (!rotated) break;
    }
    if (threadIdx.x >= 32) return;
    __syncwarp();
    // norms, a column per lane, and the descending order (ties by index; a NaN
    // counts as infinite, so that every place is filled)
    double norm = -1.0;
    if (lane < n) {
        double s2 = 0.0;
        for (int row = 0; row < n; ++row) s2 = fma(W[lane * kJacobiLd + row], W[lane * kJacobiLd + row], s2);
        norm = sqrt(s2);
    }
    const double key = norm == norm ? norm : INFINITY;
    int at = 0;
    for (int c = 0; c < n; ++c) {
        const double o = __shfl_sync(0xffffffffu, key, c);
        at += (o > key || (o == key && c < lane)) ? 1 : 0;
    }
    double col[kJacobiDim], vcol[kJacobiDim];
    if (lane < n)
        for (int row = 0; row < n; ++row) {
            col[row] = W[lane * kJacobiLd + row];
            vcol[row] = V[lane * kJacobiLd + row];
        }
    __syncwarp();
    if (lane < n) {
        sig[at] = norm;
        for (int row = 0; row < n; ++row) {
            W[at * kJacobiLd + row] = col[row];
            V[at * kJacobiLd + row] = vcol[row];
        }
    }
    __syncwarp();
}

}  // namespace pne
