// Float-float dot products of the strip rows.
#pragma once

#include <cuda_runtime.h>

namespace pne {

struct ffp { float h, l; };

__device__ __forceinline__ ffp split_double(double x)
{
    const float h = (float)x;
    return {h, (float)(x - (double)h)};
}

// A compensated dot product of N pairs on the FP32 pipes, term by term: the running
// sum by Knuth's two-sum, its error, the product's own and the low-part cross
// products gathered in one FP32 compensation, about 2^-48 of sum |a x| in all, where
// the FP64 pipe of this part retires 1/60 of the FP32 rate.
// From N = 16 on the two-sum's second difference is taken from the unrounded product
// by an FMA and so carries the product's error too: ten instructions a term.  It
// rounds once more where both differences are non-zero, that is where a term is about
// as large as the sum: 0.3 to 0.7% in the rms error of 2 to 4 terms, 0.15% of 9, below
// 0.07% of 16 and more (1.6 M sums each in numpy; 40,000 on the GPU: 0.03% of 16, none
// of 25 and 64).  Shorter sums split the product by an FMA of its own, twelve
// instructions: the first site of a row and bond dimensions 2 and 3 (row products with
// ten and with twelve, ms: chi 2, 12 wide, 16 tensors 18.95, 18.90; chi 3, 9 wide, 8
// tensors 9.0, 9.3).  At chi = 4 twelve everywhere take 116 ms where ten take 103 (8
// tensors 10 wide), and end no nearer to 64 bits (1.5e-12 against 1.4e-12).
template <int N>
struct ff_dot {
    static constexpr bool kSplit = N < 16;
    float sh, c;
    __device__ __forceinline__ void term(int i, float ah, float al, float xh, float xl)
    {
        const float pr = __fmul_rn(ah, xh);
        if (i == 0) {
            sh = pr;
            c = __fmaf_rn(ah, xh, -pr);
        } else {
            const float t = __fadd_rn(sh, pr);
            const float bb = __fsub_rn(t, sh);
            const float q = __fsub_rn(sh, __fsub_rn(t, bb));
            if (kSplit) c = __fadd_rn(c, __fadd_rn(__fadd_rn(q, __fsub_rn(pr, bb)), __fmaf_rn(ah, xh, -pr)));
            else c = __fadd_rn(c, __fadd_rn(q, __fmaf_rn(ah, xh, -bb)));
            sh = t;
        }
        c = __fmaf_rn(ah, xl, c);
        c = __fmaf_rn(al, xh, c);
    }
    __device__ __forceinline__ ffp value() const
    {
        const float hi = __fadd_rn(sh, c);
        return {hi, __fsub_rn(c, __fsub_rn(hi, sh))};
    }
};

}  // namespace pne
