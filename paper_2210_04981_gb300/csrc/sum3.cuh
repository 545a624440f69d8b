// Sums of floats carried in three floats (72 bits) at FP32 rates, for
// reductions whose result is a double or whose terms cancel.  FP64 adds run at
// 1/64 of the FP32 rate on this chip; a pair of floats (48 bits) is that fast
// too, but drops bits that a double keeps.  Host compilers take this file as
// well.
#pragma once

#ifdef __CUDACC__
#define HDOF_SUM3_FN __host__ __device__ __forceinline__
#else
#define HDOF_SUM3_FN inline
#endif

namespace hdof {

// a + b as its rounded value and the exact rest (Knuth's TwoSum)
HDOF_SUM3_FN float two_sum(float a, float b, float& rest) {
#ifdef __CUDA_ARCH__
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    rest = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
#else
    const float s = a + b, bb = s - a;
    rest = (a - (s - bb)) + (b - bb);
#endif
    return s;
}

// s0 the running sum, s1 the sum of its rounding errors, s2 the sum of theirs
// (Klein's second-order summation): n terms leave an error of about n^3 2^-72
// of the sum of their magnitudes at worst, far below a double's n 2^-53 at
// the few hundred terms of a thread and a warp.
struct Sum3 {
    float s0, s1, s2;
    HDOF_SUM3_FN void add(float x) {
        float e0, e1;
        s0 = two_sum(s0, x, e0);
        s1 = two_sum(s1, e0, e1);
        s2 += e1;
    }
    // x and the rounding error x_rest that it was left with
    HDOF_SUM3_FN void add(float x, float x_rest) {
        add(x);
        float e1;
        s1 = two_sum(s1, x_rest, e1);
        s2 += e1;
    }
    HDOF_SUM3_FN void add(const Sum3& o) {
        float e0, e1, e2;
        s0 = two_sum(s0, o.s0, e0);
        s1 = two_sum(s1, o.s1, e1);
        s1 = two_sum(s1, e0, e2);
        s2 = (s2 + o.s2) + (e1 + e2);
    }
    HDOF_SUM3_FN double value() const { return (double)s0 + ((double)s1 + (double)s2); }
};

#ifdef __CUDACC__
__device__ __forceinline__ Sum3 shfl_xor(const Sum3& s, int lanes) {
    return Sum3{__shfl_xor_sync(0xffffffffu, s.s0, lanes), __shfl_xor_sync(0xffffffffu, s.s1, lanes),
                __shfl_xor_sync(0xffffffffu, s.s2, lanes)};
}
#endif

}  // namespace hdof
