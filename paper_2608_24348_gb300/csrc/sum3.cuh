// sum3.cuh -- long sums of float pairs, kept in three floats.
//
// The FP32 phases of the solver form their inner products as float pairs, one pair
// for a column of an element or a chunk of nodes (dot2_acc): its error grows with
// the number of terms, so a thread's and a warp's whole share are summed here.
// Every addition is error-free in the first two parts and the errors are gathered
// in the third (Ogita, Rump & Oishi 2005, K = 3): 72 bits, at least as accurate as
// adding the pairs in FP64, and off the FP64 pipe, whose additions (one a chunk
// and value, and a shuffle tree a warp) would take longer than an FP64 phase's.
// They cost 3 % of a solve (4 M nodes, N = 7, 12 inner iterations: 1.65 ms with the
// pairs summed as pairs, 1.70 so) and up to 6 % of a batch of small problems.
#pragma once

struct Sum3 {
    float a, b, c;
};

__device__ __forceinline__ float two_sum(float x, float y, float &err)
{
    const float s = __fadd_rn(x, y), v = __fsub_rn(s, x);
    err = __fadd_rn(__fsub_rn(x, __fsub_rn(s, v)), __fsub_rn(y, v));
    return s;
}

__device__ __forceinline__ void sum3_add(Sum3 &S, float a, float b, float c)
{
    float e1, e2, e3;
    S.a = two_sum(S.a, a, e1);
    const float t = two_sum(S.b, b, e2);
    S.b = two_sum(t, e1, e3);
    S.c = __fadd_rn(__fadd_rn(S.c, c), __fadd_rn(e2, e3));
}

__device__ __forceinline__ double sum3_value(const Sum3 &S) { return (double)S.a + ((double)S.b + (double)S.c); }

// The sums of a warp's two values: the first on lanes 0 to 15, the second on the
// others (each half hands the other its share of the other's value first).
__device__ __forceinline__ double warp_sum3(const Sum3 (&d)[2], unsigned lane)
{
    const bool up = lane >= 16;
    Sum3 S = up ? d[1] : d[0];
    const Sum3 o = up ? d[0] : d[1];
    sum3_add(S, __shfl_xor_sync(0xffffffffu, o.a, 16), __shfl_xor_sync(0xffffffffu, o.b, 16),
             __shfl_xor_sync(0xffffffffu, o.c, 16));
#pragma unroll
    for (int m = 8; m > 0; m >>= 1)
        sum3_add(S, __shfl_xor_sync(0xffffffffu, S.a, m), __shfl_xor_sync(0xffffffffu, S.b, m),
                 __shfl_xor_sync(0xffffffffu, S.c, m));
    return sum3_value(S);
}
