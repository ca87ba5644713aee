// A thread's sum of floats that keeps what FP64 would, four values at a time:
// between flushes the values are summed exactly as three floats (Knuth's
// two-sum twice), two values per paired FP32 instruction, and a flush adds those
// to an FP64 sum. GB300's FP64 pipe takes 2 additions per clock and SM, so an
// FP64 addition per value would be the bound of kernels that add a value per
// amplitude: |a|^2 of every amplitude of n = 27 complex64 takes 0.53 ms with
// FP64 additions and 0.19 ms with these sums (the read of the state). flush()
// belongs outside the loop over the values: inside, under a condition, its FP64
// instructions were issued in every iteration (0.37 ms).
#pragma once

#include "device.cuh"

namespace qsim {

#ifdef __CUDACC__
struct FloatSum {
    double sum = 0.0;
    float2 a = {0.f, 0.f}, b = {0.f, 0.f}, c = {0.f, 0.f};  // a + b + c, both lanes: the values since the last flush
    __device__ __forceinline__ static float2 two_sum(float2 &s, float2 v) {
        const float2 t = padd(s, v), bv = psub(t, s);
        const float2 e = padd(psub(s, psub(t, bv)), psub(v, bv));
        s = t;
        return e;
    }
    __device__ __forceinline__ void add(const float *v) {
        float2 na = a, nb = b, nc = c;
#pragma unroll
        for (int j = 0; j < 4; j += 2) {
            const float2 e = two_sum(na, make_float2(v[j], v[j + 1]));
            nc = padd(nc, two_sum(nb, e));
        }
        if (fabsf(na.x) + fabsf(na.y) <= 3.402823466e38f) {
            a = na;
            b = nb;
            c = nc;
        } else {  // near the end of the floats' range, infinite or NaN: FP64's result
            flush();
            for (int j = 0; j < 4; ++j) sum += (double)v[j];
        }
    }
    __device__ __forceinline__ void flush() {
        sum += (double)a.x + ((double)b.x + (double)c.x);
        sum += (double)a.y + ((double)b.y + (double)c.y);
        a = b = c = make_float2(0.f, 0.f);
    }
    __device__ __forceinline__ double value() const { return sum; }
};
#endif  // __CUDACC__

}  // namespace qsim
