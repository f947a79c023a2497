// FP32 sums that keep the rounding error of every addition (TwoSum, Knuth) beside the total, for sums of tens of
// terms: an FP64 addition per term would issue at 1/64 of the FP32 rate.
#pragma once

#include <cuda_runtime.h>

#include <cmath>

namespace ddamg {

struct Sum2 {
    float s = 0.f, e = 0.f;  // the sum is s + e
    __host__ __device__ __forceinline__ void add(float t) {
        const float n = s + t, b = n - s;
        e += (s - (n - b)) + (t - b);
        s = n;
    }
};

// one lane's part of <a, w>, two complex numbers a float4: words first, first + 32, ... below cnt, at most
// kLaneWords of them
constexpr int kLaneWords = 32;
__host__ __device__ __forceinline__ void lane_dot(const float4* a4, const float4* w4, int first, int cnt, Sum2& re, Sum2& im) {
#pragma unroll 8
    for (int j = 0; j < kLaneWords; ++j) {
        const int e = first + 32 * j;
        if (e < cnt) {
            const float4 a = a4[e], v = w4[e];
            re.add(fmaf(a.x, v.x, a.y * v.y) + fmaf(a.z, v.z, a.w * v.w));
            im.add(fmaf(a.x, v.y, -a.y * v.x) + fmaf(a.z, v.w, -a.w * v.z));
        }
    }
}

}  // namespace ddamg
