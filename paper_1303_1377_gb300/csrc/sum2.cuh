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
// kLaneWords of them; first < 32.  Eight words at a time without branches (zeros past the end), so that their loads
// and the error terms of their additions overlap.
constexpr int kLaneWords = 32;
__host__ __device__ __forceinline__ void lane_dot(const float4* a4, const float4* w4, int first, int cnt, Sum2& re, Sum2& im) {
    constexpr int B = 8;
#pragma unroll 1
    for (int j = 0; j < 32 * kLaneWords && j < cnt; j += 32 * B) {
        float4 a[B], v[B];
#pragma unroll
        for (int q = 0; q < B; ++q) {
            const int e = j + 32 * q + first;
            const bool on = e < cnt;
            a[q] = on ? a4[e] : float4{0.f, 0.f, 0.f, 0.f};
            v[q] = on ? w4[e] : float4{0.f, 0.f, 0.f, 0.f};
        }
#pragma unroll
        for (int q = 0; q < B; ++q) {
            re.add(fmaf(a[q].x, v[q].x, a[q].y * v[q].y) + fmaf(a[q].z, v[q].z, a[q].w * v[q].w));
            im.add(fmaf(a[q].x, v[q].y, -a[q].y * v[q].x) + fmaf(a[q].z, v[q].w, -a[q].w * v[q].z));
        }
    }
}

}  // namespace ddamg
