// Test harness: the FP32 lane sums of sum2.cuh on the host.  Built by the tests as a host-only shared library; the
// product never loads it.
#include "sum2.cuh"

// out[lane] = {re.s, re.e, im.s, im.e} of the 32 lanes of a warp
extern "C" void sum_lane_dot(const float* a, const float* w, int cnt, float* out) {
    for (int lane = 0; lane < 32; ++lane) {
        ddamg::Sum2 re, im;
        ddamg::lane_dot(reinterpret_cast<const float4*>(a), reinterpret_cast<const float4*>(w), lane, cnt, re, im);
        out[4 * lane] = re.s, out[4 * lane + 1] = re.e, out[4 * lane + 2] = im.s, out[4 * lane + 3] = im.e;
    }
}
