// Links, site terms and full hops of two right-hand sides in packed FP32 on 4^4 blocks, from the
// block-ordered operator copies; shared by the SAP and the Dslash kernels.
#pragma once

#include "block44.cuh"
#include "f32x2.cuh"
#include "kernels.h"

namespace ddamg {

// ---- operator copies of the 4^4 blocks (common.cuh): all words of a block sit together, [word][site]
// W = U_mu at local site l of block c; on = false: zero, nothing is read
__device__ __forceinline__ void load_link44(cplx<float> (&W)[9], const LinksB& U, int c, int mu, int l, bool on = true) {
    const float4* q = U.p + (size_t)c * (20 * 256) + mu * (5 * 256) + l;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    float4 a = zero, b = zero, d = zero, e = zero, f = zero;
    if (on) a = __ldg(q), b = __ldg(q + 256), d = __ldg(q + 512), e = __ldg(q + 768), f = __ldg(q + 1024);
    W[0] = mk(a.x, a.y), W[1] = mk(a.z, a.w), W[2] = mk(b.x, b.y), W[3] = mk(b.z, b.w), W[4] = mk(d.x, d.y);
    W[5] = mk(d.z, d.w), W[6] = mk(e.x, e.y), W[7] = mk(e.z, e.w), W[8] = mk(f.x, f.y);
}
__device__ __forceinline__ void load_link44(cplx<float> (&W)[9], const LinksB16& U, int c, int mu, int l, bool on = true) {
    const uint4* q = U.p + (size_t)c * (12 * 256) + mu * (3 * 256) + l;
    uint4 a = make_uint4(0u, 0u, 0u, 0u), b = a;
    unsigned d = 0u;
    if (on) a = __ldg(q), b = __ldg(q + 256), d = __ldg(&(q + 512)->x);
    const unsigned w[9] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, d};
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const float2 f = h2f(w[k]);
        W[k] = mk(f.x, f.y);
    }
}
// y = (block h of the site term) x, h = 0, 1
template <int HB>
__device__ __forceinline__ void herm44(const CloverB& cl, int c, int l, const c2 (&x)[6], c2 (&y)[6]) {
    const float4* q = cl.p + (size_t)c * (18 * 256) + HB * (9 * 256) + l;
    float w[36];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const float4 v = __ldg(q + k * 256);
        w[4 * k] = v.x, w[4 * k + 1] = v.y, w[4 * k + 2] = v.z, w[4 * k + 3] = v.w;
    }
    herm6_apply2([&](int j) { return w[j]; }, x, y);
}
template <int HB>
__device__ __forceinline__ void herm44(const CloverB16& cl, int c, int l, const c2 (&x)[6], c2 (&y)[6]) {
    const uint4* q = cl.p + (size_t)c * (10 * 256) + HB * (5 * 256) + l;
    unsigned w[20];
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        const uint4 v = __ldg(q + k * 256);
        w[4 * k] = v.x, w[4 * k + 1] = v.y, w[4 * k + 2] = v.z, w[4 * k + 3] = v.w;
    }
    herm6_apply2(
        [&](int j) {
            const float2 f = h2f(w[j / 2]);
            return (j & 1) ? f.y : f.x;
        },
        x, y);
}

// both hops of D in direction MU with the field read from global memory
template <int MU, typename UT>
__device__ __forceinline__ void hop_pair44_global(const UT& U, const cplx<float>* z0, const cplx<float>* z1, int V, int L, int p, int c,
                                                  int bf, int bb, c2 (&acc)[12]) {
    cplx<float> W[9];
    const int f = nbr44<MU, true>(L, p, c, bf), b = nbr44<MU, false>(L, p, c, bb);
    load_link44(W, U, c, MU, (p << 7) | (L >> 1));
    hop_acc2<MU, true>(acc, [&](int k) { return c2pair(z0[(size_t)k * V + f], z1[(size_t)k * V + f]); }, W);
    load_link44(W, U, b >> 8, MU, b & 255);
    hop_acc2<MU, false>(acc, [&](int k) { return c2pair(z0[(size_t)k * V + b], z1[(size_t)k * V + b]); }, W);
}

}  // namespace ddamg
