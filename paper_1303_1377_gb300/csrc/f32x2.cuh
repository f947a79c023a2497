// Packed FP32 arithmetic: one instruction on two FP32 numbers (add/sub/mul/fma.rn.f32x2, each half
// rounded as the scalar instruction rounds), used with the two halves holding the same component of
// two right-hand sides.
#pragma once

#include "dirac.cuh"

namespace ddamg {

__device__ __forceinline__ unsigned long long f2_bits(float2 a) { return *reinterpret_cast<unsigned long long*>(&a); }
__device__ __forceinline__ float2 f2_of(unsigned long long u) { return *reinterpret_cast<float2*>(&u); }
__device__ __forceinline__ float2 f2add(float2 a, float2 b) {
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(f2_bits(a)), "l"(f2_bits(b)));
    return f2_of(d);
}
__device__ __forceinline__ float2 f2sub(float2 a, float2 b) {
    unsigned long long d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(f2_bits(a)), "l"(f2_bits(b)));
    return f2_of(d);
}
__device__ __forceinline__ float2 f2mul(float2 a, float2 b) {
    unsigned long long d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(f2_bits(a)), "l"(f2_bits(b)));
    return f2_of(d);
}
__device__ __forceinline__ float2 f2fma(float2 a, float2 b, float2 c) {
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(f2_bits(a)), "l"(f2_bits(b)), "l"(f2_bits(c)));
    return f2_of(d);
}
__device__ __forceinline__ float2 f2dup(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 f2neg(float2 a) { return make_float2(-a.x, -a.y); }

// one complex component of two right-hand sides
struct c2 {
    float2 re, im;
};
__device__ __forceinline__ c2 c2zero() { return {make_float2(0.f, 0.f), make_float2(0.f, 0.f)}; }
__device__ __forceinline__ c2 c2pair(cplx<float> a, cplx<float> b) { return {make_float2(a.re, b.re), make_float2(a.im, b.im)}; }
__device__ __forceinline__ c2 operator+(c2 a, c2 b) { return {f2add(a.re, b.re), f2add(a.im, b.im)}; }
__device__ __forceinline__ c2 operator-(c2 a, c2 b) { return {f2sub(a.re, b.re), f2sub(a.im, b.im)}; }
__device__ __forceinline__ c2 c2scale(float s, c2 a) { return {f2mul(f2dup(s), a.re), f2mul(f2dup(s), a.im)}; }
// a + s b for a power of two (or any) factor s
__device__ __forceinline__ c2 c2axpy(c2 a, float s, c2 b) { return {f2fma(f2dup(s), b.re, a.re), f2fma(f2dup(s), b.im, a.im)}; }
__device__ __forceinline__ float4 c2_f4(c2 a) { return make_float4(a.re.x, a.re.y, a.im.x, a.im.y); }
__device__ __forceinline__ c2 c2_of(float4 v) { return {make_float2(v.x, v.y), make_float2(v.z, v.w)}; }

// a + i^P b (P mod 4)
template <int P>
__device__ __forceinline__ c2 c2_add_ipow(c2 a, c2 b) {
    if constexpr ((P & 3) == 0) return {f2add(a.re, b.re), f2add(a.im, b.im)};
    else if constexpr ((P & 3) == 1) return {f2sub(a.re, b.im), f2add(a.im, b.re)};
    else if constexpr ((P & 3) == 2) return {f2sub(a.re, b.re), f2sub(a.im, b.im)};
    else return {f2add(a.re, b.im), f2sub(a.im, b.re)};
}

// acc += hop of the neighbour's spinor pn (pn(k) gives component k) through link W in direction MU,
// forward or backward (hop_acc of dirac.cuh on two right-hand sides, the same order of operations)
template <int MU, bool FWD, typename PN>
__device__ __forceinline__ void hop_acc2(c2 (&acc)[12], const PN& pn, const cplx<float> (&W)[9]) {
    using B = SpinB<MU>;
    constexpr int S = FWD ? 2 : 0;  // h = up -+ i^p low
    c2 h[2][3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const c2 l2 = pn(6 + c), l3 = pn(9 + c);
        h[0][c] = c2_add_ipow<B::p0 + S>(pn(c), B::c0 ? l3 : l2);
        h[1][c] = c2_add_ipow<B::p1 + S>(pn(3 + c), B::c1 ? l3 : l2);
    }
    float2 n[2][3];  // the negated part that the complex product subtracts
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int c = 0; c < 3; ++c) n[s][c] = f2neg(FWD ? h[s][c].im : h[s][c].re);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        c2 g[2];
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const cplx<float> w = FWD ? W[a * 3 + b] : W[b * 3 + a];
            const float2 wr = f2dup(w.re), wi = f2dup(w.im);
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                const c2 v = h[s][b];
                if (b == 0) g[s].re = f2mul(wr, v.re), g[s].im = f2mul(wr, v.im);
                else g[s].re = f2fma(wr, v.re, g[s].re), g[s].im = f2fma(wr, v.im, g[s].im);
                if (FWD) g[s].re = f2fma(wi, n[s][b], g[s].re), g[s].im = f2fma(wi, v.re, g[s].im);
                else g[s].re = f2fma(wi, v.im, g[s].re), g[s].im = f2fma(wi, n[s][b], g[s].im);
            }
        }
        acc[a] = acc[a] + g[0];
        acc[3 + a] = acc[3 + a] + g[1];
        acc[6 + a] = c2_add_ipow<B::hp0 + S>(acc[6 + a], g[B::hc0]);
        acc[9 + a] = c2_add_ipow<B::hp1 + S>(acc[9 + a], g[B::hc1]);
    }
}

// y = (hermitian 6x6 block with packed entries cf(0..35)) x
template <typename CF>
__device__ __forceinline__ void herm6_apply2(const CF& cf, const c2 (&x)[6], c2 (&y)[6]) {
    c2 n[6];
#pragma unroll
    for (int a = 0; a < 6; ++a) {
        n[a] = {f2neg(x[a].re), f2neg(x[a].im)};
        const float2 d = f2dup(cf(a));
        y[a] = {f2mul(d, x[a].re), f2mul(d, x[a].im)};
    }
    int m = 0;
#pragma unroll
    for (int a = 0; a < 6; ++a) {
#pragma unroll
        for (int b = a + 1; b < 6; ++b) {
            const float2 er = f2dup(cf(6 + 2 * m)), ei = f2dup(cf(7 + 2 * m));
            y[a].re = f2fma(er, x[b].re, y[a].re);
            y[a].re = f2fma(ei, n[b].im, y[a].re);
            y[a].im = f2fma(er, x[b].im, y[a].im);
            y[a].im = f2fma(ei, x[b].re, y[a].im);
            y[b].re = f2fma(er, x[a].re, y[b].re);
            y[b].re = f2fma(ei, x[a].im, y[b].re);
            y[b].im = f2fma(er, x[a].im, y[b].im);
            y[b].im = f2fma(ei, n[a].re, y[b].im);
            ++m;
        }
    }
}

}  // namespace ddamg
