// Double-word D on FP32 fields: D z with an FP64-accurate result.
#include <cuda_fp16.h>

#include <algorithm>

#include "dw.cuh"
#include "f32x2.cuh"
#include "kernels.h"

namespace ddamg {

// ---------------------------------------------------------------------------
// D z for an FP32 field z with an FP64-accurate result, evaluated in double-word
// FP32 arithmetic (pairs hi + lo of floats; error-free transformations TwoSum
// (Knuth) and TwoProduct via FMA, as in Joldes, Muller, Popescu, "Tight and
// rigorous error bounds for basic building blocks of double-word arithmetic",
// ACM TOMS 2017).  Used for w = D z_k inside FGMRES, where z_k is the V-cycle
// output and hence exactly an FP32 vector.  On GB300 an FP64 instruction costs
// about sixty FP32 instructions, and the double-word form needs about twelve per
// real multiply-add, with relative accuracy ~1e-14.
// Links and site terms are stored as double-word pairs (same bytes as FP64).
// ---------------------------------------------------------------------------
namespace {

__device__ __forceinline__ cdw ld_cdw(const float4* p) {
    float4 v = __ldg(p);
    return {{v.x, v.y}, {v.z, v.w}};
}

__device__ __forceinline__ cdw cdw_ipow_rt(const cdw& a, int p) {
    cdw b = (p & 1) ? cdw{dw_neg(a.im), a.re} : a;
    return (p & 2) ? cdw{dw_neg(b.re), dw_neg(b.im)} : b;
}

// one hop of D (direction mu, orientation fwd, given at run time) in double-word arithmetic
__device__ __noinline__ void dw_hop_rt(cdw (&acc)[12], const cplx<float>* __restrict__ in, int V, int nb, const float4* __restrict__ U,
                                       int link_site, int mu, bool fwd) {
    const int c0 = c_spinb[mu][0], p0 = c_spinb[mu][1], c1 = c_spinb[mu][2], p1 = c_spinb[mu][3];
    const int hc0 = c_spinb[mu][4], hp0 = c_spinb[mu][5], hc1 = c_spinb[mu][6], hp1 = c_spinb[mu][7];
    cdw h[2][3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        cplx<float> u0 = in[(size_t)(0 * 3 + c) * V + nb], u1 = in[(size_t)(1 * 3 + c) * V + nb];
        cplx<float> l2 = in[(size_t)(2 * 3 + c) * V + nb], l3 = in[(size_t)(3 * 3 + c) * V + nb];
        cdw b0 = cdw_ipow_rt(c0 ? cdw{{l3.re, 0.f}, {l3.im, 0.f}} : cdw{{l2.re, 0.f}, {l2.im, 0.f}}, p0);
        cdw b1 = cdw_ipow_rt(c1 ? cdw{{l3.re, 0.f}, {l3.im, 0.f}} : cdw{{l2.re, 0.f}, {l2.im, 0.f}}, p1);
        cdw a0 = {{u0.re, 0.f}, {u0.im, 0.f}}, a1 = {{u1.re, 0.f}, {u1.im, 0.f}};
        h[0][c] = fwd ? cdw_sub(a0, b0) : cdw_add(a0, b0);
        h[1][c] = fwd ? cdw_sub(a1, b1) : cdw_add(a1, b1);
    }
    cdw W[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) W[q] = ld_cdw(U + (size_t)(mu * 9 + q) * V + link_site);
    cdw gv[2][3];
#pragma unroll
    for (int s = 0; s < 2; ++s) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            cdw t = cdw_zero();
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                if (fwd) cdw_mac(t, W[a * 3 + b], h[s][b]);
                else cdw_mac_conj(t, W[b * 3 + a], h[s][b]);
            }
            t.re = dw_norm(t.re);
            t.im = dw_norm(t.im);
            gv[s][a] = t;
            acc[s * 3 + a] = cdw_add(acc[s * 3 + a], t);
        }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        cdw l0 = cdw_ipow_rt(hc0 ? gv[1][c] : gv[0][c], hp0);
        cdw l1 = cdw_ipow_rt(hc1 ? gv[1][c] : gv[0][c], hp1);
        acc[2 * 3 + c] = fwd ? cdw_sub(acc[2 * 3 + c], l0) : cdw_add(acc[2 * 3 + c], l0);
        acc[3 * 3 + c] = fwd ? cdw_sub(acc[3 * 3 + c], l1) : cdw_add(acc[3 * 3 + c], l1);
    }
}

}  // namespace

// one right-hand side: a thread per site, one warp per CTA
template <bool OUT_DW>
__global__ void __launch_bounds__(128) dslash_dw_kernel(Geom g, const float4* __restrict__ U, const float2* __restrict__ clov,
                                                        const cplx<float>* __restrict__ inr, void* __restrict__ outp) {
    const int i = blockIdx.x * 32 + threadIdx.x;
    if (i >= g.V) return;
    cdw acc[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) acc[k] = cdw_zero();
#pragma unroll 1
    for (int d = 0; d < 8; ++d) {
        const int nb = fine_nbr(g, i, d);
        const bool fwd = (d & 1) == 0;
        dw_hop_rt(acc, inr, g.V, nb, U, fwd ? i : nb, d >> 1, fwd);
    }
    // site term: y = A x with two packed hermitian 6x6 blocks (double-word entries), x FP32
    cdw y[12];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        float x[12];
#pragma unroll
        for (int a = 0; a < 6; ++a) {
            cplx<float> v = inr[(size_t)(h * 6 + a) * g.V + i];
            x[2 * a] = v.re;
            x[2 * a + 1] = v.im;
        }
        const float2* base = clov + (size_t)(h * 36) * g.V + i;
#pragma unroll
        for (int a = 0; a < 6; ++a) {
            float2 dv = __ldg(base + (size_t)a * g.V);
            dw d = {dv.x, dv.y};
            cdw t = cdw_zero();
            dw_macf(t.re, d, x[2 * a]);
            dw_macf(t.im, d, x[2 * a + 1]);
            y[h * 6 + a] = t;
        }
        int q = 0;
#pragma unroll
        for (int a = 0; a < 6; ++a) {
#pragma unroll
            for (int b = a + 1; b < 6; ++b) {
                float2 mr = __ldg(base + (size_t)(6 + 2 * q) * g.V), mi = __ldg(base + (size_t)(7 + 2 * q) * g.V);
                dw m_re = {mr.x, mr.y}, m_im = {mi.x, mi.y};
                // y[a] += m x[b];  y[b] += conj(m) x[a]
                dw_macf(y[h * 6 + a].re, m_re, x[2 * b]);
                dw_macf(y[h * 6 + a].re, dw_neg(m_im), x[2 * b + 1]);
                dw_macf(y[h * 6 + a].im, m_re, x[2 * b + 1]);
                dw_macf(y[h * 6 + a].im, m_im, x[2 * b]);
                dw_macf(y[h * 6 + b].re, m_re, x[2 * a]);
                dw_macf(y[h * 6 + b].re, m_im, x[2 * a + 1]);
                dw_macf(y[h * 6 + b].im, m_re, x[2 * a + 1]);
                dw_macf(y[h * 6 + b].im, dw_neg(m_im), x[2 * a]);
                ++q;
            }
        }
    }
    if (OUT_DW) {
        float4* o = reinterpret_cast<float4*>(outp);
#pragma unroll
        for (int k = 0; k < 12; ++k) {
            dw re = dw_norm(dw_add(y[k].re, {-0.5f * acc[k].re.h, -0.5f * acc[k].re.l}));
            dw im = dw_norm(dw_add(y[k].im, {-0.5f * acc[k].im.h, -0.5f * acc[k].im.l}));
            o[(size_t)k * g.V + i] = make_float4(re.h, re.l, im.h, im.l);
        }
    } else {
        cplx<double>* o = reinterpret_cast<cplx<double>*>(outp);
#pragma unroll
        for (int k = 0; k < 12; ++k) {
            double re = (double)y[k].re.h + (double)y[k].re.l - 0.5 * ((double)acc[k].re.h + (double)acc[k].re.l);
            double im = (double)y[k].im.h + (double)y[k].im.l - 0.5 * ((double)acc[k].im.h + (double)acc[k].im.l);
            o[(size_t)k * g.V + i] = mk(re, im);
        }
    }
}

// ---------------------------------------------------------------------------
// Two right-hand sides per thread in packed FP32 (f32x2.cuh): the same double-word operations, each issued
// once for two fields, with the links' and site terms' words loaded once for two.
//
// Two threads share a site: thread s takes row s of the projected half spinors in the hops (the upper row s and
// one lower row out) and chirality half s of the site term; their parts meet by shuffles after the last hop.
// Bound by the latency of its chains (a double-word multiply-add is 12 packed instructions of two cycles) at 12
// warps per SM (168 registers; one thread per site held 24 accumulators, 254 registers, 8 warps).  The call against
// one right-hand side per thread: 12 fields of 24^4 4680 -> 3000 us, two of 8^4 90 -> 62 us, of 16^4 208 -> 168 us;
// error against 64 bits 5.8e-15 both.  (The site term added straight onto -acc / 2 is quicker but errs by 7.5e-15.)
// The loop over the eight directions is rolled (one hop is about 10 KB of code) with the spin structure as
// run-time selects and sign flips on the integer pipe.  FP64 instructions issue at 1/64 of the FP32 rate,
// conversions included: y - acc / 2 is summed in FP32 words and takes one FP64 addition a number (formed in
// FP64 from its four words the call took 0.94 ms longer).
// ---------------------------------------------------------------------------
namespace {

struct dw2 {
    float2 h, l;
};
struct cdw2 {
    dw2 re, im;
};
__device__ __forceinline__ dw2 two_sum2(float2 a, float2 b) {
    const float2 s = f2add(a, b), bb = f2sub(s, a);
    return {s, f2add(f2sub(a, f2sub(s, bb)), f2sub(b, bb))};
}
__device__ __forceinline__ cdw2 cdw2_zero() {
    const float2 z = make_float2(0.f, 0.f);
    return {{z, z}, {z, z}};
}
// acc += x y for x = (xh, xl), passed as xh and its negatives nh = -xh, nl = -xl (the error terms are formed
// with the opposite sign and subtracted, which rounds the same)
__device__ __forceinline__ void dw2_mac(dw2& acc, float2 xh, float2 nh, float2 nl, const dw2& y) {
    const float2 p = f2mul(xh, y.h);
    float2 e = f2fma(nh, y.h, p);
    e = f2fma(nh, y.l, e);
    e = f2fma(nl, y.h, e);
    const dw2 s = two_sum2(acc.h, p);
    acc.h = s.h;
    acc.l = f2add(acc.l, f2sub(s.l, e));
}
__device__ __forceinline__ void dw2_macf(dw2& acc, float2 xh, float2 nh, float2 nl, float2 y) {
    const float2 p = f2mul(xh, y);
    float2 e = f2fma(nh, y, p);
    e = f2fma(nl, y, e);
    const dw2 s = two_sum2(acc.h, p);
    acc.h = s.h;
    acc.l = f2add(acc.l, f2sub(s.l, e));
}
__device__ __forceinline__ dw2 dw2_add(const dw2& a, const dw2& b) {
    const dw2 s = two_sum2(a.h, b.h);
    return {s.h, f2add(s.l, f2add(a.l, b.l))};
}
__device__ __forceinline__ dw2 dw2_norm(const dw2& a) {
    const float2 s = f2add(a.h, a.l);
    return {s, f2sub(a.l, f2sub(s, a.h))};
}
// flip the signs where m = 0x80000000
__device__ __forceinline__ float flip(float x, unsigned m) { return __uint_as_float(__float_as_uint(x) ^ m); }
__device__ __forceinline__ float2 flip2(float2 x, unsigned m) { return make_float2(flip(x.x, m), flip(x.y, m)); }
__device__ __forceinline__ float2 sel2(bool c, float2 a, float2 b) { return make_float2(c ? a.x : b.x, c ? a.y : b.y); }
__device__ __forceinline__ dw2 sel_flip(bool c, const dw2& a, const dw2& b, unsigned m) {
    return {flip2(sel2(c, a.h, b.h), m), flip2(sel2(c, a.l, b.l), m)};
}
// signs of the real and imaginary part of i^p (a + i b): (a, b), (-b, a), (-a, -b), (b, -a)
__device__ __forceinline__ unsigned sign_re(int p) { return ((p + 1) & 2) ? 0x80000000u : 0u; }
__device__ __forceinline__ unsigned sign_im(int p) { return (p & 2) ? 0x80000000u : 0u; }

}  // namespace

template <bool OUT_DW>
__global__ void __launch_bounds__(128, 3) dslash_dw_pair_kernel(Geom g, const float4* __restrict__ U, const float2* __restrict__ clov,
                                                                const cplx<float>* __restrict__ in, void* __restrict__ outp, int nrhs,
                                                                int rows) {
    const int r0 = 2 * (blockIdx.x % rows * blockDim.y + threadIdx.y);
    const int lane = threadIdx.x, s = lane >> 4, i = blockIdx.x / rows * 16 + (lane & 15);  // V is a multiple of 16
    if (r0 >= nrhs) return;  // (a whole warp)
    const bool two = r0 + 1 < nrhs;  // an odd batch computes its last right-hand side twice and stores it once
    const size_t V = g.V, o0 = (size_t)r0 * 12 * V, o1 = o0 + (two ? 12 * V : 0);
    const cplx<float>*z0 = in + o0, *z1 = in + o1;
    cdw2 up[3], same[3], oth[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) up[k] = same[k] = oth[k] = cdw2_zero();
#pragma unroll 1
    for (int d = 0; d < 8; ++d) {
        const int nb = fine_nbr(g, i, d), mu = d >> 1;
        const bool fwd = (d & 1) == 0;
        const unsigned sf = fwd ? 0x80000000u : 0u;  // h = up -+ i^p low
        // row s of B_mu reads lower row c with factor i^p; the same lower row takes i^hp of the product
        const int c = c_spinb[mu][2 * s], p = c_spinb[mu][2 * s + 1];
        const int hp = c_spinb[mu][5 + 2 * c];  // (lower row c: B_mu and B_mu^H both keep the spins or both swap them)
        const size_t ro = (size_t)(3 * s) * V + nb, rl = (size_t)(6 + 3 * c) * V + nb;
        const unsigned mr = sign_re(p) ^ sf, mi = sign_im(p) ^ sf;
        cdw2 h[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const c2 u = c2pair(z0[ro + k * V], z1[ro + k * V]), l = c2pair(z0[rl + k * V], z1[rl + k * V]);
            h[k].re = two_sum2(u.re, flip2(sel2(p & 1, l.im, l.re), mr));
            h[k].im = two_sum2(u.im, flip2(sel2(p & 1, l.re, l.im), mi));
        }
        const float4* W = U + (size_t)(mu * 9) * V + (fwd ? i : nb);
        const unsigned cj = fwd ? 0u : 0x80000000u;  // W^H backwards
        const size_t sa = (fwd ? 3 : 1) * V, sb = (fwd ? 1 : 3) * V;
        const unsigned gr = sign_re(hp) ^ sf, gi = sign_im(hp) ^ sf;
        const bool swap = mu < 2;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            cdw2 t = cdw2_zero();
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                const float4 w = __ldg(W + a * sa + b * sb);
                const float ih = flip(w.z, cj), il = flip(w.w, cj);
                const float2 rh = f2dup(w.x), nrh = f2dup(-w.x), nrl = f2dup(-w.y);
                const float2 ph = f2dup(ih), nh = f2dup(-ih), pl = f2dup(il), nl = f2dup(-il);
                dw2_mac(t.re, rh, nrh, nrl, h[b].re);
                dw2_mac(t.re, nh, ph, pl, h[b].im);
                dw2_mac(t.im, rh, nrh, nrl, h[b].im);
                dw2_mac(t.im, ph, nh, nl, h[b].re);
            }
            t.re = dw2_norm(t.re), t.im = dw2_norm(t.im);
            up[a].re = dw2_add(up[a].re, t.re), up[a].im = dw2_add(up[a].im, t.im);
            const dw2 lr = sel_flip(hp & 1, t.im, t.re, gr), li = sel_flip(hp & 1, t.re, t.im, gi);
            if (swap) oth[a].re = dw2_add(oth[a].re, lr), oth[a].im = dw2_add(oth[a].im, li);
            else same[a].re = dw2_add(same[a].re, lr), same[a].im = dw2_add(same[a].im, li);
        }
    }
    // thread s = 0 takes the upper two spin rows, thread s = 1 the lower two
    cdw2 acc[6];
    {
        auto sh = [](const dw2& v) -> dw2 {
            return {make_float2(__shfl_xor_sync(0xffffffffu, v.h.x, 16), __shfl_xor_sync(0xffffffffu, v.h.y, 16)),
                    make_float2(__shfl_xor_sync(0xffffffffu, v.l.x, 16), __shfl_xor_sync(0xffffffffu, v.l.y, 16))};
        };
        auto pick = [&](const dw2& v, const dw2& w) -> dw2 { return {sel2(s, v.h, w.h), sel2(s, v.l, w.l)}; };
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            auto part = [&](const dw2& u, const dw2& sa, const dw2& ot, dw2& lo, dw2& hi) {
                const dw2 x = sh(pick(u, sa)), z = sh(ot);  // for s = 0: x = row 1; for s = 1: parts of rows 2 and 3
                lo = pick(dw2_add(ot, x), u);
                hi = pick(dw2_add(sa, z), x);
            };
            part(up[a].re, same[a].re, oth[a].re, acc[a].re, acc[3 + a].re);
            part(up[a].im, same[a].im, oth[a].im, acc[a].im, acc[3 + a].im);
        }
    }
    // the site term of this thread's chirality half (a packed hermitian 6x6 block of double-word entries)
    c2 x[6];
    cdw2 y[6];
    const float2* base = clov + (size_t)(s * 36) * V + i;
    const size_t k0 = (size_t)(6 * s) * V + i;
#pragma unroll
    for (int a = 0; a < 6; ++a) {
        x[a] = c2pair(z0[k0 + a * V], z1[k0 + a * V]);
        const float2 e = __ldg(base + a * V);
        y[a] = cdw2_zero();
        dw2_macf(y[a].re, f2dup(e.x), f2dup(-e.x), f2dup(-e.y), x[a].re);
        dw2_macf(y[a].im, f2dup(e.x), f2dup(-e.x), f2dup(-e.y), x[a].im);
    }
    int q = 0;
#pragma unroll
    for (int a = 0; a < 6; ++a) {
#pragma unroll
        for (int b = a + 1; b < 6; ++b) {
            const float2 er = __ldg(base + (6 + 2 * q) * V), ei = __ldg(base + (7 + 2 * q) * V);
            const float2 rh = f2dup(er.x), nrh = f2dup(-er.x), nrl = f2dup(-er.y);
            const float2 ph = f2dup(ei.x), nh = f2dup(-ei.x), pl = f2dup(ei.y), nl = f2dup(-ei.y);
            // y[a] += m x[b];  y[b] += conj(m) x[a]
            dw2_macf(y[a].re, rh, nrh, nrl, x[b].re);
            dw2_macf(y[a].re, nh, ph, pl, x[b].im);
            dw2_macf(y[a].im, rh, nrh, nrl, x[b].im);
            dw2_macf(y[a].im, ph, nh, nl, x[b].re);
            dw2_macf(y[b].re, rh, nrh, nrl, x[a].re);
            dw2_macf(y[b].re, ph, nh, nl, x[a].im);
            dw2_macf(y[b].im, rh, nrh, nrl, x[a].im);
            dw2_macf(y[b].im, nh, ph, pl, x[a].re);
            ++q;
        }
    }
    const float2 mh = f2dup(-0.5f);
    // y - acc / 2: the sum of the high words and its exact error, with the low words added to that error by
    // error-free sums, so that only the last word is rounded
    auto sub = [&](const dw2& u, const dw2& v) -> dw2 {
        const dw2 p = two_sum2(u.h, f2mul(mh, v.h)), q = two_sum2(u.l, f2mul(mh, v.l)), t = two_sum2(p.l, q.h);
        const float2 m = f2add(t.h, f2add(t.l, q.l)), h = f2add(p.h, m);
        return {h, f2add(f2sub(m, f2sub(h, p.h)), f2add(f2sub(t.h, m), f2add(t.l, q.l)))};
    };
#pragma unroll
    for (int a = 0; a < 6; ++a) {
        const dw2 re = sub(y[a].re, acc[a].re), im = sub(y[a].im, acc[a].im);
        const size_t k = k0 + a * V;
        if (OUT_DW) {
            float4* o = reinterpret_cast<float4*>(outp);
            o[o0 + k] = make_float4(re.h.x, re.l.x, im.h.x, im.l.x);
            if (two) o[o1 + k] = make_float4(re.h.y, re.l.y, im.h.y, im.l.y);
        } else {
            cplx<double>* o = reinterpret_cast<cplx<double>*>(outp);
            o[o0 + k] = mk((double)re.h.x + (double)re.l.x, (double)im.h.x + (double)im.l.x);
            if (two) o[o1 + k] = mk((double)re.h.y + (double)re.l.y, (double)im.h.y + (double)im.l.y);
        }
    }
}

int launch_dslash_dw(const Geom& g, const float4* U, const float2* clov, const cplx<float>* in, void* out, bool out_dw, int nrhs,
                     cudaStream_t st) {
    if (nrhs >= 2) {
        // pairs dealt out evenly to CTAs of up to four, the CTAs of the same sites one after another: six pairs as
        // 4 + 2 in separate grid rows left half of the second row's warps idle and read the operator twice
        // (12 fields of 24^4, the call: 3270 -> 3000 us; DRAM reads of the kernel 1.97 GB with the rows apart, 0.76 GB needed)
        const int pairs = (nrhs + 1) / 2, rows = ceil_div(pairs, 4), ry = ceil_div(pairs, rows);
        const dim3 grid((unsigned)(g.V / 16) * (unsigned)rows), block(32, ry);
        if (out_dw) dslash_dw_pair_kernel<true><<<grid, block, 0, st>>>(g, U, clov, in, out, nrhs, rows);
        else dslash_dw_pair_kernel<false><<<grid, block, 0, st>>>(g, U, clov, in, out, nrhs, rows);
        DD_CHECK_LAUNCH();
        return 0;
    }
    const unsigned grid = (unsigned)ceil_div(g.V, 32);
    if (out_dw) dslash_dw_kernel<true><<<grid, 32, 0, st>>>(g, U, clov, in, out);
    else dslash_dw_kernel<false><<<grid, 32, 0, st>>>(g, U, clov, in, out);
    DD_CHECK_LAUNCH();
    return 0;
}

}  // namespace ddamg
