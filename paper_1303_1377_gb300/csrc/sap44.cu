// Red-black SAP block solver (Sec. 2.3, local odd-even MR of Sec. 6) on 4^4 blocks in FP32 arithmetic.
//
// A CTA of 128 threads owns one block of the colour and two right-hand sides; each thread owns one even
// and one odd site and computes both right-hand sides in packed FP32 instructions (f32x2.cuh), so a link
// or site-term entry is loaded and converted once for two right-hand sides and a multiply-add issues
// once for two.  x_o stays in registers (255 a thread, two CTAs per SM); the even work vector and rho
// take 49 KB of shared memory, which leaves the rest of the SM's 256 KB to L1 for the links and site
// terms that every MR step reads again.
//
// What bounds it: the packed multiply-adds (two cycles each) hold the FMA pipe about 60% busy in the MR
// steps; the residual at the start waits on its neighbours' spinors.  12 fields on 24^4, one colour: 740 us
// (29 TFLOP/s) with either operator; one right-hand side per thread, four per CTA (512 threads, 128 registers), took
// 1347 us (FP16) and 1399 us (FP32).  One field, or few blocks: sap44_one_kernel, by the rule in launch_sap44.
#include <type_traits>

#include "ops44.cuh"

namespace ddamg {

// ---- hops
// in-block hops in direction MU of local site (lexicographic index L, local index l) of block c; sm
// holds the field on the other parity (rank order), nb0 = local index of rank 0 of that parity.  A
// neighbour outside the block is replaced by the one on the other side with a zero link: a quarter of
// the lanes would idle in a branch anyway, and without branches the loads of the next hops are issued
// while the current one computes (one MR step of 12 fields on 24^4: 121 us with branches, 96 us without).
template <int MU, typename UT>
__device__ __forceinline__ void hop_pair44(const UT& U, const float4* sm, int L, int nb0, int c, int l, c2 (&acc)[12]) {
    constexpr int SH = 2 * (3 - MU), S = 1 << SH;
    const int y = (L >> SH) & 3;
    const bool f = y < 3, b = y > 0;
    const int nf = (f ? L + S : L - S) >> 1, nb = (b ? L - S : L + S) >> 1;
    cplx<float> Wf[9], Wb[9];
    load_link44(Wf, U, c, MU, l, f);
    load_link44(Wb, U, c, MU, nb0 + nb, b);
    hop_acc2<MU, true>(acc, [&](int k) { return c2_of(sm[k * 128 + nf]); }, Wf);
    hop_acc2<MU, false>(acc, [&](int k) { return c2_of(sm[k * 128 + nb]); }, Wb);
}
template <typename UT>
__device__ __forceinline__ void hops44(const UT& U, const float4* sm, int L, int nb0, int c, int l, c2 (&acc)[12]) {
#pragma unroll
    for (int k = 0; k < 12; ++k) acc[k] = c2zero();
    hop_pair44<0>(U, sm, L, nb0, c, l, acc);
    hop_pair44<1>(U, sm, L, nb0, c, l, acc);
    hop_pair44<2>(U, sm, L, nb0, c, l, acc);
    hop_pair44<3>(U, sm, L, nb0, c, l, acc);
}
template <typename OpT>
__global__ void __launch_bounds__(128, 2)
    sap44_kernel(Geom g, OpT op, const cplx<float>* __restrict__ bsrc, cplx<float>* z, int colour, int nrhs, int mr_steps, int npairs) {
    constexpr int H = 128;
    extern __shared__ float4 smem44[];
    const int t = threadIdx.x, r0 = 2 * (blockIdx.x % npairs);
    const bool two = r0 + 1 < nrhs;  // an odd batch computes its last right-hand side twice and stores it once
    float4* SE = smem44;                                         // [12][H] even work vector
    float4* SO = SE + 12 * H;                                    // [12][H] r_o, then rho, then x_o
    float2* red = reinterpret_cast<float2*>(smem44 + 24 * H);    // [4 warps][3]
    const int V = g.V, c = colour * (g.NB / 2) + blockIdx.x / npairs;
    const cplx<float>* b0 = bsrc + (size_t)r0 * 12 * V;
    const cplx<float>* b1 = b0 + (two ? (size_t)12 * V : 0);
    cplx<float>* z0 = z + (size_t)r0 * 12 * V;
    cplx<float>* z1 = z0 + (two ? (size_t)12 * V : 0);
    const int ie = c * 256 + t, io = ie + H;
    // z += d at component k0 .. k0 + n - 1 of site i: all loads before the first store (a store ends
    // what the compiler can prove about the other components, so a plain loop waits for each load)
    auto add_z = [&](int k0, int i, const c2* d, auto n) {
        constexpr int N = decltype(n)::value;
        cplx<float> u[N], v[N];
#pragma unroll
        for (int a = 0; a < N; ++a) u[a] = z0[(size_t)(k0 + a) * V + i], v[a] = z1[(size_t)(k0 + a) * V + i];
#pragma unroll
        for (int a = 0; a < N; ++a) {
            z0[(size_t)(k0 + a) * V + i] = u[a] + mk(d[a].re.x, d[a].im.x);
            if (two) z1[(size_t)(k0 + a) * V + i] = v[a] + mk(d[a].re.y, d[a].im.y);
        }
    };
    using I6 = std::integral_constant<int, 6>;
    using I12 = std::integral_constant<int, 12>;
    // residual r = b - D z; even sites: SE = A_ee^{-1} r_e, odd sites: SO = r_o
#pragma unroll 1
    for (int p = 0; p < 2; ++p) {
        const int l = p * H + t, i = c * 256 + l, L = lex44_of_local(l);
        int bn[8];
#pragma unroll
        for (int d = 0; d < 8; ++d) bn[d] = __ldg(g.bnbr + d * g.NB + c);
        c2 acc[12];
#pragma unroll
        for (int k = 0; k < 12; ++k) acc[k] = c2zero();
        hop_pair44_global<0>(op.U, z0, z1, V, L, p, c, bn[0], bn[1], acc);
        hop_pair44_global<1>(op.U, z0, z1, V, L, p, c, bn[2], bn[3], acc);
        hop_pair44_global<2>(op.U, z0, z1, V, L, p, c, bn[4], bn[5], acc);
        hop_pair44_global<3>(op.U, z0, z1, V, L, p, c, bn[6], bn[7], acc);
        c2 x[6], y[6];
        auto half = [&](auto hb) {
            constexpr int HB = decltype(hb)::value;
#pragma unroll
            for (int a = 0; a < 6; ++a) x[a] = c2pair(z0[(size_t)(HB * 6 + a) * V + i], z1[(size_t)(HB * 6 + a) * V + i]);
            herm44<HB>(op.clov, c, l, x, y);
#pragma unroll
            for (int a = 0; a < 6; ++a) {
                const size_t o = (size_t)(HB * 6 + a) * V + i;
                x[a] = c2pair(b0[o], b1[o]) - c2axpy(y[a], -0.5f, acc[HB * 6 + a]);
            }
            if (p == 0) {
                herm44<HB>(op.clovinv, c, l, x, y);
#pragma unroll
                for (int a = 0; a < 6; ++a) SE[(HB * 6 + a) * H + t] = c2_f4(y[a]);
            } else {
#pragma unroll
                for (int a = 0; a < 6; ++a) SO[(HB * 6 + a) * H + t] = c2_f4(x[a]);
            }
        };
        half(std::integral_constant<int, 0>());
        half(std::integral_constant<int, 1>());
    }
    __syncthreads();  // every read of z in this block is done: z may be updated from here on
    c2 xo[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) xo[k] = c2_of(SE[k * H + t]);
    add_z(0, ie, xo, I12());  // the part A_ee^{-1} r_e of x_e, which does not depend on x_o
#pragma unroll
    for (int k = 0; k < 12; ++k) xo[k] = c2zero();
    const int Le = lex44_of_local(t), Lo = lex44_of_local(H + t);
    // pass 0 forms rho = r_o - D_oe A_ee^{-1} r_e; passes 1 .. mr_steps are the MR steps on
    // S = A_oo - D_oe A_ee^{-1} D_eo; the even half of the last pass is the back-substitution
#pragma unroll 1
    for (int it = 0; it <= mr_steps; ++it) {
        {
            c2 sr[12];
            hops44(op.U, SE, Lo, 0, c, H + t, sr);
            if (it == 0) {
#pragma unroll
                for (int k = 0; k < 12; ++k) SO[k * H + t] = c2_f4(c2axpy(c2_of(SO[k * H + t]), 0.5f, sr[k]));
            } else {
                float2 nr = make_float2(0.f, 0.f), ni = nr, dd = nr;
                auto half = [&](auto hb) {
                    constexpr int HB = decltype(hb)::value;
                    c2 rho[6], y[6];
#pragma unroll
                    for (int a = 0; a < 6; ++a) rho[a] = c2_of(SO[(HB * 6 + a) * H + t]);
                    herm44<HB>(op.clov, c, H + t, rho, y);
#pragma unroll
                    for (int a = 0; a < 6; ++a) {
                        const c2 s = c2axpy(y[a], 0.5f, sr[HB * 6 + a]);
                        sr[HB * 6 + a] = s;
                        nr = f2fma(s.re, rho[a].re, nr), nr = f2fma(s.im, rho[a].im, nr);
                        ni = f2fma(s.re, rho[a].im, ni), ni = f2fma(f2neg(s.im), rho[a].re, ni);
                        dd = f2fma(s.re, s.re, dd), dd = f2fma(s.im, s.im, dd);
                    }
                };
                half(std::integral_constant<int, 0>());
                half(std::integral_constant<int, 1>());
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    nr.x += __shfl_xor_sync(0xffffffffu, nr.x, o), nr.y += __shfl_xor_sync(0xffffffffu, nr.y, o);
                    ni.x += __shfl_xor_sync(0xffffffffu, ni.x, o), ni.y += __shfl_xor_sync(0xffffffffu, ni.y, o);
                    dd.x += __shfl_xor_sync(0xffffffffu, dd.x, o), dd.y += __shfl_xor_sync(0xffffffffu, dd.y, o);
                }
                if ((t & 31) == 0) red[3 * (t >> 5)] = nr, red[3 * (t >> 5) + 1] = ni, red[3 * (t >> 5) + 2] = dd;
                __syncthreads();
                nr = f2add(f2add(red[0], red[3]), f2add(red[6], red[9]));
                ni = f2add(f2add(red[1], red[4]), f2add(red[7], red[10]));
                dd = f2add(f2add(red[2], red[5]), f2add(red[8], red[11]));
                const bool ok0 = dd.x > tiny_normal<float>(), ok1 = dd.y > tiny_normal<float>();
                const float2 ar = make_float2(ok0 ? nr.x / dd.x : 0.f, ok1 ? nr.y / dd.y : 0.f);
                const float2 ai = make_float2(ok0 ? ni.x / dd.x : 0.f, ok1 ? ni.y / dd.y : 0.f);
                const float2 mr = f2neg(ar), mi = f2neg(ai);
                const bool last = it == mr_steps;
#pragma unroll
                for (int k = 0; k < 12; ++k) {  // x_o += alpha rho, rho -= alpha S rho
                    const c2 rho = c2_of(SO[k * H + t]);
                    xo[k].re = f2fma(mi, rho.im, f2fma(ar, rho.re, xo[k].re));
                    xo[k].im = f2fma(ai, rho.re, f2fma(ar, rho.im, xo[k].im));
                    c2 nw;
                    nw.re = f2fma(ai, sr[k].im, f2fma(mr, sr[k].re, rho.re));
                    nw.im = f2fma(mi, sr[k].re, f2fma(mr, sr[k].im, rho.im));
                    if (!last) SO[k * H + t] = c2_f4(nw);
                }
            }
            if (it == mr_steps) {
#pragma unroll
                for (int k = 0; k < 12; ++k) SO[k * H + t] = c2_f4(xo[k]);
            }
        }
        __syncthreads();
        {
            c2 hs[12];
            hops44(op.U, SO, Le, H, c, t, hs);
            const bool last = it == mr_steps;
            auto half = [&](auto hb) {
                constexpr int HB = decltype(hb)::value;
                c2 x[6], y[6];
#pragma unroll
                for (int a = 0; a < 6; ++a) x[a] = c2scale(last ? 0.5f : -0.5f, hs[HB * 6 + a]);
                herm44<HB>(op.clovinv, c, t, x, y);
                if (last) add_z(HB * 6, ie, y, I6());
                else {
#pragma unroll
                    for (int a = 0; a < 6; ++a) SE[(HB * 6 + a) * H + t] = c2_f4(y[a]);
                }
            };
            half(std::integral_constant<int, 0>());
            half(std::integral_constant<int, 1>());
        }
        __syncthreads();
    }
    add_z(0, io, xo, I12());
}

// ---------------------------------------------------------------------------
// One right-hand side per CTA (grid.y = right-hand sides): one field has no second one to pack, and with few
// blocks a CTA of 128 threads leaves an SM one warp per scheduler; so two threads share a site pair: thread s takes
// spin s of the projected half spinors in the hops (psi_s and one lower row in, the upper row s and one
// lower row out) and chirality half s in the site terms, and the two exchange their parts after the hops
// by shuffles (lanes l and l ^ 16).  One field, one colour, against sap44_kernel with an idle second field: 16^4
// FP16 operator 45 -> 27 us, FP32 operator 45 -> 31 us; 24^4 151 -> 103 and 159 -> 127 us.
// ---------------------------------------------------------------------------
template <int P>
__device__ __forceinline__ cplx<float> c_fma_ipow(cplx<float> a, cplx<float> b, float g) {  // a + g i^P b
    const cplx<float> w = ipow<(P & 3)>(b);
    return mk(fmaf(g, w.re, a.re), fmaf(g, w.im, a.im));
}
struct SpinAcc {  // upper row s; lower row s (mu = 2, 3) and lower row 1 - s (mu = 0, 1)
    cplx<float> up[3], same[3], oth[3];
};
// the two threads' factors i^p differ by a sign for mu = 1, 2: sg = +1 for s = 0, -1 for s = 1
template <int MU, bool FWD, typename PU, typename PL>
__device__ __forceinline__ void hop_spin(SpinAcc& acc, const PU& up, const PL& low, const cplx<float> (&W)[9], float sg) {
    using B = SpinB<MU>;
    constexpr int S = FWD ? 2 : 0;  // h = up -+ i^p low
    const float f = (MU == 1 || MU == 2) ? sg : 1.f;
    cplx<float> h[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) h[c] = c_fma_ipow<B::p0 + S>(up(c), low(c), f);
    cplx<float>(&lo)[3] = MU < 2 ? acc.oth : acc.same;
    constexpr int HP = (MU < 2 ? B::hp1 : B::hp0) + S;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        cplx<float> g = czero<float>();
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            if (FWD) cmac(g, W[a * 3 + b], h[b]);
            else cmac_conj(g, W[b * 3 + a], h[b]);
        }
        acc.up[a] = acc.up[a] + g;
        lo[a] = c_fma_ipow<HP>(lo[a], g, f);
    }
}
__device__ __forceinline__ cplx<float> shfl16(cplx<float> a) {
    return mk(__shfl_xor_sync(0xffffffffu, a.re, 16), __shfl_xor_sync(0xffffffffu, a.im, 16));
}
// thread s = 0 gets the upper two spin rows, thread s = 1 the lower two
__device__ __forceinline__ void spin_exchange(const SpinAcc& acc, int s, cplx<float> (&out)[6]) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const cplx<float> x = shfl16(s ? acc.up[a] : acc.same[a]);  // s = 0 receives row 1, s = 1 a part of row 2
        const cplx<float> y = shfl16(acc.oth[a]);                   // s = 1 receives a part of row 3
        out[a] = s ? acc.oth[a] + x : acc.up[a];
        out[3 + a] = s ? acc.same[a] + y : x;
    }
}
__device__ __forceinline__ void spin_zero(SpinAcc& acc) {
#pragma unroll
    for (int k = 0; k < 3; ++k) acc.up[k] = acc.same[k] = acc.oth[k] = czero<float>();
}
// y = (block s of the site term) x
template <typename CF>
__device__ __forceinline__ void herm6_apply(const CF& cf, const cplx<float> (&x)[6], cplx<float> (&y)[6]) {
#pragma unroll
    for (int a = 0; a < 6; ++a) y[a] = cf(a) * x[a];
    int m = 0;
#pragma unroll
    for (int a = 0; a < 6; ++a)
#pragma unroll
        for (int b = a + 1; b < 6; ++b) {
            const cplx<float> e = mk(cf(6 + 2 * m), cf(7 + 2 * m));
            cmac(y[a], e, x[b]);
            cmac_conj(y[b], e, x[a]);
            ++m;
        }
}
__device__ __forceinline__ void herm44_one(const CloverB& cl, int c, int l, int s, const cplx<float> (&x)[6], cplx<float> (&y)[6]) {
    const float4* q = cl.p + (size_t)c * (18 * 256) + s * (9 * 256) + l;
    float w[36];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const float4 v = __ldg(q + k * 256);
        w[4 * k] = v.x, w[4 * k + 1] = v.y, w[4 * k + 2] = v.z, w[4 * k + 3] = v.w;
    }
    herm6_apply([&](int j) { return w[j]; }, x, y);
}
__device__ __forceinline__ void herm44_one(const CloverB16& cl, int c, int l, int s, const cplx<float> (&x)[6], cplx<float> (&y)[6]) {
    const uint4* q = cl.p + (size_t)c * (10 * 256) + s * (5 * 256) + l;
    unsigned w[20];
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        const uint4 v = __ldg(q + k * 256);
        w[4 * k] = v.x, w[4 * k + 1] = v.y, w[4 * k + 2] = v.z, w[4 * k + 3] = v.w;
    }
    herm6_apply(
        [&](int j) {
            const float2 f = h2f(w[j / 2]);
            return (j & 1) ? f.y : f.x;
        },
        x, y);
}
// in-block hops (as hop_pair44: a neighbour outside the block is replaced, with a zero link)
template <int MU, typename UT>
__device__ __forceinline__ void hop_pair_one(const UT& U, const cplx<float>* sm, int L, int nb0, int c, int l, int s, float sg, SpinAcc& acc) {
    constexpr int SH = 2 * (3 - MU), S = 1 << SH;
    const int y = (L >> SH) & 3;
    const bool f = y < 3, b = y > 0;
    const int nf = (f ? L + S : L - S) >> 1, nb = (b ? L - S : L + S) >> 1;
    const cplx<float>*up = sm + s * (3 * 128), *low = sm + (6 + 3 * (MU < 2 ? 1 - s : s)) * 128;
    cplx<float> Wf[9], Wb[9];
    load_link44(Wf, U, c, MU, l, f);
    load_link44(Wb, U, c, MU, nb0 + nb, b);
    hop_spin<MU, true>(acc, [&](int k) { return up[k * 128 + nf]; }, [&](int k) { return low[k * 128 + nf]; }, Wf, sg);
    hop_spin<MU, false>(acc, [&](int k) { return up[k * 128 + nb]; }, [&](int k) { return low[k * 128 + nb]; }, Wb, sg);
}
template <typename UT>
__device__ __forceinline__ void hops_one(const UT& U, const cplx<float>* sm, int L, int nb0, int c, int l, int s, float sg, cplx<float> (&out)[6]) {
    SpinAcc acc;
    spin_zero(acc);
    hop_pair_one<0>(U, sm, L, nb0, c, l, s, sg, acc);
    hop_pair_one<1>(U, sm, L, nb0, c, l, s, sg, acc);
    hop_pair_one<2>(U, sm, L, nb0, c, l, s, sg, acc);
    hop_pair_one<3>(U, sm, L, nb0, c, l, s, sg, acc);
    spin_exchange(acc, s, out);
}
template <int MU, typename UT>
__device__ __forceinline__ void hop_pair_one_global(const UT& U, const cplx<float>* z, size_t V, int L, int p, int c, int bf, int bb, int s, float sg,
                                                    SpinAcc& acc) {
    const cplx<float>*up = z + (size_t)(3 * s) * V, *low = z + (size_t)(6 + 3 * (MU < 2 ? 1 - s : s)) * V;
    const int f = nbr44<MU, true>(L, p, c, bf), b = nbr44<MU, false>(L, p, c, bb);
    cplx<float> Wf[9], Wb[9];
    load_link44(Wf, U, c, MU, (p << 7) | (L >> 1));
    load_link44(Wb, U, b >> 8, MU, b & 255);
    hop_spin<MU, true>(acc, [&](int k) { return up[k * V + f]; }, [&](int k) { return low[k * V + f]; }, Wf, sg);
    hop_spin<MU, false>(acc, [&](int k) { return up[k * V + b]; }, [&](int k) { return low[k * V + b]; }, Wb, sg);
}

template <typename OpT>
__global__ void __launch_bounds__(256, 2)
    sap44_one_kernel(Geom g, OpT op, const cplx<float>* __restrict__ bsrc, cplx<float>* zsrc, int colour, int mr_steps) {
    constexpr int H = 128;
    __shared__ cplx<float> SE[12 * H], SO[12 * H];  // even work vector; r_o, then rho, then x_o
    __shared__ float red[8][3];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, t = w * 16 + (lane & 15), s = lane >> 4;
    const float sg = s ? -1.f : 1.f;
    const size_t V = g.V, k0 = 6 * s;  // this thread's components 6 s .. 6 s + 5 of its two sites
    const cplx<float>* b = bsrc + (size_t)blockIdx.y * 12 * V;
    cplx<float>* z = zsrc + (size_t)blockIdx.y * 12 * V;
    const int c = colour * (g.NB / 2) + blockIdx.x, ie = c * 256 + t, io = ie + H;
    cplx<float>*me = SE + k0 * H + t, *mo = SO + k0 * H + t;
    auto add_z = [&](int i, const cplx<float> (&d)[6]) {  // all loads before the first store, as in sap44_kernel
        cplx<float> u[6];
#pragma unroll
        for (int a = 0; a < 6; ++a) u[a] = z[(k0 + a) * V + i];
#pragma unroll
        for (int a = 0; a < 6; ++a) z[(k0 + a) * V + i] = u[a] + d[a];
    };
    // residual r = b - D z; even sites: SE = A_ee^{-1} r_e, odd sites: SO = r_o
#pragma unroll 1
    for (int p = 0; p < 2; ++p) {
        const int l = p * H + t, i = c * 256 + l, L = lex44_of_local(l);
        int bn[8];
#pragma unroll
        for (int d = 0; d < 8; ++d) bn[d] = __ldg(g.bnbr + d * g.NB + c);
        SpinAcc acc;
        spin_zero(acc);
        hop_pair_one_global<0>(op.U, z, V, L, p, c, bn[0], bn[1], s, sg, acc);
        hop_pair_one_global<1>(op.U, z, V, L, p, c, bn[2], bn[3], s, sg, acc);
        hop_pair_one_global<2>(op.U, z, V, L, p, c, bn[4], bn[5], s, sg, acc);
        hop_pair_one_global<3>(op.U, z, V, L, p, c, bn[6], bn[7], s, sg, acc);
        cplx<float> hs[6], x[6], y[6];
        spin_exchange(acc, s, hs);
#pragma unroll
        for (int a = 0; a < 6; ++a) x[a] = z[(k0 + a) * V + i];
        herm44_one(op.clov, c, l, s, x, y);
#pragma unroll
        for (int a = 0; a < 6; ++a) x[a] = b[(k0 + a) * V + i] - (y[a] - 0.5f * hs[a]);
        if (p == 0) {
            herm44_one(op.clovinv, c, l, s, x, y);
#pragma unroll
            for (int a = 0; a < 6; ++a) me[a * H] = y[a];
        } else {
#pragma unroll
            for (int a = 0; a < 6; ++a) mo[a * H] = x[a];
        }
    }
    __syncthreads();  // every read of z in this block is done: z may be updated from here on
    cplx<float> xo[6];
#pragma unroll
    for (int a = 0; a < 6; ++a) xo[a] = me[a * H];
    add_z(ie, xo);  // the part A_ee^{-1} r_e of x_e, which does not depend on x_o
#pragma unroll
    for (int a = 0; a < 6; ++a) xo[a] = czero<float>();
    const int Le = lex44_of_local(t), Lo = lex44_of_local(H + t);
    // the passes of sap44_kernel
#pragma unroll 1
    for (int it = 0; it <= mr_steps; ++it) {
        const bool last = it == mr_steps;
        {
            cplx<float> sr[6];
            hops_one(op.U, SE, Lo, 0, c, H + t, s, sg, sr);
            if (it == 0) {
#pragma unroll
                for (int a = 0; a < 6; ++a) mo[a * H] = mo[a * H] + 0.5f * sr[a];
            } else {
                cplx<float> rho[6], y[6];
                float nr = 0.f, ni = 0.f, dd = 0.f;
#pragma unroll
                for (int a = 0; a < 6; ++a) rho[a] = mo[a * H];
                herm44_one(op.clov, c, H + t, s, rho, y);
#pragma unroll
                for (int a = 0; a < 6; ++a) {
                    const cplx<float> v = y[a] + 0.5f * sr[a];
                    sr[a] = v;
                    nr += v.re * rho[a].re + v.im * rho[a].im;
                    ni += v.re * rho[a].im - v.im * rho[a].re;
                    dd += norm2(v);
                }
                nr = warp_sum(nr), ni = warp_sum(ni), dd = warp_sum(dd);
                if (lane == 0) red[w][0] = nr, red[w][1] = ni, red[w][2] = dd;
                __syncthreads();
                nr = ni = dd = 0.f;
#pragma unroll
                for (int q = 0; q < 8; ++q) nr += red[q][0], ni += red[q][1], dd += red[q][2];
                const cplx<float> alpha = dd > tiny_normal<float>() ? mk(nr / dd, ni / dd) : czero<float>();
#pragma unroll
                for (int a = 0; a < 6; ++a) {  // x_o += alpha rho, rho -= alpha S rho
                    cmac(xo[a], alpha, rho[a]);
                    if (!last) mo[a * H] = rho[a] - alpha * sr[a];
                }
            }
            if (last) {
#pragma unroll
                for (int a = 0; a < 6; ++a) mo[a * H] = xo[a];
            }
        }
        __syncthreads();
        {
            cplx<float> x[6], y[6];
            hops_one(op.U, SO, Le, H, c, t, s, sg, x);
#pragma unroll
            for (int a = 0; a < 6; ++a) x[a] = (last ? 0.5f : -0.5f) * x[a];
            herm44_one(op.clovinv, c, t, s, x, y);
            if (last) add_z(ie, y);
            else {
#pragma unroll
                for (int a = 0; a < 6; ++a) me[a * H] = y[a];
            }
        }
        __syncthreads();
    }
    add_z(io, xo);
}

template <typename OpT>
int launch_sap44(const Geom& g, const OpT& op, const cplx<float>* b, cplx<float>* z, int colour, int nrhs, int mr_steps, cudaStream_t st) {
    // Few blocks: one CTA per block and field while they all fit on the chip, one per SM (FP32 operator) or two (FP16,
    // half the L1 footprint).  us per colour, one field per CTA / pairs: 8^4 (8 blocks) 12 fields 27 / 39 (FP16), 31 / 41
    // (FP32); 16x8^3 12 fields (192 CTAs) 41 / 45, 45 / 44; 16^4 two fields (256 CTAs) 42 / 48, 47 / 48; three 61 / 62,
    // 72 / 63; 24^4 two 177 / 159.
    const long long slots = std::is_same<OpT, FineOpB16>::value ? 2 * 152 : 152;
    if (nrhs == 1 || (long long)(g.NB / 2) * nrhs <= slots) {
        sap44_one_kernel<OpT><<<dim3((unsigned)(g.NB / 2), (unsigned)nrhs), 256, 0, st>>>(g, op, b, z, colour, mr_steps);
        DD_CHECK_LAUNCH();
        return 0;
    }
    const size_t smem = 24 * 128 * sizeof(float4) + 12 * sizeof(float2);
    DD_CUDA(allow_smem<sap44_kernel<OpT>>(100 * 1024));
    const int npairs = (nrhs + 1) / 2;
    sap44_kernel<OpT><<<(unsigned)(g.NB / 2) * (unsigned)npairs, 128, smem, st>>>(g, op, b, z, colour, nrhs, mr_steps, npairs);
    DD_CHECK_LAUNCH();
    return 0;
}
template int launch_sap44(const Geom&, const FineOpB&, const cplx<float>*, cplx<float>*, int, int, int, cudaStream_t);
template int launch_sap44(const Geom&, const FineOpB16&, const cplx<float>*, cplx<float>*, int, int, int, cudaStream_t);

}  // namespace ddamg
