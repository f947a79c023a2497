// FP32 Dslash on 4^4 blocks for two or more right-hand sides.
//
// Bound by the latency of the neighbours' spinors.  A CTA of 128 threads covers half a block (64 sites of
// either parity) and one pair of right-hand sides: 128 registers leave 16 warps on an SM, and most in-block
// neighbours are sites of the same CTA, so their spinors hit L1.  The call against one right-hand side per thread
// (24 warps, 80 registers): 12 fields of 32^4 3669 -> 1785 us, two fields of 8^4 (32 CTAs) 53 -> 43 us, of 16^4 79 ->
// 55 us, three of 24x16^3 122 -> 87 us.
#include <type_traits>

#include "ops44.cuh"

namespace ddamg {

// out = D in (RESID: out = b - D in).  One thread per site, two right-hand sides in packed FP32
// instructions.  The pairs of right-hand sides of a half block follow one another, so the links and site
// terms come from L2 after the first; the CTAs walk the blocks in lexicographic order, red and black
// interleaved, so that a block and its neighbours in three of the four directions are read close
// together in time and the neighbours' spinors are still in L2.
// lex != null: out is in the caller's layout ([field][site lex[i]][12], 16-byte aligned): a site's
// components leave as whole 16-byte words, and no separate pass has to reorder the field.
template <bool RESID>
__global__ void __launch_bounds__(128, 4)
    dslash44_pair_kernel(Geom g, FineOpB op, const cplx<float>* __restrict__ in, const cplx<float>* __restrict__ b, cplx<float>* __restrict__ out,
                         const int* __restrict__ lex, int nrhs) {
    const unsigned pairs = (unsigned)(nrhs + 1) / 2, sub = blockIdx.x / pairs;
    const int r0 = 2 * (int)(blockIdx.x % pairs);
    const bool two = r0 + 1 < nrhs;  // an odd batch computes its last right-hand side twice and stores it once
    const int c = __ldg(g.blex + (sub >> 1));
    const int l = (threadIdx.x >> 6) * 128 + (sub & 1) * 64 + (threadIdx.x & 63), i = c * 256 + l, V = g.V;
    const int L = lex44_of_local(l), p = l >> 7;
    int bn[8];
#pragma unroll
    for (int d = 0; d < 8; ++d) bn[d] = __ldg(g.bnbr + d * g.NB + c);
    const size_t o0 = (size_t)r0 * 12 * V, o1 = o0 + (two ? (size_t)12 * V : 0);
    const cplx<float>*z0 = in + o0, *z1 = in + o1;
    c2 acc[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) acc[k] = c2zero();
    hop_pair44_global<0>(op.U, z0, z1, V, L, p, c, bn[0], bn[1], acc);
    hop_pair44_global<1>(op.U, z0, z1, V, L, p, c, bn[2], bn[3], acc);
    hop_pair44_global<2>(op.U, z0, z1, V, L, p, c, bn[4], bn[5], acc);
    hop_pair44_global<3>(op.U, z0, z1, V, L, p, c, bn[6], bn[7], acc);
    auto half = [&](auto hb) {
        constexpr int HB = decltype(hb)::value;
        c2 x[6], y[6];
#pragma unroll
        for (int a = 0; a < 6; ++a) x[a] = c2pair(z0[(size_t)(HB * 6 + a) * V + i], z1[(size_t)(HB * 6 + a) * V + i]);
        herm44<HB>(op.clov, c, l, x, y);
#pragma unroll
        for (int a = 0; a < 6; ++a) {
            const size_t o = (size_t)(HB * 6 + a) * V + i;
            y[a] = c2axpy(y[a], -0.5f, acc[HB * 6 + a]);
            if (RESID) y[a] = c2pair(b[o0 + o], b[o1 + o]) - y[a];
        }
        if (lex) {
            const size_t s = (size_t)__ldg(lex + i) * 12 + HB * 6;
            float4 *u = reinterpret_cast<float4*>(out + o0 + s), *v = reinterpret_cast<float4*>(out + o1 + s);
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                u[a] = make_float4(y[2 * a].re.x, y[2 * a].im.x, y[2 * a + 1].re.x, y[2 * a + 1].im.x);
                if (two) v[a] = make_float4(y[2 * a].re.y, y[2 * a].im.y, y[2 * a + 1].re.y, y[2 * a + 1].im.y);
            }
        } else {
#pragma unroll
            for (int a = 0; a < 6; ++a) {
                const size_t o = (size_t)(HB * 6 + a) * V + i;
                out[o0 + o] = mk(y[a].re.x, y[a].im.x);
                if (two) out[o1 + o] = mk(y[a].re.y, y[a].im.y);
            }
        }
    };
    half(std::integral_constant<int, 0>());
    half(std::integral_constant<int, 1>());
}

int launch_dslash44_pair(const Geom& g, const FineOpB& op, const cplx<float>* in, const cplx<float>* b, cplx<float>* out, const int* lex,
                         int nrhs, cudaStream_t st) {
    const unsigned grid = 2u * (unsigned)g.NB * (unsigned)((nrhs + 1) / 2), block = 128;
    if (b)
        dslash44_pair_kernel<true><<<grid, block, 0, st>>>(g, op, in, b, out, lex, nrhs);
    else
        dslash44_pair_kernel<false><<<grid, block, 0, st>>>(g, op, in, b, out, lex, nrhs);
    DD_CHECK_LAUNCH();
    return 0;
}

}  // namespace ddamg
