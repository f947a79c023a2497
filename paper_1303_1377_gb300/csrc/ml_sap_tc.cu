// Level-k SAP colour step of half-precision handles on tensor cores (the algorithm of ml_sap.cu: residual,
// odd-even MR on the block, back-substitution), for the FP16 copies of D_k and D_ee^{-1}.
//
// The unit of work is one warp per (even/odd site pair of the block, four right-hand sides).  A product
// B x of an nc x nc block with the four right-hand sides is a real product [Re B; Im B] (2 nc rows) times
// [Re x_r, Im x_r interleaved] (8 columns): U = nc / 8 m-tiles of mma.sync with K = nc.  The vector enters
// as two FP16 numbers, hi + 2^-11 lo, so that the product is the FP16-stored matrix times x to about 2^-22.
// The tensor cores' FP32 accumulation truncates, so every product starts from zero and is added to the running
// sum in FP32 registers: with the accumulators kept over the nine products of a row the error grew to 1.35 times
// that of FP32 vectors on the CUDA cores (8.9e-7 against 6.6e-7 rms at nc = 40; now 1.4e-7).  A lane ends with the complex rows 8 q + g of one right-hand side, so rho, x_o
// and the MR updates stay in registers; only the staged (hi, lo) vectors of the block's sites, 1.3 KB a
// site and group at nc = 40, go through shared memory.
//
// The step is linear in (b, z), and FP16 covers 2^-36 (the low part's last bit) to 2^16 only, so every vector is
// multiplied by a power of two before it is split and the product divided by it: z by one per site read and
// right-hand side; everything after the residual by one per block and right-hand side,
// which brings the largest entry of r to 2^-4 and leaves x_o and the even vectors 2^19 to grow.  The result is
// that of FP32 vectors at any size of the fields.
//
// Matrix blocks are stored in fragment order and go straight from L2 to registers, 16 bytes a lane; a
// block is used once per product and warp, so shared memory would not save a read.  G groups of four
// right-hand sides share a CTA (and its L1) when there are enough blocks to fill the chip; with fewer
// blocks each group is its own CTA.  mma.sync rather than tcgen05: a product has 80 rows and 8 columns
// per site, each site has its own matrix, and the result feeds the next product of the chain.
//
// 12 right-hand sides, nu = 2, the call: 32^4 (128 level-1 blocks of 2^4 sites, nc = 40) 2244 -> 645 us, a colour
// from 531 us with one thread per row on the CUDA cores; 16 blocks 249 us.
#include <algorithm>

#include <cuda_fp16.h>

#include "kernels.h"
#include "ml_ops.cuh"

namespace ddamg {

namespace {

constexpr float kSplit = 2048.f;  // scale of the low FP16 part

__device__ __forceinline__ void mma_k16(float (&d)[4], const uint4& a, unsigned b0, unsigned b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_k8(float (&d)[4], const uint2& a, unsigned b0) {
    asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};\n"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a.x), "r"(a.y), "r"(b0));
}
__device__ __forceinline__ unsigned h2u(__half2 v) { return *reinterpret_cast<unsigned*>(&v); }
// exponent of m >= 0 within -120 .. 120 (zero and subnormal numbers: -120), and 2^e for |e| <= 126
__device__ __forceinline__ int exponent_of(float m) { return max(-120, min(120, (int)(__float_as_uint(m) >> 23) - 127)); }
__device__ __forceinline__ float pow2(int e) { return __int_as_float((e + 127) << 23); }
constexpr int kTop = -4;  // scaled vectors start with their largest entry in [2^kTop, 2^(kTop + 1))

// two values as packed hi and lo halves
__device__ __forceinline__ void split2(float a, float b, unsigned& hi, unsigned& lo) {
    const __half2 h = __floats2half2_rn(a, b);
    const float2 f = __half22float2(h);
    hi = h2u(h);
    lo = h2u(__floats2half2_rn((a - f.x) * kSplit, (b - f.y) * kSplit));
}

// geometry of one block's fragments: U m-tiles, each KT k16 tiles of 512 bytes and, for odd U, one k8 tile of 256
template <int U>
struct Frag {
    static constexpr int KT = U / 2, REM = U & 1, CHUNK = KT * 512 + REM * 256, BYTES = U * CHUNK, NC = 8 * U;
    static constexpr int LDX = 8 * (U | 1);  // halves per staged column: an odd number of 16-byte pieces (no bank conflicts)
    static constexpr int PLANE = 8 * LDX, SLOT = 2 * PLANE;  // halves of one plane / of one site's (hi, lo) vectors
};

template <int U>
struct Acc {
    float hi[U][4], lo[U][4];
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int m = 0; m < U; ++m)
#pragma unroll
            for (int i = 0; i < 4; ++i) hi[m][i] = lo[m][i] = 0.f;
    }
    __device__ __forceinline__ float at(int m, int i) const { return fmaf(lo[m][i], 1.f / kSplit, hi[m][i]); }
    // y += f times the complex rows 8 q + g of right-hand side t
    __device__ __forceinline__ void add_rows(cplx<float> (&y)[U], float f = 1.f) const {
#pragma unroll
        for (int q = 0; q < U; ++q) {
            const int a = q >> 1, i = 2 * (q & 1), b = (q + U) >> 1, j = 2 * ((q + U) & 1);
            y[q].re = fmaf(f, at(a, i) - at(b, j + 1), y[q].re);
            y[q].im = fmaf(f, at(b, j) + at(a, i + 1), y[q].im);
        }
    }
};

// acc += B x for the staged vector x (SLOT halves in shared memory)
template <int U>
__device__ __forceinline__ void times_staged(Acc<U>& acc, const unsigned char* B, const __half* x, int lane) {
    using F = Frag<U>;
    const unsigned row = (unsigned)__cvta_generic_to_shared(x + (lane >> 4) * F::PLANE + (lane & 7) * F::LDX + 8 * ((lane >> 3) & 1));
#pragma unroll
    for (int kt = 0; kt < F::KT; ++kt) {
        unsigned b0, b1, c0, c1;
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(b0), "=r"(b1), "=r"(c0), "=r"(c1) : "r"(row + kt * 32) : "memory");
#pragma unroll
        for (int m = 0; m < U; ++m) {
            const uint4 a = __ldg(reinterpret_cast<const uint4*>(B + m * F::CHUNK + kt * 512) + lane);
            mma_k16(acc.hi[m], a, b0, b1);
            mma_k16(acc.lo[m], a, c0, c1);
        }
    }
    if constexpr (F::REM) {
        unsigned b0, c0;
        const unsigned r8 = (unsigned)__cvta_generic_to_shared(x + ((lane >> 3) & 1) * F::PLANE + (lane & 7) * F::LDX + 16 * F::KT);
        asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];" : "=r"(b0), "=r"(c0) : "r"(r8) : "memory");
#pragma unroll
        for (int m = 0; m < U; ++m) {
            const uint2 a = __ldg(reinterpret_cast<const uint2*>(B + m * F::CHUNK + F::KT * 512) + lane);
            mma_k8(acc.hi[m], a, b0);
            mma_k8(acc.lo[m], a, c0);
        }
    }
}
// acc += 2^(kTop - ex) B x for the vector x read from global memory: xr = this lane's right-hand side (column
// g >> 1) at the site, part = g & 1 (real or imaginary), on = false: zero; ex = the exponent of its largest entry
template <int U>
__device__ __forceinline__ void times_global(Acc<U>& acc, int& ex, const unsigned char* B, const cplx<float>* xr, int part, bool on, int lane) {
    using F = Frag<U>;
    const int t = lane & 3;
    float4 v[U];  // entries 8 j + 2 t, 8 j + 2 t + 1
#pragma unroll
    for (int j = 0; j < U; ++j) {
        v[j] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (on) v[j] = *reinterpret_cast<const float4*>(xr + 8 * j + 2 * t);
    }
    float m = 0.f;
#pragma unroll
    for (int j = 0; j < U; ++j) m = fmaxf(fmaxf(m, fmaxf(fabsf(v[j].x), fabsf(v[j].y))), fmaxf(fabsf(v[j].z), fabsf(v[j].w)));
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 1));
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 2));
    ex = exponent_of(m);
    const float f = pow2(kTop - ex);
    unsigned b[U], c[U];
#pragma unroll
    for (int j = 0; j < U; ++j) split2(f * (part ? v[j].y : v[j].x), f * (part ? v[j].w : v[j].z), b[j], c[j]);
#pragma unroll
    for (int kt = 0; kt < F::KT; ++kt)
#pragma unroll
        for (int m = 0; m < U; ++m) {
            const uint4 a = __ldg(reinterpret_cast<const uint4*>(B + m * F::CHUNK + kt * 512) + lane);
            mma_k16(acc.hi[m], a, b[2 * kt], b[2 * kt + 1]);
            mma_k16(acc.lo[m], a, c[2 * kt], c[2 * kt + 1]);
        }
    if constexpr (F::REM) {
#pragma unroll
        for (int m = 0; m < U; ++m) {
            const uint2 a = __ldg(reinterpret_cast<const uint2*>(B + m * F::CHUNK + F::KT * 512) + lane);
            mma_k8(acc.hi[m], a, b[U - 1]);
            mma_k8(acc.lo[m], a, c[U - 1]);
        }
    }
}
// stage sign * y (this lane's rows 8 q + g of right-hand side t) as (hi, lo) columns 2 t, 2 t + 1
template <int U>
__device__ __forceinline__ void stage(__half* x, const cplx<float> (&y)[U], float sign, int lane) {
    using F = Frag<U>;
    const int g = lane >> 2, t = lane & 3;
    __half* p = x + 2 * t * F::LDX + g;
#pragma unroll
    for (int q = 0; q < U; ++q) {
        const float re = sign * y[q].re, im = sign * y[q].im;
        const __half hr = __float2half_rn(re), hi = __float2half_rn(im);
        p[8 * q] = hr;
        p[F::LDX + 8 * q] = hi;
        p[F::PLANE + 8 * q] = __float2half_rn((re - __half2float(hr)) * kSplit);
        p[F::PLANE + F::LDX + 8 * q] = __float2half_rn((im - __half2float(hi)) * kSplit);
    }
}

}  // namespace

// grid: blocks of the colour x sets of G groups of four right-hand sides; 32 He threads per group
template <int U, int G>
__global__ void __launch_bounds__(G == 1 ? 512 : 256 * G, 1)
    ml_sap_tc_kernel(MLView<float> v, const cplx<float>* __restrict__ b, cplx<float>* z, int nrhs, int colour, int mr_steps) {
    using F = Frag<U>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int He = v.Vb1e, Vb = v.Vb1, NB = v.NB;
    const size_t fs = (size_t)NB * F::NC;
    const int nblk = v.NB2 / 2, c2 = colour * nblk + blockIdx.x % nblk;
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int grp = wid / He, s = wid % He;
    // shared memory: staged vectors of the even sites, the odd sites and each warp's own, [He][SLOT] per
    // group; r_e and x_o of each warp, [2][U][32]; partial products [He][4][3] per group; site tables
    __half* XE = reinterpret_cast<__half*>(smem_raw) + (size_t)grp * He * F::SLOT;
    __half* XO = XE + (size_t)G * He * F::SLOT;
    __half* XU = XO + (size_t)G * He * F::SLOT + (size_t)s * F::SLOT;
    cplx<float>* own = reinterpret_cast<cplx<float>*>(smem_raw + (size_t)3 * G * He * F::SLOT * sizeof(__half)) + (size_t)wid * 2 * U * 32 + lane;
    float* red_all = reinterpret_cast<float*>(smem_raw + (size_t)3 * G * He * F::SLOT * sizeof(__half) + (size_t)G * He * 2 * U * 32 * sizeof(cplx<float>));
    float* red = red_all + grp * He * 12;
    int* site = reinterpret_cast<int*>(red_all + G * He * 12);  // [Vb] level-k site of local index l
    int* nbl = site + Vb;                                       // [Vb][8] local index of the in-block neighbour, or -1
    for (int l = threadIdx.x; l < Vb; l += blockDim.x) site[l] = v.sites[(size_t)c2 * Vb + l];
    __syncthreads();
    for (int q = threadIdx.x; q < Vb * 8; q += blockDim.x) {
        const int l = q / 8, d = q % 8, c = site[l];
        nbl[q] = v.same[(size_t)d * NB + c] ? v.loc_of[v.nbr1[(size_t)d * NB + c]] : -1;
    }
    __syncthreads();
    const int r0 = (blockIdx.x / nblk * G + grp) * 4;
    const int nr = nrhs - r0;
    if (nr <= 0) return;  // the barriers below are per group
    auto sync = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(grp + 1), "r"(32 * He) : "memory"); };
    const unsigned char* Bm = reinterpret_cast<const unsigned char*>(v.B1h);
    const unsigned char* Dm = reinterpret_cast<const unsigned char*>(v.Dinv1h);
    auto blk = [&](int c, int d) { return Bm + ((size_t)c * 9 + d) * F::BYTES; };
    const int ce = site[s], co = site[He + s];  // this warp's even and odd site
    Acc<U> acc;
    cplx<float> y[U], rho[U];
    auto clear = [](cplx<float> (&v)[U]) {
#pragma unroll
        for (int q = 0; q < U; ++q) v[q] = czero<float>();
    };
    // y = r at site c: b - D_k z (z of out-of-block neighbours belongs to the other colour, not written here)
    auto residual = [&](int c) {
        clear(y);
        const bool on = (g >> 1) < nr;
        const cplx<float>* zr = z + (size_t)(r0 + (on ? g >> 1 : 0)) * fs;
#pragma unroll 1
        for (int d = 0; d < 9; ++d) {
            const int n = d == 0 ? c : __ldg(v.nbr1 + (size_t)(d - 1) * NB + c);
            int ex;
            acc.zero();
            times_global<U>(acc, ex, blk(c, d), zr + (size_t)n * F::NC, g & 1, on, lane);
            acc.add_rows(y, pow2(__shfl_sync(0xffffffffu, ex, 8 * t) - kTop));
        }
        const cplx<float>* br = b + (size_t)(r0 + (t < nr ? t : 0)) * fs + (size_t)c * F::NC + g;
#pragma unroll
        for (int q = 0; q < U; ++q) y[q] = t < nr ? br[8 * q] - y[q] : czero<float>();
    };
    float big = 0.f;  // largest entry of r on this warp's sites, of right-hand side t
    auto note = [&]() {
#pragma unroll
        for (int q = 0; q < U; ++q) big = fmaxf(big, fmaxf(fabsf(y[q].re), fabsf(y[q].im)));
    };
    // acc += sum of the in-block hops of the staged field X (sites of the other parity, local indices from l0)
    auto hops = [&](cplx<float> (&v)[U], int l, int c, const __half* X, int l0) {
#pragma unroll 1
        for (int d = 0; d < 8; ++d) {
            const int n = nbl[l * 8 + d];
            if (n >= 0) {
                acc.zero();
                times_staged<U>(acc, blk(c, 1 + d), X + (size_t)(n - l0) * F::SLOT, lane);
                acc.add_rows(v);
            }
        }
    };
    // y <- D_ee^{-1} y on the even site
    auto inv_even = [&]() {
        __syncwarp();
        stage<U>(XU, y, 1.f, lane);
        __syncwarp();
        acc.zero();
        times_staged<U>(acc, Dm + (size_t)ce * F::BYTES, XU, lane);
        clear(y);
        acc.add_rows(y);
    };
    residual(ce);
    note();
#pragma unroll
    for (int q = 0; q < U; ++q) own[q * 32] = y[q];  // r_e
    residual(co);
    note();
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) big = fmaxf(big, __shfl_xor_sync(0xffffffffu, big, o));
    if (g == 0) red[s * 4 + t] = big;
    sync();
    for (int q = 0; q < He; ++q) big = fmaxf(big, red[q * 4 + t]);
    // from here on the block's vectors are 2^(kTop - ex) times r and x
    const int ex = exponent_of(big);
    const float down = pow2(kTop - ex);
#pragma unroll
    for (int q = 0; q < U; ++q) {
        rho[q] = down * y[q];
        y[q] = down * own[q * 32];
        own[q * 32] = y[q];
        own[(U + q) * 32] = czero<float>();
    }
    inv_even();
    stage<U>(XE + (size_t)s * F::SLOT, y, -1.f, lane);
    sync();
    // rho = r_o - A_oe A_ee^{-1} r_e
    hops(rho, He + s, co, XE, 0);
#pragma unroll
    for (int q = 0; q < U; ++q) y[q] = mr_steps > 0 ? rho[q] : czero<float>();
    stage<U>(XO + (size_t)s * F::SLOT, y, 1.f, lane);
    sync();
#pragma unroll 1
    for (int it = 0; it < mr_steps; ++it) {
        clear(y);  // t_e = A_ee^{-1} A_eo rho, staged with the sign it enters S rho with
        hops(y, s, ce, XO, He);
        inv_even();
        stage<U>(XE + (size_t)s * F::SLOT, y, -1.f, lane);
        sync();
        clear(y);  // S rho = A_oo rho - A_oe t_e
        acc.zero();
        times_staged<U>(acc, blk(co, 0), XO + (size_t)s * F::SLOT, lane);
        acc.add_rows(y);
        hops(y, He + s, co, XE, 0);
        float nre = 0.f, nim = 0.f, den = 0.f;
#pragma unroll
        for (int q = 0; q < U; ++q) {
            nre += y[q].re * rho[q].re + y[q].im * rho[q].im;
            nim += y[q].re * rho[q].im - y[q].im * rho[q].re;
            den += y[q].re * y[q].re + y[q].im * y[q].im;
        }
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) {
            nre += __shfl_xor_sync(0xffffffffu, nre, o);
            nim += __shfl_xor_sync(0xffffffffu, nim, o);
            den += __shfl_xor_sync(0xffffffffu, den, o);
        }
        if (g == 0) red[(s * 4 + t) * 3] = nre, red[(s * 4 + t) * 3 + 1] = nim, red[(s * 4 + t) * 3 + 2] = den;
        sync();
        nre = nim = den = 0.f;
        for (int q = 0; q < He; ++q) nre += red[(q * 4 + t) * 3], nim += red[(q * 4 + t) * 3 + 1], den += red[(q * 4 + t) * 3 + 2];
        const cplx<float> alpha = den > ml_den_floor<float>() ? mk(nre / den, nim / den) : czero<float>();
        const bool last = it == mr_steps - 1;
#pragma unroll
        for (int q = 0; q < U; ++q) {  // x_o += alpha rho, rho -= alpha S rho; the staged field is rho, at the end -x_o
            cplx<float> xo = own[(U + q) * 32];
            cmac(xo, alpha, rho[q]);
            own[(U + q) * 32] = xo;
            rho[q] = rho[q] - alpha * y[q];
            y[q] = last ? mk(-xo.re, -xo.im) : rho[q];
        }
        stage<U>(XO + (size_t)s * F::SLOT, y, 1.f, lane);
        sync();
    }
    // x_e = A_ee^{-1} (r_e - A_eo x_o); z += x on the block
#pragma unroll
    for (int q = 0; q < U; ++q) y[q] = own[q * 32];
    hops(y, s, ce, XO, He);
    inv_even();
    if (t < nr) {
        const float f = pow2(ex - kTop);
        cplx<float>* ze = z + (size_t)(r0 + t) * fs + (size_t)ce * F::NC + g;
        cplx<float>* zo = z + (size_t)(r0 + t) * fs + (size_t)co * F::NC + g;
        cplx<float> u[U], w[U];
#pragma unroll
        for (int q = 0; q < U; ++q) u[q] = ze[8 * q], w[q] = zo[8 * q];
#pragma unroll
        for (int q = 0; q < U; ++q) ze[8 * q] = u[q] + f * y[q], zo[8 * q] = w[q] + f * own[(U + q) * 32];
    }
}

// FP64 column-major blocks -> FP16 fragments: per block, m-tile by m-tile, the k16 tiles (a lane's four
// registers side by side) and the k8 tile (two registers)
__global__ void pack_frag_kernel(const double* __restrict__ in, __half2* __restrict__ out, size_t nblk, int nc) {
    const int U = nc / 8, KT = U / 2, per_m = KT * 128 + (U & 1) * 64;  // half2 per m-tile
    const size_t tot = nblk * U * per_m;
    for (size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x; q < tot; q += (size_t)gridDim.x * blockDim.x) {
        const size_t blk = q / ((size_t)U * per_m);
        const int e = (int)(q % ((size_t)U * per_m)), m = e / per_m, f = e % per_m;
        int lane, reg, k0;
        if (f < KT * 128) {
            lane = (f % 128) / 4, reg = f % 4;
            k0 = (f / 128) * 16 + 2 * (lane & 3) + 8 * (reg >> 1);
        } else {
            lane = (f - KT * 128) / 2, reg = f & 1;
            k0 = KT * 16 + 2 * (lane & 3);
        }
        const int row = m * 16 + (lane >> 2) + 8 * (reg & 1);
        const int a = row < nc ? row : row - nc, part = row < nc ? 0 : 1;
        const double* B = in + blk * nc * nc * 2;
        const float x = (float)B[((size_t)k0 * nc + a) * 2 + part], y = (float)B[((size_t)(k0 + 1) * nc + a) * 2 + part];
        out[q] = __halves2half2(__float2half_rn(x), __float2half_rn(y));
    }
}
int pack_ml_frag(const double* in, void* out, size_t nblk, int nc, cudaStream_t st) {
    const size_t tot = nblk * nc * nc;
    pack_frag_kernel<<<std::min<size_t>((tot + 255) / 256, 152 * 16), 256, 0, st>>>(in, reinterpret_cast<__half2*>(out), nblk, nc);
    DD_CHECK_LAUNCH();
    return 0;
}

bool ml_sap_tc_supported(int nc, int Vb1, int Vb1e) { return nc % 8 == 0 && nc >= 16 && nc <= 48 && Vb1 == 2 * Vb1e && Vb1e <= 16; }

template <int U, int G>
static int launch_ug(const MLView<float>& v, const cplx<float>* b, cplx<float>* z, int nrhs, int colour, int mr_steps, cudaStream_t st) {
    using F = Frag<U>;
    const int He = v.Vb1e;
    const size_t smem = (size_t)3 * G * He * F::SLOT * sizeof(__half) + (size_t)G * He * 2 * U * 32 * sizeof(cplx<float>) +
                        (size_t)G * He * 12 * sizeof(float) + (size_t)v.Vb1 * 9 * sizeof(int);
    DD_CUDA((allow_smem<ml_sap_tc_kernel<U, G>>(200 * 1024)));
    const unsigned grid = (unsigned)(v.NB2 / 2) * (unsigned)ceil_div(nrhs, 4 * G);
    ml_sap_tc_kernel<U, G><<<grid, 32 * He * G, smem, st>>>(v, b, z, nrhs, colour, mr_steps);
    DD_CHECK_LAUNCH();
    return 0;
}
template <int U>
static int launch_u(const MLView<float>& v, const cplx<float>* b, cplx<float>* z, int nrhs, int colour, int mr_steps, cudaStream_t st) {
    // Three groups per CTA read each matrix block once from L2 (12 fields, 128 blocks of nc = 40, the call: 641 us
    // against 695 us with one group per CTA); one group per CTA spreads few blocks over more SMs (16 blocks, a
    // colour: 62 against about 134 us).  The line is one CTA per SM at one group each.  At nc = 48 the 80 registers
    // of the wide form spill (blocks of 8 sites, the call: 826 us with one group, 996 us with three).
    const bool wide = v.Vb1e <= 8 && nrhs > 4 && (long long)(v.NB2 / 2) * ceil_div(nrhs, 4) > 152;
    if constexpr (U < 6)
        if (wide) return launch_ug<U, 3>(v, b, z, nrhs, colour, mr_steps, st);
    return launch_ug<U, 1>(v, b, z, nrhs, colour, mr_steps, st);
}
int launch_ml_sap_tc(const MLView<float>& v, const cplx<float>* b, cplx<float>* z, int nrhs, int colour, int mr_steps, cudaStream_t st) {
    switch (v.nc / 8) {
        case 2: return launch_u<2>(v, b, z, nrhs, colour, mr_steps, st);
        case 3: return launch_u<3>(v, b, z, nrhs, colour, mr_steps, st);
        case 4: return launch_u<4>(v, b, z, nrhs, colour, mr_steps, st);
        case 5: return launch_u<5>(v, b, z, nrhs, colour, mr_steps, st);
        case 6: return launch_u<6>(v, b, z, nrhs, colour, mr_steps, st);
        default: return DDAMG_ERR_INVALID_ARG;
    }
}

}  // namespace ddamg
