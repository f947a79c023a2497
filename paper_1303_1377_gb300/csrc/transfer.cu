// Aggregation-based transfer operators (Sec. 3.1-3.2): restriction P^H,
// prolongation P, the local orthonormalisation of the test vectors on every
// aggregate, and the assembly of the coarse stencil D_c = P^H D P.
//
// P is stored as N fine spinor fields P_j [N][12][V] (internal order): column
// (c, h, j) of P is P_j restricted to block c and spins {2h, 2h+1}.
// Coarse vectors: cplx[nrhs][NB][2N], component h*N + j.
#include <cuda_fp16.h>

#include "kernels.h"
#include "dirac.cuh"

namespace ddamg {

// ---------------------------------------------------------------------------
// restriction out[r][c][h*N + j] = sum_{x in c, k in half h} conj(P_j[k][x]) in[r][k][x]
// CTA = (block c, group of R right-hand sides), one thread per site of the block:
// every P_j entry loaded once serves R right-hand sides.  The 4R partial sums of one
// j are reduced over the warp by recursive halving (each lane keeps half of its
// values and trades the other half with its partner, so 4R values cost about 4R
// shuffles, not 4R log2(32)), then over the warps through shared memory.
// ---------------------------------------------------------------------------
template <int K>
__device__ __forceinline__ int bitrev_idx(int lane) {
    // value index held by a lane after the halving levels 1, 2, ..., K/2
    int q = 0;
#pragma unroll
    for (int m = 1, b = K >> 1; m < K; m <<= 1, b >>= 1)
        if (lane & m) q |= b;
    return q;
}

template <typename T, int K>
__device__ __forceinline__ T warp_transpose_sum(T (&v)[K], int lane) {
    // on return lane l holds the warp sum of value bitrev_idx<K>(l & (K-1))
#pragma unroll
    for (int m = 1, half = K >> 1; half >= 1; m <<= 1, half >>= 1) {
        const bool up = lane & m;
#pragma unroll
        for (int q = 0; q < half; ++q) {
            T send = up ? v[q] : v[q + half];
            T keep = up ? v[q + half] : v[q];
            v[q] = keep + __shfl_xor_sync(0xffffffffu, send, m);
        }
    }
    T s = v[0];
#pragma unroll
    for (int m = K; m < 32; m <<= 1) s += __shfl_xor_sync(0xffffffffu, s, m);
    return s;
}

template <typename T, typename Tp, int R, bool SPLIT>
__global__ void restrict_kernel(Geom g, const cplx<Tp>* __restrict__ P, int N, const cplx<T>* __restrict__ in,
                                cplx<T>* __restrict__ out, int r0, int ngroups) {
    // accumulation in the V-cycle precision T (FP64 arithmetic is a small fraction of FP32 on GB300)
    constexpr int K = 4 * R;
    extern __shared__ unsigned char smem_raw[];
    T* red = reinterpret_cast<T*>(smem_raw);  // [nwarps][N][K]
    const int rb = r0 + (blockIdx.x % ngroups) * R;
    const int c = blockIdx.x / ngroups;
    const int l = threadIdx.x;
    const bool act = l < g.Vb;
    const int i = c * g.Vb + l;
    cplx<T> x[R][12];
#pragma unroll
    for (int u = 0; u < R; ++u) {
        const cplx<T>* inr = in + (size_t)(rb + u) * 12 * g.V;
#pragma unroll
        for (int k = 0; k < 12; ++k) x[u][k] = act ? inr[(size_t)k * g.V + i] : czero<T>();
    }
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    const int myq = bitrev_idx<K>(lane & (K - 1));
    // SPLIT: gridDim.y CTAs per aggregate, each with its part of the test vectors
    const int j0 = SPLIT ? blockIdx.y * N / gridDim.y : 0, j1 = SPLIT ? (blockIdx.y + 1) * N / gridDim.y : N;
#pragma unroll 2
    for (int j = j0; j < j1; ++j) {
        T v[K];
#pragma unroll
        for (int q = 0; q < K; ++q) v[q] = 0;
        if (act) {
            const cplx<Tp>* pj = P + (size_t)j * 12 * g.V;
#pragma unroll
            for (int k = 0; k < 12; ++k) {
                const cplx<T> p = ccast<T>(pj[(size_t)k * g.V + i]);
                const int o = k < 6 ? 0 : 2;
#pragma unroll
                for (int u = 0; u < R; ++u) {
                    // conj(p) * x
                    v[4 * u + o] += p.re * x[u][k].re + p.im * x[u][k].im;
                    v[4 * u + o + 1] += p.re * x[u][k].im - p.im * x[u][k].re;
                }
            }
        }
        T s = warp_transpose_sum<T, K>(v, lane);
        if (lane < K) red[((size_t)w * N + j) * K + myq] = s;
    }
    __syncthreads();
    for (int q = K * j0 + threadIdx.x; q < K * j1; q += blockDim.x) {
        T s = 0;
        for (int ww = 0; ww < nw; ++ww) s += red[(size_t)ww * K * N + q];
        const int j = q / K, t = q % K;
        const int u = t >> 2, h = (t >> 1) & 1, im = t & 1;  // t = 4 u + 2 h + im
        T* o = reinterpret_cast<T*>(out + ((size_t)(rb + u) * g.NB + c) * (2 * N) + h * N + j);
        o[im] = s;
    }
}

// Few aggregates: several CTAs share one, each with a part of the test vectors (restriction) or of the twelve
// components (prolongation); a CTA reads its part of P one vector after the other and waits for each.  Up to 1216
// CTAs (eight of 256 threads per SM).  N = 20, one field: FP32 16^4 (256 aggregates) restriction 78 -> 37 us,
// prolongation 52 -> 32 us; 8^4 31 -> 10 and 19 -> 10 us; FP64 16^4 231 -> 203 and 131 -> 113 us.  The restriction of
// two fields per CTA is not split: with the vector range at run time the compiler keeps fewer loads in flight
// (24^4, 12 fields: 640 -> 1630 us).
static unsigned transfer_split(long long nblk, int parts) {
    unsigned s = 1;
    while (s < 4 && (int)(2 * s) <= parts && nblk * s * 2 <= 4 * 304) s *= 2;
    return s;
}

template <typename T, typename Tp, int R>
static int launch_restrict_r(const Geom& g, const cplx<Tp>* P, int N, const cplx<T>* in, cplx<T>* out, int r0, int ngroups,
                             cudaStream_t st) {
    const int nt = ((g.Vb + 31) / 32) * 32;
    const long long nblk = (long long)g.NB * ngroups;
    size_t sm = (size_t)(nt / 32) * 4 * R * N * sizeof(T);
    const unsigned split = R == 1 ? transfer_split(nblk, N) : 1;
    auto* kernel = restrict_kernel<T, Tp, R, false>;
    if constexpr (R == 1)
        if (split > 1) kernel = restrict_kernel<T, Tp, R, true>;
    if (sm > 48 * 1024) cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    kernel<<<dim3((unsigned)nblk, split), nt, sm, st>>>(g, P, N, in, out, r0, ngroups);
    DD_CHECK_LAUNCH();
    return 0;
}

// FP32 (and half-P) restriction takes 2 right-hand sides per CTA, FP64 one (register budget)
template <typename T, typename Tp>
int launch_restrict(const Geom& g, const cplx<Tp>* P, int N, const cplx<T>* in, cplx<T>* out, int nrhs, cudaStream_t st) {
    int r0 = 0;
    if constexpr (sizeof(T) == 4) if (nrhs >= 2) {
        { int e_ = (launch_restrict_r<T, Tp, 2>(g, P, N, in, out, 0, nrhs / 2, st)); if (e_) return e_; }
        r0 = nrhs / 2 * 2;
    }
    if (r0 < nrhs) { int e_ = (launch_restrict_r<T, Tp, 1>(g, P, N, in, out, r0, nrhs - r0, st)); if (e_) return e_; }
    return 0;
}

// ---------------------------------------------------------------------------
// prolongation out[r][k][x] = sum_j P_j[k][x] in[r][c(x)][h(k)*N + j]
// CTA = (block c, group of R right-hand sides); every P_j entry loaded once serves R.
// ---------------------------------------------------------------------------
// KC components per CTA: blockIdx.y * KC ...
template <typename T, typename Tp, int R, int KC>
__global__ void prolong_kernel(Geom g, const cplx<Tp>* __restrict__ P, int N, const cplx<T>* __restrict__ in,
                               cplx<T>* __restrict__ out, int r0, int ngroups) {
    extern __shared__ unsigned char smem_raw[];
    cplx<T>* e = reinterpret_cast<cplx<T>*>(smem_raw);  // [R][2N]
    const int rb = r0 + (blockIdx.x % ngroups) * R;
    const int c = blockIdx.x / ngroups;
    for (int q = threadIdx.x; q < 2 * N * R; q += blockDim.x) {
        const int u = q / (2 * N), t = q % (2 * N);
        e[q] = in[((size_t)(rb + u) * g.NB + c) * (2 * N) + t];
    }
    __syncthreads();
    const int l = threadIdx.x;
    if (l >= g.Vb) return;
    const int i = c * g.Vb + l;
    const int k0 = blockIdx.y * KC;
    cplx<T> acc[R][KC];
#pragma unroll
    for (int u = 0; u < R; ++u)
#pragma unroll
        for (int k = 0; k < KC; ++k) acc[u][k] = czero<T>();
#pragma unroll(R == 1 && (KC < 12 || sizeof(T) == 8) ? 4 : 1)
    for (int j = 0; j < N; ++j) {
        const cplx<Tp>* pj = P + (size_t)j * 12 * g.V;
        cplx<T> e0[R], e1[R];
#pragma unroll
        for (int u = 0; u < R; ++u) {
            e0[u] = e[u * 2 * N + j];
            e1[u] = e[u * 2 * N + N + j];
        }
#pragma unroll
        for (int k = 0; k < KC; ++k) {
            const cplx<T> p = ccast<T>(pj[(size_t)(k0 + k) * g.V + i]);
#pragma unroll
            for (int u = 0; u < R; ++u) cmac(acc[u][k], p, k0 + k < 6 ? e0[u] : e1[u]);
        }
    }
#pragma unroll
    for (int u = 0; u < R; ++u) {
        cplx<T>* o = out + (size_t)(rb + u) * 12 * g.V;
#pragma unroll
        for (int k = 0; k < KC; ++k) o[(size_t)(k0 + k) * g.V + i] = acc[u][k];
    }
}

template <typename T, typename Tp, int R>
static int launch_prolong_r(const Geom& g, const cplx<Tp>* P, int N, const cplx<T>* in, cplx<T>* out, int r0, int ngroups,
                            cudaStream_t st) {
    const int nt = ((g.Vb + 31) / 32) * 32;
    const long long nblk = (long long)g.NB * ngroups;
    const size_t sm = 2 * N * R * sizeof(cplx<T>);
    const unsigned split = transfer_split(nblk, 12);
    if (split == 4) prolong_kernel<T, Tp, R, 3><<<dim3((unsigned)nblk, 4), nt, sm, st>>>(g, P, N, in, out, r0, ngroups);
    else if (split == 2) prolong_kernel<T, Tp, R, 6><<<dim3((unsigned)nblk, 2), nt, sm, st>>>(g, P, N, in, out, r0, ngroups);
    else prolong_kernel<T, Tp, R, 12><<<(unsigned)nblk, nt, sm, st>>>(g, P, N, in, out, r0, ngroups);
    DD_CHECK_LAUNCH();
    return 0;
}

template <typename T, typename Tp>
int launch_prolong(const Geom& g, const cplx<Tp>* P, int N, const cplx<T>* in, cplx<T>* out, int nrhs, cudaStream_t st) {
    int r0 = 0;
    if constexpr (sizeof(T) == 4) if (nrhs >= 4) {
        { int e_ = (launch_prolong_r<T, Tp, 4>(g, P, N, in, out, 0, nrhs / 4, st)); if (e_) return e_; }
        r0 = nrhs / 4 * 4;
    }
    if (r0 < nrhs) { int e_ = (launch_prolong_r<T, Tp, 1>(g, P, N, in, out, r0, nrhs - r0, st)); if (e_) return e_; }
    return 0;
}

template int launch_restrict<double, double>(const Geom&, const cplx<double>*, int, const cplx<double>*, cplx<double>*, int,
                                             cudaStream_t);
template int launch_restrict<float, float>(const Geom&, const cplx<float>*, int, const cplx<float>*, cplx<float>*, int,
                                           cudaStream_t);
template int launch_restrict<float, __half>(const Geom&, const cplx<__half>*, int, const cplx<float>*, cplx<float>*, int,
                                            cudaStream_t);
template int launch_prolong<float, __half>(const Geom&, const cplx<__half>*, int, const cplx<float>*, cplx<float>*, int,
                                           cudaStream_t);
template int launch_prolong<double, double>(const Geom&, const cplx<double>*, int, const cplx<double>*, cplx<double>*, int,
                                            cudaStream_t);
template int launch_prolong<float, float>(const Geom&, const cplx<float>*, int, const cplx<float>*, cplx<float>*, int,
                                          cudaStream_t);

// ---------------------------------------------------------------------------
// local orthonormalisation (Sec. 3.1): modified Gram-Schmidt of P_1..P_N on every
// aggregate (block c, half h), in place, FP64.  CTA = (c, h), thread = site.
// ---------------------------------------------------------------------------
constexpr int kMaxVec = 32;  // params.n_vec is at most 32
__device__ __forceinline__ double block_sum_d(double v, double* red) {
    v = warp_sum(v);
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    __syncthreads();
    if (lane == 0) red[w] = v;
    __syncthreads();
    double s = 0;
    for (int q = 0; q < nw; ++q) s += red[q];
    return s;
}

// Right-looking: once p_j is normalised, all later vectors are projected against it, eight at a time, so that
// one block reduction serves eight inner products; each vector meets p_0, p_1, ... in the same order as in the
// left-looking form.  Bound by FP64 arithmetic (N^2 / 2 products and updates of 6 Vb components per aggregate
// half): 20 vectors on 16^4 5.08 -> 2.93 ms, where the left-looking form waited for two block reductions per
// pair of vectors.
template <int MAXT>
__global__ void __launch_bounds__(MAXT) gram_schmidt_kernel(Geom g, cplx<double>* __restrict__ P, int N, int* __restrict__ fail) {
    constexpr int Q = 8, K = 2 * Q;  // vectors and real numbers per reduction
    __shared__ double red[32], part[32][K], tot[K], orig_s[kMaxVec];
    const int c = blockIdx.x >> 1, h = blockIdx.x & 1;
    const int l = threadIdx.x, w = l >> 5, lane = l & 31, nw = blockDim.x >> 5;
    const bool act = l < g.Vb;
    const size_t V = g.V;
    cplx<double>* base = P + (size_t)(6 * h) * V + (size_t)c * g.Vb + (act ? l : 0);
    const int myq = bitrev_idx<K>(lane & (K - 1));
    // sums over the CTA of v[0..K) into tot (all threads may read it on return)
    auto sum_all = [&](double (&v)[K]) {
        const double t = warp_transpose_sum<double, K>(v, lane);
        __syncthreads();
        if (lane < K) part[w][myq] = t;
        __syncthreads();
        if (l < K) {
            double a = 0;
            for (int q = 0; q < nw; ++q) a += part[q][l];
            tot[l] = a;
        }
        __syncthreads();
    };
    for (int j0 = 0; j0 < N; j0 += K) {  // ||p_j||^2 as given
        double v[K];
#pragma unroll
        for (int u = 0; u < K; ++u) {
            v[u] = 0;
            if (act && j0 + u < N)
                for (int k = 0; k < 6; ++k) v[u] += norm2(base[((size_t)(j0 + u) * 12 + k) * V]);
        }
        sum_all(v);
        if (l < K && j0 + l < N) orig_s[j0 + l] = tot[l];
    }
    for (int j = 0; j < N; ++j) {
        cplx<double>* pj = base + (size_t)j * 12 * V;
        cplx<double> x[6];
        double nn = 0;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            x[k] = act ? pj[k * V] : czero<double>();
            nn += norm2(x[k]);
        }
        nn = block_sum_d(nn, red);
        const double orig = orig_s[j];
        if (!(nn > 1e-24 * orig) || !(orig > 0)) {
            if (threadIdx.x == 0) atomicExch(fail, 1);
            nn = 1.0;
        }
        const double inv = 1.0 / sqrt(nn);
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            x[k] = inv * x[k];
            if (act) pj[k * V] = x[k];
        }
        for (int q0 = j + 1; q0 < N; q0 += Q) {
            double v[K];
#pragma unroll
            for (int u = 0; u < Q; ++u) {
                cplx<double> d = czero<double>();
                if (act && q0 + u < N) {
                    const cplx<double>* pq = base + (size_t)(q0 + u) * 12 * V;
#pragma unroll
                    for (int k = 0; k < 6; ++k) cmac_conj(d, x[k], pq[k * V]);
                }
                v[2 * u] = d.re, v[2 * u + 1] = d.im;
            }
            sum_all(v);
            if (act)
#pragma unroll 2
                for (int u = 0; u < Q; ++u) {
                    if (q0 + u >= N) break;
                    const cplx<double> d = mk(-tot[2 * u], -tot[2 * u + 1]);
                    cplx<double>* pq = base + (size_t)(q0 + u) * 12 * V;
                    cplx<double> y[6];
#pragma unroll
                    for (int k = 0; k < 6; ++k) y[k] = pq[k * V];
#pragma unroll
                    for (int k = 0; k < 6; ++k) {
                        cmac(y[k], d, x[k]);
                        pq[k * V] = y[k];
                    }
                }
        }
    }
}

int launch_gram_schmidt(const Geom& g, cplx<double>* P, int N, int* fail, cudaStream_t st) {
    const int nt = ((g.Vb + 31) / 32) * 32;
    if (nt <= 256) gram_schmidt_kernel<256><<<2 * g.NB, nt, 0, st>>>(g, P, N, fail);
    else gram_schmidt_kernel<1024><<<2 * g.NB, nt, 0, st>>>(g, P, N, fail);
    DD_CHECK_LAUNCH();
    return 0;
}

// ---------------------------------------------------------------------------
// D_c assembly.  D = Gamma5 D^H Gamma5 and P commutes with Gamma5 (chirality halves), so half of the stencil
// follows from the other half:
//   B_{-mu}(c + mu) = Gamma5 B_{+mu}(c)^H Gamma5,   B_0 = X + Gamma5 X^H Gamma5,
// where X takes the forward hops inside the block and half of the (hermitian, chirality-diagonal) site term.
// For every column (h, j) of P (P_j restricted to spins {2h, 2h+1}) the forward direction dir gives
//   T_(h,j) = (A / 2 + forward in-block hops) P_j^(h)       (dir = 0)
//   T_(h,j) = forward hop in direction mu on the face sites (dir = 1 + 2 mu)
// and X / B_dir(c)[(h',j')][(h,j)] = sum_{x in c, k in half h'} conj(P_j'[k][x]) T_(h,j)[k][x].
// All of it is bound by FP64 arithmetic (1/64 of the FP32 rate); the symmetry leaves five of nine products
// with P^H and four of eight hops.  20 vectors on 16^4: T 9.51 -> 2.99 ms, products 15.35 -> 10.24 ms.
// ---------------------------------------------------------------------------

// acc += -1/2 (I - gamma_mu) (x) U_mu(x) psi for psi = the spins of half h of P_j at site nb
template <int MU, int H>
__device__ __forceinline__ void asm_hop(const cplx<double>* __restrict__ U, const cplx<double>* __restrict__ pj, size_t V, int i, int nb,
                                        cplx<double> (&acc)[12]) {
    using B = SpinB<MU>;
    cplx<double> hs[2][3];  // psi_up, or -B psi_low
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        if constexpr (H == 0) {
            hs[0][c] = pj[c * V + nb], hs[1][c] = pj[(3 + c) * V + nb];
        } else {
            const cplx<double> l2 = pj[(6 + c) * V + nb], l3 = pj[(9 + c) * V + nb];
            hs[0][c] = ipow<(B::p0 + 2) & 3>(B::c0 ? l3 : l2), hs[1][c] = ipow<(B::p1 + 2) & 3>(B::c1 ? l3 : l2);
        }
    }
    const cplx<double>* W = U + (size_t)(MU * 9) * V + i;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        cplx<double> g[2] = {czero<double>(), czero<double>()};
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const cplx<double> u = ldg_c(W + (size_t)(a * 3 + b) * V);
            cmac(g[0], u, hs[0][b]);
            cmac(g[1], u, hs[1][b]);
        }
        acc[a] = acc[a] + g[0], acc[3 + a] = acc[3 + a] + g[1];
        acc[6 + a] = acc[6 + a] - ipow<B::hp0>(g[B::hc0]), acc[9 + a] = acc[9 + a] - ipow<B::hp1>(g[B::hc1]);
    }
}
// in-block forward hop in direction MU
template <int MU, int H>
__device__ __forceinline__ void asm_hop_in(const Geom& g, const cplx<double>* U, const cplx<double>* pj, int c, int l, cplx<double> (&acc)[12]) {
    const int e = __ldg(g.lnbr + 2 * MU * g.Vb + l);
    if (!(e >> 16)) asm_hop<MU, H>(U, pj, g.V, c * g.Vb + l, c * g.Vb + (e & 0xffff), acc);
}
template <int H>
__device__ __forceinline__ void asm_self(const Geom& g, const FineOp<double>& op, const cplx<double>* __restrict__ pj, int i,
                                         cplx<double>* __restrict__ o) {
    const int c = block_of(g, i), l = i - c * g.Vb;
    const size_t V = g.V;
    cplx<double> acc[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) acc[k] = czero<double>();
    asm_hop_in<0, H>(g, op.U, pj, c, l, acc);
    asm_hop_in<1, H>(g, op.U, pj, c, l, acc);
    asm_hop_in<2, H>(g, op.U, pj, c, l, acc);
    asm_hop_in<3, H>(g, op.U, pj, c, l, acc);
    cplx<double> x[6], y[6];  // the site term acts inside half H
    const double* cl = op.clov + (size_t)(H * 36) * V + i;
#pragma unroll
    for (int a = 0; a < 6; ++a) {
        x[a] = pj[(size_t)(6 * H + a) * V + i];
        y[a] = __ldg(cl + a * V) * x[a];
    }
    int q = 0;
#pragma unroll
    for (int a = 0; a < 6; ++a)
#pragma unroll
        for (int b = a + 1; b < 6; ++b) {
            const cplx<double> m = mk(__ldg(cl + (size_t)(6 + 2 * q) * V), __ldg(cl + (size_t)(7 + 2 * q) * V));
            cmac(y[a], m, x[b]);
            cmac_conj(y[b], m, x[a]);
            ++q;
        }
#pragma unroll
    for (int k = 0; k < 12; ++k) o[(size_t)k * V + i] = (k / 6 == H) ? 0.5 * (y[k % 6] - acc[k]) : -0.5 * acc[k];
}

// dir = 0: thread = (site, column); dir = 1 + 2 mu: thread = (face site of a block, column)
__global__ void __launch_bounds__(128) assemble_T_kernel(Geom g, FineOp<double> op, const cplx<double>* __restrict__ P, int N, int dir, int col0,
                                                         int ncols, const int* __restrict__ sites, int nsites, cplx<double>* __restrict__ Tout) {
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int per = g.NB * nsites;  // sites of one column
    if (tid >= (long long)per * ncols) return;
    const int col = col0 + (int)(tid / per), q = (int)(tid % per);
    const int c = q / nsites, l = dir == 0 ? q % nsites : __ldg(sites + q % nsites);
    const int i = c * g.Vb + l, h = col / N, j = col % N;
    const size_t V = g.V;
    const cplx<double>* pj = P + (size_t)j * 12 * V;
    cplx<double>* o = Tout + (size_t)(col - col0) * 12 * V;
    if (dir == 0) {
        if (h == 0) asm_self<0>(g, op, pj, i, o);
        else asm_self<1>(g, op, pj, i, o);
        return;
    }
    const int nb = fine_nbr(g, i, dir - 1);
    cplx<double> acc[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) acc[k] = czero<double>();
    switch ((dir - 1) + h) {  // dir - 1 = 2 mu
        case 0: asm_hop<0, 0>(op.U, pj, V, i, nb, acc); break;
        case 1: asm_hop<0, 1>(op.U, pj, V, i, nb, acc); break;
        case 2: asm_hop<1, 0>(op.U, pj, V, i, nb, acc); break;
        case 3: asm_hop<1, 1>(op.U, pj, V, i, nb, acc); break;
        case 4: asm_hop<2, 0>(op.U, pj, V, i, nb, acc); break;
        case 5: asm_hop<2, 1>(op.U, pj, V, i, nb, acc); break;
        case 6: asm_hop<3, 0>(op.U, pj, V, i, nb, acc); break;
        default: asm_hop<3, 1>(op.U, pj, V, i, nb, acc); break;
    }
#pragma unroll
    for (int k = 0; k < 12; ++k) o[(size_t)k * V + i] = -0.5 * acc[k];
}

// T[col - col0] for the columns col0 .. col0 + ncols - 1 of the 2N, on the listed local sites of every block
// (dir = 0: all sites)
int launch_assemble_T(const Geom& g, const FineOp<double>& op, const cplx<double>* P, int N, int dir, int col0, int ncols, const int* sites,
                      int nsites, cplx<double>* T, cudaStream_t st) {
    const long long n = (long long)g.NB * nsites * ncols;
    assemble_T_kernel<<<ceil_div(n, 128), 128, 0, st>>>(g, op, P, N, dir, col0, ncols, sites, nsites, T);
    DD_CHECK_LAUNCH();
    return 0;
}

// The other half of the stencil: B_0 = X + Gamma5 X^H Gamma5 in place, B_{-mu}(c + mu) = Gamma5 B_{+mu}(c)^H Gamma5.
// One CTA per (site, direction: 0 = self, 1 + mu); blocks are [column][row].
__global__ void __launch_bounds__(256) complete_stencil_kernel(Geom g, int N, cplx<double>* __restrict__ B) {
    const int c = blockIdx.x, d = blockIdx.y, nc = 2 * N, nn = nc * nc;
    cplx<double>* src = B + ((size_t)c * 9 + (d == 0 ? 0 : 2 * d - 1)) * nn;
    auto flip = [&](int row, int col, cplx<double> v) { return (row < N) == (col < N) ? conj(v) : mk(-v.re, v.im); };
    if (d == 0) {
        for (int q = threadIdx.x; q < nn; q += blockDim.x) {
            const int col = q / nc, row = q % nc;
            if (row > col) continue;
            const cplx<double> a = src[col * nc + row], b = src[row * nc + col];
            src[col * nc + row] = a + flip(row, col, b);
            src[row * nc + col] = b + flip(row, col, a);
        }
    } else {
        const int mu = d - 1;
        cplx<double>* dst = B + ((size_t)__ldg(g.bnbr + 2 * mu * g.NB + c) * 9 + 2 + 2 * mu) * nn;
        for (int q = threadIdx.x; q < nn; q += blockDim.x) {
            const int col = q / nc, row = q % nc;
            dst[q] = flip(row, col, src[row * nc + col]);
        }
    }
}
int launch_complete_stencil(const Geom& g, int N, double* B, cudaStream_t st) {
    complete_stencil_kernel<<<dim3(g.NB, 5), 256, 0, st>>>(g, N, reinterpret_cast<cplx<double>*>(B));
    DD_CHECK_LAUNCH();
    return 0;
}

// B_dir(c) = P_c^H T on the listed local sites (all sites for dir 0, the face for dir > 0).
// CTA = (c, output tile); outputs column-major: o = col * nc + row.
constexpr int kProjThreads = 256;
constexpr int kProjPerThread = 8;

__global__ void __launch_bounds__(kProjThreads) block_project_kernel(Geom g, const cplx<double>* __restrict__ P, int N,
                                                                     const cplx<double>* __restrict__ Tin, int col0, int ncols,
                                                                     const int* __restrict__ sites, int nsites, int CH,
                                                                     double* __restrict__ Bout, size_t site_stride) {
    extern __shared__ unsigned char smem_raw[];
    const int nc = 2 * N;
    cplx<double>* Pc = reinterpret_cast<cplx<double>*>(smem_raw);  // [N][12][CH]
    cplx<double>* Tc = Pc + (size_t)N * 12 * CH;                      // [ncols][12][CH]
    const int c = blockIdx.x;
    // outputs o = (col - col0) * nc + row of this launch's columns
    const int o0 = blockIdx.y * kProjThreads * kProjPerThread;
    cplx<double> acc[kProjPerThread];
#pragma unroll
    for (int m = 0; m < kProjPerThread; ++m) acc[m] = czero<double>();
    for (int s0 = 0; s0 < nsites; s0 += CH) {
        __syncthreads();
        for (int q = threadIdx.x; q < N * 12 * CH; q += blockDim.x) {
            int s = q % CH, k = (q / CH) % 12, j = q / (12 * CH);
            cplx<double> v = czero<double>();
            if (s0 + s < nsites) v = P[((size_t)j * 12 + k) * g.V + (size_t)c * g.Vb + sites[s0 + s]];
            Pc[q] = v;
        }
        for (int q = threadIdx.x; q < ncols * 12 * CH; q += blockDim.x) {
            int s = q % CH, k = (q / CH) % 12, col = q / (12 * CH);
            cplx<double> v = czero<double>();
            if (s0 + s < nsites) v = Tin[((size_t)col * 12 + k) * g.V + (size_t)c * g.Vb + sites[s0 + s]];
            Tc[q] = v;
        }
        __syncthreads();
#pragma unroll
        for (int m = 0; m < kProjPerThread; ++m) {
            int o = o0 + m * kProjThreads + threadIdx.x;
            if (o >= ncols * nc) break;
            int col = o / nc, row = o % nc;  // col relative to col0
            int hp = row / N, jp = row % N;
            const cplx<double>* pr = Pc + ((size_t)jp * 12 + 6 * hp) * CH;
            const cplx<double>* tc = Tc + ((size_t)col * 12 + 6 * hp) * CH;
            for (int q = 0; q < 6 * CH; ++q) cmac_conj(acc[m], pr[q], tc[q]);
        }
    }
#pragma unroll
    for (int m = 0; m < kProjPerThread; ++m) {
        int o = o0 + m * kProjThreads + threadIdx.x;
        if (o >= ncols * nc) break;
        double* b = Bout + ((size_t)c * site_stride + (size_t)col0 * nc + o) * 2;
        b[0] = acc[m].re;
        b[1] = acc[m].im;
    }
}

int launch_block_project(const Geom& g, const cplx<double>* P, int N, const cplx<double>* T, int col0, int ncols, const int* sites,
                         int nsites, double* Bout, size_t site_stride, cudaStream_t st) {
    const int nc = 2 * N;
    int CH = (int)((160 * 1024) / ((size_t)(N + ncols) * 12 * sizeof(cplx<double>)));
    if (CH > 8) CH = 8;
    if (CH < 1) CH = 1;
    size_t smem = (size_t)(N + ncols) * 12 * CH * sizeof(cplx<double>);
    cudaFuncSetAttribute(block_project_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    dim3 grid(g.NB, ceil_div((long long)ncols * nc, kProjThreads * kProjPerThread));
    block_project_kernel<<<grid, kProjThreads, smem, st>>>(g, P, N, T, col0, ncols, sites, nsites, CH, Bout, site_stride);
    DD_CHECK_LAUNCH();
    return 0;
}

}  // namespace ddamg
