// One Arnoldi step of the batched FP32 GMRES on short vectors as one kernel: w = A V_k (in the V_{k+1}
// slot) is orthogonalised against V_0 .. V_k by one classical Gram-Schmidt pass, the Hessenberg column is
// rotated, and V_{k+1} = w / ||w|| is written.  The same steps as multidot_f32, axpy_norm_f32,
// arnoldi_update and scale_f32, which stay for long vectors.
//
// What bounds a step of these solvers is latency, not bytes: on the coarse lattices the vectors are tens of
// KB per right-hand side and sit in L2, while four launches with a grid-wide reduction each took about 25 us.
// Here a cluster of 8 CTAs owns one right-hand side: each CTA keeps its slice of w in shared memory, and the
// two reductions and the step size cross the cluster through distributed shared memory.
#include <cooperative_groups.h>

#include "blas.h"
#include "kernels.h"
#include "sum2.cuh"

namespace ddamg {

namespace cg = cooperative_groups;

constexpr int kOrthoCluster = 8, kOrthoThreads = 256, kOrthoWarps = kOrthoThreads / 32, kOrthoMaxK = 64;
// Largest slice of w, 1024 float4 (vectors of 16384 numbers).  A step with two stencil launches, k = 8 .. 30, one
// kernel against four: 320 numbers 32 / 42 us (1 field), 10240 numbers 38 / 48 us (1) and 48 / 61 us (12); at 25920
// numbers 61 / 62, 72 / 70 (4 fields) and 102 / 111 us (12), where eight CTAs per field begin to be too few.
constexpr size_t kOrthoMaxSlice = 1024;
static_assert(kOrthoMaxSlice <= 32 * kLaneWords);

__global__ void __cluster_dims__(kOrthoCluster, 1, 1) __launch_bounds__(kOrthoThreads)
    ortho_step_kernel(KrylovState s, int k, float4* __restrict__ V, size_t bstride4, size_t n4) {
    extern __shared__ float4 wsm[];
    __shared__ double part[2 * kOrthoMaxK], h[2 * kOrthoMaxK], nred[kOrthoWarps], npart, scale_s;
    __shared__ float2 cs[kOrthoMaxK];
    __shared__ ArnoldiWork aw;
    cg::cluster_group cl = cg::this_cluster();
    const int r = blockIdx.x / kOrthoCluster, rank = (int)cl.block_rank(), tid = threadIdx.x, wi = tid >> 5, lane = tid & 31, m = s.m;
    const size_t per = (n4 + kOrthoCluster - 1) / kOrthoCluster, e0 = rank * per;
    const int cnt = e0 < n4 ? (int)(n4 - e0 < per ? n4 - e0 : per) : 0;
    const float4* Vr = V + (size_t)r * n4 + e0;              // V_0's slice of this right-hand side
    float4* w = V + (size_t)(k + 1) * bstride4 + (size_t)r * n4 + e0;
    if (!s.active[r]) {  // a converged right-hand side is frozen (every CTA of the cluster leaves here)
        for (int e = tid; e < cnt; e += kOrthoThreads) w[e] = make_float4(0.f, 0.f, 0.f, 0.f);
        return;
    }
    for (int e = tid; e < cnt; e += kOrthoThreads) wsm[e] = w[e];
    __syncthreads();
    // <V_i, w>: one warp per product.  A lane's sums carry their rounding errors along, so that FP32 rounds a term and
    // five additions over the warp, as in multidot_f32, whatever the length of the slice (30 steps on 10240 numbers: 1.09
    // ms, with plain sums word by word 1.12 ms; multidot_f32 and the rest as separate kernels 2.17 ms); lanes 0 .. 3 end
    // with the two parts and their errors, which one FP64 conversion and one addition put together.
    for (int i = wi; i <= k; i += kOrthoWarps) {
        Sum2 re, im;
        lane_dot(Vr + (size_t)i * bstride4, wsm, lane, cnt, re, im);
        float v[4] = {re.s, im.s, re.e, im.e};
        warp_reduce_scatter<4>(v, lane);
        double t = (double)v[0];
        t += __shfl_down_sync(0xffffffffu, t, 2);
        if (lane < 2) part[2 * i + lane] = t;
    }
    cl.sync();
    for (int q = tid; q < 2 * (k + 1); q += kOrthoThreads) {
        double t = 0;
#pragma unroll
        for (int c = 0; c < kOrthoCluster; ++c) t += *cl.map_shared_rank(part + q, c);
        h[q] = t;
        reinterpret_cast<float*>(cs)[q] = -(float)t;
    }
    __syncthreads();
    // w -= sum_i h_i V_i, ||w||^2
    double nrm = 0;
    for (int e = tid; e < cnt; e += kOrthoThreads) {
        float4 acc = wsm[e];
#pragma unroll 4
        for (int i = 0; i <= k; ++i) {
            const float2 c = cs[i];
            const float4 a = Vr[(size_t)i * bstride4 + e];
            acc.x = fmaf(c.x, a.x, fmaf(-c.y, a.y, acc.x));
            acc.y = fmaf(c.x, a.y, fmaf(c.y, a.x, acc.y));
            acc.z = fmaf(c.x, a.z, fmaf(-c.y, a.w, acc.z));
            acc.w = fmaf(c.x, a.w, fmaf(c.y, a.z, acc.w));
        }
        wsm[e] = acc;
        nrm += (double)(acc.x * acc.x + acc.y * acc.y) + (double)(acc.z * acc.z + acc.w * acc.w);
    }
    nrm = warp_sum(nrm);
    if (lane == 0) nred[wi] = nrm;
    __syncthreads();
    if (tid == 0) {
        double t = 0;
        for (int q = 0; q < kOrthoWarps; ++q) t += nred[q];
        npart = t;
    }
    cl.sync();
    if (rank == 0 && wi == 0) {  // the Hessenberg column, rotated; the step size goes to every CTA of the cluster
        for (int i = lane; i <= k; i += 32) aw.col[i] = mk(h[2 * i], h[2 * i + 1]);
        double n2 = lane < kOrthoCluster ? *cl.map_shared_rank(&npart, lane) : 0.0;
        n2 = warp_sum(n2);
        if (lane == 0) aw.col[k + 1] = mk(n2, 0.0);
        __syncwarp();
        const double sc = arnoldi_column(s, r, k, lane, aw);
        if (lane < kOrthoCluster) *cl.map_shared_rank(&scale_s, lane) = sc;
    }
    cl.sync();
    const float a = (float)scale_s;
    for (int e = tid; e < cnt; e += kOrthoThreads) {
        float4 v = wsm[e];
        v.x *= a, v.y *= a, v.z *= a, v.w *= a;
        w[e] = v;
    }
}

bool ortho_step_supported(const cplx<float>* V, size_t bstride, size_t n, int k) {
    return n % 2 == 0 && bstride % 2 == 0 && ((uintptr_t)V & 15) == 0 && k + 1 <= kOrthoMaxK &&
           (n / 2 + kOrthoCluster - 1) / kOrthoCluster <= kOrthoMaxSlice;
}
int ortho_step_f32(const KrylovState& s, int k, cplx<float>* V, size_t bstride, size_t n, cudaStream_t st) {
    if (s.m > kOrthoMaxK || k >= s.m) return DDAMG_ERR_INVALID_ARG;
    const size_t n4 = n / 2, per = (n4 + kOrthoCluster - 1) / kOrthoCluster;
    ortho_step_kernel<<<(unsigned)kOrthoCluster * (unsigned)s.nrhs, kOrthoThreads, per * sizeof(float4), st>>>(s, k, reinterpret_cast<float4*>(V), bstride / 2, n4);
    DD_CHECK_LAUNCH();
    return 0;
}

}  // namespace ddamg
