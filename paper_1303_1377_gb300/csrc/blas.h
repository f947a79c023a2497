// Batched vector kernels and the device-side state of the batched (F)GMRES.
#pragma once
#include "common.cuh"

namespace ddamg {

// Per-right-hand-side Arnoldi/Givens state of a batched restarted (F)GMRES(m),
// all on the device.  H[r][i][k] (i <= m, k < m) is the rotated Hessenberg
// matrix, (cs, sn) the Givens rotations, g the rotated right-hand side.
struct KrylovState {
    int nrhs, m;
    cplx<double>* H;   // [nrhs][m+1][m]
    double* cs;        // [nrhs][m]
    cplx<double>* sn;  // [nrhs][m]
    cplx<double>* g;   // [nrhs][m+1]
    int* steps;        // Arnoldi steps taken in the current cycle
    double* resid;     // current residual estimate |g_{k+1}|
    int* active;       // still iterating in this cycle
    int* enabled;      // takes part in this solve at all
    int* flags;        // bit 1: non-finite value met
    double* target;    // absolute residual target tol * ||b||
    double* ctarget;   // target of the current cycle: max(target, cycle_tol * beta of the cycle)
    double cycle_tol;  // 0: a cycle runs to target (or the restart length)
};

// One Arnoldi step's Hessenberg column of right-hand side r, by one warp: w.col[0..k] = <V_i, w>, w.col[k+1].re =
// ||w||^2.  Rotates the column by the stored Givens rotations, forms the new one, updates the residual estimate
// and the flags, and returns on every lane the factor that normalises w (0: the right-hand side has converged or
// broken down).  An FP64 instruction occupies the warp's unit for 64 cycles whatever the number of active lanes
// (1/64 of the FP32 rate), so what the rotations do not chain is spread over the lanes: of a rotation only the
// running entry r <- c_i col_{i+1} - conj(sn_i) r is sequential (lane parity = real / imaginary part: two
// multiply-adds and a shuffle), and the square roots and quotients run side by side in four lanes.  One lane
// doing all of it took about 1 us per rotation and 10 us besides.
constexpr int kArnoldiMaxM = 64;
struct ArnoldiWork {
    cplx<double> col[kArnoldiMaxM + 1], sn[kArnoldiMaxM], d[kArnoldiMaxM], run[kArnoldiMaxM + 1];
    double cs[kArnoldiMaxM];
};
__device__ __forceinline__ double arnoldi_column(const KrylovState& s, int r, int k, int lane, ArnoldiWork& w) {
    const int m = s.m;
    cplx<double>* H = s.H + (size_t)r * (m + 1) * m;  // H[i * m + k]
    const cplx<double> gk = s.g[r * (m + 1) + k];
    const double prev = s.resid[r], ctarget = s.ctarget[r];  // prev = |g_k|
    for (int i = lane; i < k; i += 32) {
        w.cs[i] = s.cs[r * m + i];
        w.sn[i] = s.sn[r * m + i];
    }
    __syncwarp();
    for (int i = lane; i < k; i += 32) w.d[i] = w.cs[i] * w.col[i + 1];
    const int part = lane & 1;
    double x = part ? w.col[0].im : w.col[0].re;
    __syncwarp();
    for (int i = 0; i < k; ++i) {
        const double y = __shfl_xor_sync(0xffffffffu, x, 1);
        const cplx<double> sn = w.sn[i];
        if (lane < 2) reinterpret_cast<double*>(&w.run[i])[part] = x;
        x = fma(part ? sn.im : -sn.im, y, fma(-sn.re, x, part ? w.d[i].im : w.d[i].re));
    }
    const double y = __shfl_xor_sync(0xffffffffu, x, 1);
    const cplx<double> a = part ? mk(y, x) : mk(x, y);
    __syncwarp();
    for (int i = lane; i < k; i += 32) H[i * m + k] = w.cs[i] * w.run[i] + w.sn[i] * w.col[i + 1];
    const double n2 = w.col[k + 1].re, a2 = norm2(a);
    const double root = sqrt(lane == 0 ? n2 : lane == 1 ? a2 : a2 + n2);
    const double hk = __shfl_sync(0xffffffffu, root, 0), na = __shfl_sync(0xffffffffu, root, 1), den = __shfl_sync(0xffffffffu, root, 2);
    const double quot = (lane == 0 ? 1.0 : lane == 1 ? na : hk) / (lane == 0 ? hk : lane == 2 ? na * den : den);
    const double inv = __shfl_sync(0xffffffffu, quot, 0), q1 = __shfl_sync(0xffffffffu, quot, 1), q2 = __shfl_sync(0xffffffffu, quot, 2),
                 q3 = __shfl_sync(0xffffffffu, quot, 3);
    double sc = 0.0;
    if (lane == 0) {
        double c = q1, red = q3;
        cplx<double> sn = q2 * a;  // (a/|a|) conj(hk)/den, hk real
        if (den == 0.0) c = 1.0, red = 0.0, sn = mk(0.0, 0.0);
        else if (na == 0.0) c = 0.0, red = 1.0, sn = mk(1.0, 0.0);
        s.cs[r * m + k] = c;
        s.sn[r * m + k] = sn;
        H[k * m + k] = c * a + hk * sn;
        s.g[r * (m + 1) + k + 1] = -1.0 * (conj(sn) * gk);
        s.g[r * (m + 1) + k] = c * gk;
        const double est = red * prev;  // |g_{k+1}| = |sn| |g_k|
        s.steps[r] = k + 1;
        s.resid[r] = est;
        const bool nonfinite = !(est == est) || !(hk == hk);
        if (nonfinite) s.flags[r] |= 2;
        const bool done = est <= ctarget || nonfinite;
        if (done) s.active[r] = 0;
        sc = hk > 0.0 && !done ? inv : 0.0;
    }
    return __shfl_sync(0xffffffffu, sc, 0);
}

// Reduce-scatter of NV = 2 KB per-lane FP32 values across a warp (NV a power of two, <= 32): on
// return v[0] of lane l holds the sum over the 32 lanes of value (l mod NV).  Each halving step
// sends the half of the live values that the partner lane keeps, so the whole reduction costs
// NV - 1 shuffles (plus log2(32 / NV) for the lanes beyond NV) instead of 5 NV.
template <int NV>
__device__ __forceinline__ void warp_reduce_scatter(float (&v)[NV], int lane) {
#pragma unroll
    for (int s = NV / 2; s >= 1; s >>= 1) {
        const bool upper = lane & s;
#pragma unroll
        for (int j = 0; j < s; ++j) {
            const float send = upper ? v[j] : v[j + s];
            const float keep = upper ? v[j + s] : v[j];
            v[j] = keep + __shfl_xor_sync(0xffffffffu, send, s);
        }
    }
#pragma unroll
    for (int s = NV; s < 32; s <<= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], s);
}

// One Arnoldi step on short FP32 vectors (ortho.cu): V_{k+1} holds A V_k on entry and the next basis vector
// on exit; the Hessenberg column, the residual estimate and the flags of s are updated.
bool ortho_step_supported(const cplx<float>* V, size_t bstride, size_t n, int k);
int ortho_step_f32(const KrylovState& s, int k, cplx<float>* V, size_t bstride, size_t n, cudaStream_t st);

template <typename Ta, typename Tb>
int multidot(const cplx<Ta>* A, size_t istride, size_t arstride, int k, const cplx<Tb>* w, size_t wrstride, size_t n, int nrhs,
             cplx<double>* out, int ostride_i, double* scratch, cudaStream_t st);
template <typename To, typename Ta>
int lincomb(cplx<To>* out, size_t ors, double beta, const cplx<Ta>* A, size_t istride, size_t ars, int k, const cplx<double>* coef,
            int cstride_i, size_t n, int nrhs, const int* mask, cudaStream_t st, double alpha = 1.0);
int add_columns(cplx<double>* a, const cplx<double>* b, int n, cudaStream_t st);
// double-word vectors
template <>
int multidot<dwf, dwf>(const cplx<dwf>* A, size_t istride, size_t arstride, int k, const cplx<dwf>* w, size_t wrstride, size_t n,
                       int nrhs, cplx<double>* out, int ostride_i, double* scratch, cudaStream_t st);
int multidot_dw(const cplx<dwf>* A, size_t istride, size_t arstride, int k, const cplx<dwf>* w, size_t wrstride, size_t n, int nrhs,
                cplx<double>* out, int ostride_i, double* scratch, const int* run_flag, cudaStream_t st);
int axpy_norm_dw(cplx<dwf>* w, const cplx<dwf>* A, size_t istride, size_t rstride, int k, const cplx<double>* coef, int cstride_i,
                 size_t n, int nrhs, double alpha, float4* coef_scratch, double* scratch, cplx<double>* norm_out, const int* run_flag,
                 cudaStream_t st);
int dgks(const cplx<double>* before, const cplx<double>* after, const int* active, int nrhs, double eta, int* flag, cudaStream_t st);
int add_columns_flag(cplx<double>* a, const cplx<double>* b, int n, const int* flag, cudaStream_t st);
int lincomb_dw(cplx<dwf>* out, size_t ors, int beta1, const cplx<dwf>* A, size_t istride, size_t ars, int k, const cplx<double>* coef,
               int cstride_i, size_t n, int nrhs, double alpha, float4* coef_scratch, cudaStream_t st);
int xupdate_dw(cplx<double>* x, const cplx<float>* Z, size_t istride, size_t n, int k, const cplx<double>* coef, int nrhs,
               float4* coef_scratch, cudaStream_t st);
// FP32 basis (even n, 16-byte aligned vectors; -1 otherwise).  ticket: nrhs zeroed counters (left
// zeroed), used to let the last CTA of each right-hand side finish the reduction.  copy_last: also
// receives the last of the k products (may be null).
int multidot_f32(const cplx<float>* A, size_t istride, size_t arstride, int k, const cplx<float>* w, size_t wrstride, size_t n, int nrhs,
                 cplx<double>* out, int ostride_i, double* scratch, unsigned* ticket, cplx<double>* copy_last, const int* run_flag,
                 cudaStream_t st);
int axpy_norm_f32(cplx<float>* w, const cplx<float>* A, size_t istride, size_t rstride, int k, const cplx<double>* coef, int cstride_i,
                  size_t n, int nrhs, double alpha, double* scratch, unsigned* ticket, cplx<double>* norm_out, const int* run_flag,
                  cudaStream_t st);
int scale_f32(cplx<float>* w, const cplx<double>* scale, size_t n, int nrhs, cudaStream_t st);
int residual_f32(const cplx<double>* b, const cplx<double>* w, const cplx<float>* t, cplx<float>* out, size_t n, cudaStream_t st);
int split_f64(const cplx<double>* x, cplx<float>* hi, cplx<float>* lo, size_t n, cudaStream_t st);
int convert_d2dw(const double* in, cplx<dwf>* out, size_t nreal, cudaStream_t st);
int convert_dw2f(const cplx<dwf>* in, float* out, size_t nreal, cudaStream_t st);
template <typename To, typename Ti>
int convert(const Ti* in, To* out, size_t n, cudaStream_t st);
template <typename To, typename Ti>
int to_internal(const cplx<Ti>* in, cplx<To>* out, const int* lex_of, int V, int ncomp, int nrhs, cudaStream_t st);
// to_internal<float, double> that also leaves the bits of max |Re|, |Im| of each field in rmax
int to_internal_max(const cplx<double>* in, cplx<float>* out, const int* lex_of, int V, int ncomp, int nrhs, int* rmax, cudaStream_t st);
template <typename To, typename Ti>
int from_internal(const cplx<Ti>* in, cplx<To>* out, const int* lex_of, int V, int ncomp, int nrhs, cudaStream_t st);
template <typename To, typename Ti>
int coarse_perm(const cplx<Ti>* in, cplx<To>* out, const int* clex_of, int NB, int nc, int nrhs, int to_int, cudaStream_t st);
int gauge_to_internal(const cplx<double>* in, cplx<double>* out, const int* lex_of, int V, cudaStream_t st);

int arnoldi_start(const KrylovState& s, const cplx<double>* nrm2, cplx<double>* scale, int force_all, cudaStream_t st);
int arnoldi_update(const KrylovState& s, int k, const cplx<double>* hcol, cplx<double>* scale, cudaStream_t st);
int arnoldi_solve(const KrylovState& s, cplx<double>* y, cudaStream_t st);

// scratch size (doubles) needed by multidot for nrhs right-hand sides
inline size_t multidot_scratch_doubles(int nrhs) { return (size_t)(1216 / (nrhs > 0 ? nrhs : 1) + 1) * nrhs * 2 * 32 + 64; }

}  // namespace ddamg
