// The two-dimensional flows of Sec. 6.1 with the exact trace: joint state y = [z; l],
//   z' = v(t, z) = (1/w) sum_j U_j(t) tanh(W_j(t) . z + b_j(t)),     l' = -tr(dv/dz) = -(1/w) sum_j (U_j . W_j) (1 - tanh^2(W_j . z + b_j)),
// the w weight sets (W_j, b_j, U_j) produced from t by three fully connected layers of hidden width h (tanh between them).
// State width d <= 8, so nothing here is a tensor-core contraction.  The usual path is hyper_solve.cu (the whole solve per launch).
// This file has the stage-by-stage kernels for shapes whose weight sets of a step's stages do not fit shared memory: per stage
// evaluation one launch in which every block evaluates the hypernetwork for the stage time into its
// shared memory (block 0 keeps a copy for the backward pass) and then the velocity with one thread per sample; the
// vector-Jacobian product is two launches: per-sample unit cotangents and psi, then one block per weight set that sums its
// cotangents over the batch in a fixed order, and the block that finishes last runs the hypernetwork backwards.
// Rounding points (the paper lists none): the hypernetwork's two hidden layers and its output, the products c_j = Q16(U_j . W_j),
// the units a_j = Q16(tanh(.)), the two outputs; in the vector-Jacobian product the unit cotangents, psi, and the batch-summed
// cotangents of the hypernetwork's output and hidden layers.  Sums are fp32 in a fixed order, one rounding per tensor.
#include "hyper_cnf.h"

#include <math.h>

namespace mpode {
namespace {

#define MPODE_DISPATCH_T(dt, T, ...)                                         \
    do {                                                                     \
        if ((dt) == MPODE_BF16) { using T = __nv_bfloat16; __VA_ARGS__; }    \
        else if ((dt) == MPODE_F16) { using T = __half; __VA_ARGS__; }       \
        else { using T = float; __VA_ARGS__; }                               \
    } while (0)

template <typename T> __device__ __forceinline__ float q16(float x) { return Low<T>::to_f(Low<T>::from_f(x)); }
template <typename T> __device__ __forceinline__ bool q_bad(float rounded) { return Low<T>::nonfinite(Low<T>::from_f(rounded)); }

// Layout of the per-stage block of floats `hyp`: h1 [h], h2 [h], o [m] = W [w][d], b [w], U [w][d], then c [w].

// theta: A1 [h][1], c1 [h], A2 [h][h], c2 [h], A3 [m][h], c3 [m]
struct ThetaOffsets { int A1, c1, A2, c2, A3, c3; };
__host__ __device__ inline ThetaOffsets theta_offsets(int h, int m) {
    ThetaOffsets o;
    o.A1 = 0; o.c1 = h; o.A2 = 2 * h; o.c2 = 2 * h + h * h; o.A3 = 3 * h + h * h; o.c3 = o.A3 + m * h;
    return o;
}

// The hypernetwork for one stage time, by all threads of a block: h1, h2 (shared memory, h floats each), `ws` = W [w][d], b [w],
// U [w][d], c [w] (shared memory).  `keep` (global, or null): h1, h2, ws in that order, for the backward pass.
template <typename T>
__device__ void hyper_eval_block(const float* __restrict__ theta, float tau16, int h, int w, int d, float* h1, float* h2, float* ws,
                                 float* __restrict__ keep) {
    const int m = w * (2 * d + 1);
    const ThetaOffsets o = theta_offsets(h, m);
    for (int i = threadIdx.x; i < h; i += blockDim.x)
        h1[i] = q16<T>(tanhf(fmaf(q16<T>(theta[o.A1 + i]), tau16, q16<T>(theta[o.c1 + i]))));
    __syncthreads();
    for (int i = threadIdx.x; i < h; i += blockDim.x) {
        float z = 0.f;
        for (int j = 0; j < h; ++j) z = fmaf(q16<T>(theta[o.A2 + i * h + j]), h1[j], z);
        h2[i] = q16<T>(tanhf(z + q16<T>(theta[o.c2 + i])));
    }
    __syncthreads();
    for (int i = threadIdx.x; i < m; i += blockDim.x) {
        float z = 0.f;
#pragma unroll 4
        for (int j = 0; j < h; ++j) z = fmaf(q16<T>(theta[o.A3 + i * h + j]), h2[j], z);
        ws[i] = q16<T>(z + q16<T>(theta[o.c3 + i]));
    }
    __syncthreads();
    const float* W = ws;
    const float* U = ws + w * d + w;
    for (int j = threadIdx.x; j < w; j += blockDim.x) {
        float c = 0.f;
        for (int k = 0; k < d; ++k) c = fmaf(U[j * d + k], W[j * d + k], c);
        ws[m + j] = q16<T>(c);
    }
    __syncthreads();
    if (keep != nullptr) {
        for (int i = threadIdx.x; i < h; i += blockDim.x) { keep[i] = h1[i]; keep[h + i] = h2[i]; }
        for (int i = threadIdx.x; i < m + w; i += blockDim.x) keep[2 * h + i] = ws[i];
    }
}

// k = [v; -tr]: one thread per sample; A [w][B] keeps the units for the vector-Jacobian product.  DC: the state width when it is a
// compile-time constant (loops unrolled, the sample's vectors in registers), 0 = any width up to HYPER_MAX_D.
template <typename T, int DC>
__global__ void __launch_bounds__(256) hyper_forward_kernel(const float* __restrict__ theta, float tau16, int h, int w, int d_rt,
                                                             float* __restrict__ hyp, const T* __restrict__ Y, T* __restrict__ A,
                                                             T* __restrict__ k, T* __restrict__ k_l, int B) {
    chain_begin();
    constexpr int DM = DC > 0 ? DC : HYPER_MAX_D;
    const int d = DC > 0 ? DC : d_rt;
    extern __shared__ float sm[];                     // h1 [h], h2 [h], W [w][d], b [w], U [w][d], c [w]
    hyper_eval_block<T>(theta, tau16, h, w, d, sm, sm + h, sm + 2 * h, blockIdx.x == 0 ? hyp : nullptr);
    const float* W = sm + 2 * h;
    const float* bb = W + w * d;
    const float* U = bb + w;
    const float* c = U + w * d;
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B) return;
    float z[DM], v[DM];
#pragma unroll
    for (int i = 0; i < DM; ++i) { z[i] = i < d ? Low<T>::to_f(Y[(long long)b * d + i]) : 0.f; v[i] = 0.f; }
    float tr = 0.f;
#pragma unroll 4
    for (int j = 0; j < w; ++j) {
        float s = 0.f;
#pragma unroll
        for (int i = 0; i < DM; ++i)
            if (i < d) s = fmaf(W[j * d + i], z[i], s);
        const T aq = Low<T>::from_f(tanhf(s + bb[j]));
        A[(long long)j * B + b] = aq;
        const float a = Low<T>::to_f(aq);
#pragma unroll
        for (int i = 0; i < DM; ++i)
            if (i < d) v[i] = fmaf(U[j * d + i], a, v[i]);
        tr = fmaf(c[j], 1.f - a * a, tr);
    }
    const float inv_w = 1.f / (float)w;
#pragma unroll
    for (int i = 0; i < DM; ++i)
        if (i < d) k[(long long)b * d + i] = Low<T>::from_f(v[i] * inv_w);
    k_l[b] = Low<T>::from_f(-tr * inv_w);
}

// Per sample: the unit cotangents sbar_j = Q16(abar_j (1 - a_j^2)) into Sb [w][B], and psi = Q16(sum_j sbar_j W_j)
template <typename T, int DC>
__global__ void __launch_bounds__(256) hyper_unit_cot_kernel(const float* __restrict__ hyp, int h, int w, int d_rt, const T* __restrict__ A,
                                                              const T* __restrict__ kappa, const T* __restrict__ kappa_l, T* __restrict__ Sb,
                                                              T* __restrict__ psi, int B, unsigned* __restrict__ flag) {
    chain_begin();
    constexpr int DM = DC > 0 ? DC : HYPER_MAX_D;
    const int d = DC > 0 ? DC : d_rt;
    extern __shared__ float sm[];                     // W, b, U, c
    const int n = w * (2 * d + 1) + w;
    for (int i = threadIdx.x; i < n; i += blockDim.x) sm[i] = hyp[2 * h + i];
    __syncthreads();
    const float* W = sm;
    const float* U = sm + w * d + w;
    const float* c = U + w * d;
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    const bool on = b < B;
    float kz[DM], ps[DM];
#pragma unroll
    for (int i = 0; i < DM; ++i) { kz[i] = (on && i < d) ? Low<T>::to_f(kappa[(long long)b * d + i]) : 0.f; ps[i] = 0.f; }
    const float kl = on ? Low<T>::to_f(kappa_l[b]) : 0.f;
    const float inv_w = 1.f / (float)w;
    bool bad = false;
    if (on) {
#pragma unroll 4
        for (int j = 0; j < w; ++j) {
            const float a = Low<T>::to_f(A[(long long)j * B + b]);
            float ku = 0.f;
#pragma unroll
            for (int i = 0; i < DM; ++i)
                if (i < d) ku = fmaf(kz[i], U[j * d + i], ku);
            // l' = -tr: the trace's unit derivative -2 a c_j / w meets the cotangent -kappa_l
            const float abar = fmaf(kl * (2.f * inv_w) * c[j], a, ku * inv_w);
            const T sq = Low<T>::from_f(abar * (1.f - a * a));
            bad |= Low<T>::nonfinite(sq);
            Sb[(long long)j * B + b] = sq;
            const float sbar = Low<T>::to_f(sq);
#pragma unroll
            for (int i = 0; i < DM; ++i)
                if (i < d) ps[i] = fmaf(sbar, W[j * d + i], ps[i]);
        }
#pragma unroll
        for (int i = 0; i < DM; ++i)
            if (i < d) {
                const T pq = Low<T>::from_f(ps[i]);
                bad |= Low<T>::nonfinite(pq);
                psi[(long long)b * d + i] = pq;
            }
    }
    warp_flag_or(flag, bad);
}

// The batch sums of weight set j's cotangents, Wbar_j = sum_b sbar z, bbar_j = sum_b sbar, Ubar_j = sum_b a kappa_z / w,
// cbar_j = -sum_b kappa_l (1 - a^2) / w (samples strided over the threads, lanes by shuffles, warps in ascending order), by all
// threads of a block into out[2 d + 2].  sm: [warps][2 d + 2] floats.
template <typename T>
__device__ void hyper_cot_sums(int j, int w, int d, const T* __restrict__ Y, const T* __restrict__ A, const T* __restrict__ Sb,
                               const T* __restrict__ kappa, const T* __restrict__ kappa_l, int B, float* __restrict__ out, float* sm) {
    const int nv = 2 * d + 2;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const float inv_w = 1.f / (float)w;
    float acc[2 * HYPER_MAX_D + 2];
#pragma unroll
    for (int q = 0; q < 2 * HYPER_MAX_D + 2; ++q) acc[q] = 0.f;
    for (int b = threadIdx.x; b < B; b += blockDim.x) {
        const float a = Low<T>::to_f(A[(long long)j * B + b]), sbar = Low<T>::to_f(Sb[(long long)j * B + b]);
        const float kl = Low<T>::to_f(kappa_l[b]);
#pragma unroll
        for (int i = 0; i < HYPER_MAX_D; ++i)
            if (i < d) {
                acc[i] = fmaf(sbar, Low<T>::to_f(Y[(long long)b * d + i]), acc[i]);
                acc[HYPER_MAX_D + 1 + i] = fmaf(a * inv_w, Low<T>::to_f(kappa[(long long)b * d + i]), acc[HYPER_MAX_D + 1 + i]);
            }
        acc[HYPER_MAX_D] += sbar;
        acc[2 * HYPER_MAX_D + 1] = fmaf(-kl * inv_w, 1.f - a * a, acc[2 * HYPER_MAX_D + 1]);
    }
    // registers are laid out for HYPER_MAX_D; the sums are stored densely: Wbar [d], bbar, Ubar [d], cbar
#pragma unroll
    for (int q = 0; q < 2 * HYPER_MAX_D + 2; ++q) {
        const bool used = q < HYPER_MAX_D ? q < d : (q == HYPER_MAX_D ? true : (q <= 2 * HYPER_MAX_D ? q - HYPER_MAX_D - 1 < d : true));
        if (used) {
            float x = acc[q];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
            const int dense = q < HYPER_MAX_D ? q : (q == HYPER_MAX_D ? d : (q <= 2 * HYPER_MAX_D ? d + 1 + (q - HYPER_MAX_D - 1) : 2 * d + 1));
            if (lane == 0) sm[warp * nv + dense] = x;
        }
    }
    __syncthreads();
    if (threadIdx.x < nv) {
        float x = 0.f;
        for (int ww = 0; ww < (int)(blockDim.x >> 5); ++ww) x += sm[ww * nv + threadIdx.x];
        out[threadIdx.x] = x;
        __threadfence();
    }
    __syncthreads();
}

// One stage's parameter gradient from the batch sums of its w weight sets, by all threads of a block: the chain rule through
// c_j = U_j . W_j, the rounded cotangent of the hypernetwork's output, then the hypernetwork backwards:
// dg = (beta != 0 ? beta * dg : 0) + gradient of this stage.  Every entry of dg is written by the same thread for every stage.
// sm: obar [m], h2bar [h], h1bar [h], partial sums [max(256, h)].  Returns whether a rounded value was non-finite.
template <typename T>
__device__ bool hyper_backprop(const float* __restrict__ hyp, const float* __restrict__ theta, float tau16, int h, int w, int d,
                               const float* __restrict__ sums, float* __restrict__ dg, float beta, float* sm) {
    const int m = w * (2 * d + 1), nv = 2 * d + 2;
    const ThetaOffsets o = theta_offsets(h, m);
    float* obar = sm;
    float* h2bar = sm + m;
    float* h1bar = h2bar + h;
    float* psum = h1bar + h;
    const float* h1 = hyp;
    const float* h2 = hyp + h;
    const float* W = hyp + 2 * h;
    const float* U = W + w * d + w;
    bool bad = false;
    for (int jj = threadIdx.x; jj < w; jj += blockDim.x) {
        const float* s = sums + (long long)jj * nv;
        const float cbar = __ldcg(s + 2 * d + 1);
        for (int i = 0; i < d; ++i) {
            const float wb = q16<T>(fmaf(cbar, U[jj * d + i], __ldcg(s + i)));
            const float ub = q16<T>(fmaf(cbar, W[jj * d + i], __ldcg(s + d + 1 + i)));
            bad |= q_bad<T>(wb) | q_bad<T>(ub);
            obar[jj * d + i] = wb;
            obar[w * d + w + jj * d + i] = ub;
        }
        const float bq = q16<T>(__ldcg(s + d));
        bad |= q_bad<T>(bq);
        obar[w * d + jj] = bq;
    }
    __syncthreads();
    auto put = [&](int idx, float v) { dg[idx] = (beta != 0.f ? beta * dg[idx] : 0.f) + v; };
    for (int i = threadIdx.x; i < m * h; i += blockDim.x) put(o.A3 + i, obar[i / h] * h2[i % h]);
    for (int i = threadIdx.x; i < m; i += blockDim.x) put(o.c3 + i, obar[i]);
    {   // t[k] = sum_i A3[i][k] obar[i]: the block's threads take interleaved pieces of the sum over i, added in ascending order
        const int parts = h <= (int)blockDim.x ? (int)blockDim.x / h : 1;
        const int k = threadIdx.x % h, pc = threadIdx.x / h;
        if (pc < parts) {
            for (int k0 = k; k0 < h; k0 += (int)blockDim.x) {      // one pass unless h exceeds the block
                float t = 0.f;
#pragma unroll 4
                for (int i = pc; i < m; i += parts) t = fmaf(q16<T>(theta[o.A3 + i * h + k0]), obar[i], t);
                psum[pc * h + k0] = t;
            }
        }
        __syncthreads();
        for (int k0 = threadIdx.x; k0 < h; k0 += blockDim.x) {
            float t = 0.f;
            for (int q = 0; q < parts; ++q) t += psum[q * h + k0];
            const float v = q16<T>((1.f - h2[k0] * h2[k0]) * t);
            bad |= q_bad<T>(v);
            h2bar[k0] = v;
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < h * h; i += blockDim.x) put(o.A2 + i, h2bar[i / h] * h1[i % h]);
    for (int i = threadIdx.x; i < h; i += blockDim.x) put(o.c2 + i, h2bar[i]);
    for (int l = threadIdx.x; l < h; l += blockDim.x) {
        float t = 0.f;
        for (int k = 0; k < h; ++k) t = fmaf(q16<T>(theta[o.A2 + k * h + l]), h2bar[k], t);
        const float v = q16<T>((1.f - h1[l] * h1[l]) * t);
        bad |= q_bad<T>(v);
        h1bar[l] = v;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < h; i += blockDim.x) { put(o.A1 + i, h1bar[i] * tau16); put(o.c1 + i, h1bar[i]); }
    __syncthreads();
    return bad;
}

// Block j: the batch sums of weight set j into sums[j][2 d + 2].  The block that finishes last (a counter that it sets back to
// zero) runs the hypernetwork backwards.
template <typename T>
__global__ void __launch_bounds__(256) hyper_param_cot_kernel(const float* __restrict__ hyp, const float* __restrict__ theta, float tau16, int h,
                                                               int w, int d, const T* __restrict__ Y, const T* __restrict__ A,
                                                               const T* __restrict__ Sb, const T* __restrict__ kappa, const T* __restrict__ kappa_l,
                                                               float* __restrict__ sums, float* __restrict__ dg, float beta, int B,
                                                               unsigned* __restrict__ flag, unsigned* __restrict__ counter) {
    chain_begin();
    extern __shared__ float sm[];
    __shared__ bool last;
    const int j = blockIdx.x, nv = 2 * d + 2;
    hyper_cot_sums<T>(j, w, d, Y, A, Sb, kappa, kappa_l, B, sums + (long long)j * nv, sm);
    if (threadIdx.x == 0) last = atomicAdd(counter, 1u) == (unsigned)(gridDim.x - 1);
    __syncthreads();
    if (!last) return;
    __threadfence();
    const bool bad = hyper_backprop<T>(hyp, theta, tau16, h, w, d, sums, dg, beta, sm);
    warp_flag_or(flag, bad);
    if (threadIdx.x == 0) *counter = 0u;
}

}  // namespace

size_t hyper_param_count(int h, int w, int d) {
    const int m = w * (2 * d + 1);
    return (size_t)3 * h + (size_t)h * h + (size_t)m * h + m;
}
size_t hyper_stage_floats(int h, int w, int d) { return (size_t)2 * h + (size_t)w * (2 * d + 1) + w; }
size_t hyper_scratch_floats(int w, int d) { return (size_t)w * (2 * d + 2); }
bool hyper_shape_ok(int h, int w, int d) {
    // the hypernetwork and the weight sets of one stage time live in shared memory
    const size_t fwd = ((size_t)2 * h + (size_t)w * (2 * d + 1) + w) * sizeof(float);
    const size_t fin = ((size_t)w * (2 * d + 1) + 2 * h + (h > 256 ? h : 256)) * sizeof(float);
    return d >= 1 && d <= HYPER_MAX_D && h >= 1 && w >= 1 && fwd <= 48 * 1024 && fin <= 48 * 1024;
}

void launch_hyper_forward(mpode_dtype dt, const float* theta, float tau16, int h, int w, int d, float* hyp, const void* Y, void* A, void* k,
                          void* k_l, int B, cudaStream_t st, long long* launches) {
    const size_t smem = ((size_t)2 * h + (size_t)w * (2 * d + 1) + w) * sizeof(float);
    const int blocks = (B + 255) / 256;
    if (d == 2) {
        MPODE_DISPATCH_T(dt, T, (launch_chain(hyper_forward_kernel<T, 2>, dim3(blocks), dim3(256), smem, st, theta, tau16, h, w, d, hyp, (const T*)Y, (T*)A, (T*)k, (T*)k_l, B)));
    } else {
        MPODE_DISPATCH_T(dt, T, (launch_chain(hyper_forward_kernel<T, 0>, dim3(blocks), dim3(256), smem, st, theta, tau16, h, w, d, hyp, (const T*)Y, (T*)A, (T*)k, (T*)k_l, B)));
    }
    if (launches) ++*launches;
}

void launch_hyper_vjp(mpode_dtype dt, const float* theta, float tau16, int h, int w, int d, const float* hyp, const void* Y, const void* A,
                      void* Sb, const void* kappa, const void* kappa_l, void* psi, float* sums, float* dg, float beta, int B, unsigned* flag,
                      unsigned* counter, cudaStream_t st, long long* launches) {
    const int blocks = (B + 255) / 256, nv = 2 * d + 2, m = w * (2 * d + 1);
    const size_t sm_unit = ((size_t)w * (2 * d + 1) + w) * sizeof(float);
    size_t sm_par = ((size_t)m + 2 * h + (h > 256 ? h : 256)) * sizeof(float);
    if (sm_par < (size_t)8 * nv * sizeof(float)) sm_par = (size_t)8 * nv * sizeof(float);
    if (d == 2) {
        MPODE_DISPATCH_T(dt, T, (launch_chain(hyper_unit_cot_kernel<T, 2>, dim3(blocks), dim3(256), sm_unit, st, hyp, h, w, d, (const T*)A, (const T*)kappa, (const T*)kappa_l,
                                                                                           (T*)Sb, (T*)psi, B, flag)));
    } else {
        MPODE_DISPATCH_T(dt, T, (launch_chain(hyper_unit_cot_kernel<T, 0>, dim3(blocks), dim3(256), sm_unit, st, hyp, h, w, d, (const T*)A, (const T*)kappa, (const T*)kappa_l,
                                                                                           (T*)Sb, (T*)psi, B, flag)));
    }
    if (launches) ++*launches;
    MPODE_DISPATCH_T(dt, T, (launch_chain(hyper_param_cot_kernel<T>, dim3(w), dim3(256), sm_par, st, hyp, theta, tau16, h, w, d, (const T*)Y, (const T*)A, (const T*)Sb,
                                                                               (const T*)kappa, (const T*)kappa_l, sums, dg, beta, B, flag, counter)));
    if (launches) ++*launches;
}

}  // namespace mpode
