// Whole-solve kernels of the hypernetwork flow with the exact trace (the velocity of hyper_cnf.cu): the time loop of Alg. 1 in one
// launch, and Alg. 2 with its scale decisions in one cooperative launch.  One warp per sample, a lane per weight set (w / 32 rounds),
// sums over the weight sets by a butterfly of shuffles.  Nothing here is bound by bytes or arithmetic: a step is a chain of stages
// (tanh and five shuffles each, about 0.4 us) and, backwards, two grid barriers.
//   forward  : samples are independent through the whole solve; the weight sets of the next step are copied to shared memory while
//              this one runs.
//   backward : per step every block recomputes its samples' stages and forms their stage and unit cotangents (group phase), then
//              sums the weight-set cotangents over its samples into its row of partial sums; barrier; the block that owns a weight
//              set adds the blocks' rows in ascending order, applies the chain rule and the last layer's gradient (set phase);
//              barrier; every block runs the two hidden layers backwards (they are small, and doing so in all blocks saves a third
//              barrier), takes Alg. 2's decision from the same words, and commits its share.  The stages of the step before are
//              recomputed while the first barrier is waited for: they do not depend on the outcome.
// Measured (1024 samples, 128 weight sets, 128 RK4 steps, float16 with dynamic scaling): 14.3 ms per training pass with launches per
// step, 3.56 ms with these two (forward 0.35, backward 3.25).
// Rounding points and formulas are those of hyper_cnf.cu; sums run in another, fixed order.
#include <math.h>

#include "hyper_cnf.h"
#include "tc_ptx.cuh"
#include "tensormap.h"

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

__device__ __forceinline__ float warp_sum(float x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

__device__ __forceinline__ void cp_async4(float* dst, const float* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// theta: A1 [h][1], c1 [h], A2 [h][h], c2 [h], A3 [m][h], c3 [m]
struct Offsets { int A1, c1, A2, c2, A3, c3; };
__host__ __device__ inline Offsets offsets(int h, int m) {
    Offsets o;
    o.A1 = 0; o.c1 = h; o.A2 = 2 * h; o.c2 = 2 * h + h * h; o.A3 = 3 * h + h * h; o.c3 = o.A3 + m * h;
    return o;
}

// ---------------------------------------------------------------- the weight sets of every stage time
// One block per step: h1, h2 and the weight sets of its (up to four) stage times, the last layer's rows read once for all of them.
template <typename T>
__global__ void __launch_bounds__(256) hyper_table_kernel(const float* __restrict__ theta, const RkStepScalars* __restrict__ scal, int stages, int h, int w,
                                                           int d, float* __restrict__ table, long long stage_floats) {
    extern __shared__ float sm[];                     // h1 [4][h], h2 [4][h]
    const int m = w * (2 * d + 1);
    const Offsets o = offsets(h, m);
    float* tab = table + (long long)blockIdx.x * RK_MAX_STAGES * stage_floats;
    float* h1 = sm;
    float* h2 = sm + RK_MAX_STAGES * h;
    for (int i = threadIdx.x; i < stages * h; i += blockDim.x) {
        const int j = i / h, k = i - j * h;
        h1[i] = q16<T>(tanhf(fmaf(q16<T>(theta[o.A1 + k]), scal[blockIdx.x].tau16[j], q16<T>(theta[o.c1 + k]))));
        tab[j * stage_floats + k] = h1[i];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < stages * h; i += blockDim.x) {
        const int j = i / h, k = i - j * h;
        float z = 0.f;
#pragma unroll 8
        for (int q = 0; q < h; ++q) z = fmaf(q16<T>(theta[o.A2 + k * h + q]), h1[j * h + q], z);
        h2[i] = q16<T>(tanhf(z + q16<T>(theta[o.c2 + k])));
        tab[j * stage_floats + h + k] = h2[i];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < m; i += blockDim.x) {
        float z[RK_MAX_STAGES] = {0.f, 0.f, 0.f, 0.f};
        const float* row = theta + o.A3 + (long long)i * h;
#pragma unroll 8
        for (int q = 0; q < h; ++q) {
            const float a = q16<T>(row[q]);
#pragma unroll
            for (int j = 0; j < RK_MAX_STAGES; ++j)
                if (j < stages) z[j] = fmaf(a, h2[j * h + q], z[j]);
        }
        const float c = q16<T>(theta[o.c3 + i]);
#pragma unroll
        for (int j = 0; j < RK_MAX_STAGES; ++j)
            if (j < stages) tab[j * stage_floats + 2 * h + i] = q16<T>(z[j] + c);
    }
    __syncthreads();                                  // the block reads back what it wrote
    for (int i = threadIdx.x; i < stages * w; i += blockDim.x) {
        const int j = i / w, u = i - j * w;
        float* ws = tab + j * stage_floats + 2 * h;
        float c = 0.f;
        for (int k = 0; k < d; ++k) c = fmaf(ws[w * d + w + u * d + k], ws[u * d + k], c);
        ws[m + u] = q16<T>(c);
    }
}

// One step's stage blocks and its scalars into shared memory (asynchronous); `step_floats` is their length there.
constexpr int kScalarFloats = sizeof(RkStepScalars) / sizeof(float);
__device__ __forceinline__ int step_length(const HyperSolve& p) { return p.stages * (int)p.stage_floats + kScalarFloats; }
__device__ __forceinline__ void load_step(const HyperSolve& p, int step, float* dst) {
    const int n = p.stages * (int)p.stage_floats;
    const float* src = p.table + (long long)step * RK_MAX_STAGES * p.stage_floats;
    const float* sc = (const float*)(p.scal + step);
    for (int i = threadIdx.x; i < n + kScalarFloats; i += blockDim.x) cp_async4(dst + i, i < n ? src + i : sc + i - n);
}

// ---------------------------------------------------------------- one stage of one sample, by one warp
// ws: W [w][d], b [w], U [w][d], c [w] (shared memory); units: the sample's rounded units [w] (shared memory, or null)
template <typename T, int DC>
__device__ __forceinline__ void hyper_stage(const float* ws, int w, int d_rt, int lane, const float* z, T* units, float* k, float& kl) {
    constexpr int DM = DC > 0 ? DC : HYPER_MAX_D;
    const int d = DC > 0 ? DC : d_rt;
    const float* W = ws;
    const float* bb = ws + w * d;
    const float* U = bb + w;
    const float* c = U + w * d;
    float v[DM], tr = 0.f;
#pragma unroll
    for (int i = 0; i < DM; ++i) v[i] = 0.f;
#pragma unroll 4
    for (int u = lane; u < w; u += 32) {
        float s = 0.f;
#pragma unroll
        for (int i = 0; i < DM; ++i)
            if (i < d) s = fmaf(W[u * d + i], z[i], s);
        const T aq = Low<T>::from_f(tanhf(s + bb[u]));
        if (units != nullptr) units[u] = aq;
        const float a = Low<T>::to_f(aq);
#pragma unroll
        for (int i = 0; i < DM; ++i)
            if (i < d) v[i] = fmaf(U[u * d + i], a, v[i]);
        tr = fmaf(c[u], 1.f - a * a, tr);
    }
    const float inv_w = 1.f / (float)w;
#pragma unroll
    for (int i = 0; i < DM; ++i) k[i] = i < d ? q16<T>(warp_sum(v[i]) * inv_w) : 0.f;
    kl = q16<T>(-warp_sum(tr) * inv_w);
}

// Y_j = Q16(ybar + sum_{l<j} (h a_jl) k_l)
template <typename T, int DM>
__device__ __forceinline__ void stage_state(const RkStepScalars& sc, int j, const float* y0, const float (*K)[DM], float* z) {
#pragma unroll
    for (int i = 0; i < DM; ++i) {
        float acc = y0[i];
#pragma unroll
        for (int l = 0; l < RK_MAX_STAGES; ++l)
            if (l < j && sc.a[j][l] != 0.f) acc = fmaf(sc.ha[j][l], K[l][i], acc);
        z[i] = j == 0 ? y0[i] : q16<T>(acc);
    }
}

template <typename T, int DC>
__global__ void __launch_bounds__(256) hyper_solve_forward_kernel(HyperSolve p) {
    constexpr int DM = DC > 0 ? DC : HYPER_MAX_D;
    const int d = DC > 0 ? DC : p.d;
    extern __shared__ float sm[];                     // two steps' stage blocks and scalars
    const int sf = (int)p.stage_floats, step_floats = step_length(p);
    const int lane = threadIdx.x & 31;
    const int smp = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const bool on = smp < p.B;
    const int b = on ? smp : p.B - 1;
    auto load = [&](int step) { load_step(p, step, sm + (step & 1) * step_floats); };
    load(0);
    T* traj = (T*)p.traj;
    float y[DM], ybar[DM], l = 0.f;
#pragma unroll
    for (int i = 0; i < DM; ++i) {
        y[i] = i < d ? p.y0[(long long)b * d + i] : 0.f;
        const T q = Low<T>::from_f(y[i]);
        if (i < d && on && lane == 0) traj[(long long)b * d + i] = q;
        ybar[i] = Low<T>::to_f(q);
    }
    for (int n = 0; n < p.n_steps; ++n) {
        cp_async_wait_all();
        __syncthreads();                              // this step's sets have landed, everybody is done with the other buffer
        if (n + 1 < p.n_steps) load(n + 1);
        const RkStepScalars& sc = *(const RkStepScalars*)(sm + (n & 1) * step_floats + p.stages * sf);
        float K[RK_MAX_STAGES][DM], KL[RK_MAX_STAGES];
#pragma unroll
        for (int j = 0; j < RK_MAX_STAGES; ++j) {
            if (j < p.stages) {
                float z[DM];
                stage_state<T, DM>(sc, j, ybar, K, z);
                hyper_stage<T, DC>(sm + (n & 1) * step_floats + j * sf + 2 * p.h, p.w, d, lane, z, (T*)nullptr, K[j], KL[j]);
            }
        }
        float acc_l = 0.f;
#pragma unroll
        for (int i = 0; i < DM; ++i) {
            float acc = 0.f;
#pragma unroll
            for (int j = 0; j < RK_MAX_STAGES; ++j)
                if (j < p.stages) acc = fmaf(sc.hb[j], K[j][i], acc);
            y[i] += p.round_increment ? sc.h * q16<T>(acc) : acc;
            const T q = Low<T>::from_f(y[i]);
            if (i < d && on && lane == 0) traj[((long long)(n + 1) * p.B + b) * d + i] = q;
            ybar[i] = Low<T>::to_f(q);
        }
#pragma unroll
        for (int j = 0; j < RK_MAX_STAGES; ++j)
            if (j < p.stages) acc_l = fmaf(sc.hb[j], KL[j], acc_l);
        l += p.round_increment ? sc.h * q16<T>(acc_l) : acc_l;
    }
    if (on && lane == 0) {
#pragma unroll
        for (int i = 0; i < DM; ++i)
            if (i < d) p.yT[(long long)b * (d + 1) + i] = y[i];
        p.yT[(long long)b * (d + 1) + d] = l;
    }
}

// ---------------------------------------------------------------- grid barrier (cooperative launch), in two halves
// Everything the block wrote before arrive() is visible to every block that has passed wait().  Bounded: a wait that gives up raises
// the error word and returns false, and so does every later one.  Its block leaves without committing; the others may have passed (it had
// arrived), so it is the error word that says whether the pass is good.
__device__ __forceinline__ void grid_arrive(unsigned* counter) {
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(counter, 1u);
    }
}
__device__ __forceinline__ bool grid_wait(unsigned* counter, unsigned target, unsigned* err, unsigned long long limit_ns) {
    bool ok = true;
    if (threadIdx.x == 0) {
        unsigned it = 0;
        const unsigned long long t0 = tc::globaltimer_ns();
        while (tc::ld_acquire_gpu(counter) < target) {
            if ((++it & 255u) == 0u && (tc::globaltimer_ns() - t0 > limit_ns || *(volatile unsigned*)err != 0u)) {
                atomicOr(err, 1024u);
                ok = false;
                break;
            }
        }
        __threadfence();
    }
    return __syncthreads_and(ok) != 0;
}

__device__ __forceinline__ int initial_exponent(float m, int pbits) {
    if (m == 0.f) return 0;
    int E;
    const float f = frexpf(m, &E);
    const int e = pbits - ((f > 0.5f) ? E : E - 1);
    return e < -100 ? -100 : (e > 100 ? 100 : e);
}

constexpr int kMaxKept = 64;                                     // hidden widths up to this keep the second layer in shared memory
// the last layer's row of entry r of weight set u (W_u, b_u, U_u)
__device__ __forceinline__ int set_row(int u, int r, int w, int d) { return r < d ? u * d + r : (r == d ? w * d + u : w * d + w + u * d + r - d - 1); }

// Device words: [0] barrier counter, [1] error, [2 .. 5] flag of attempt n in word 2 + n % 4, [6 .. 9] ||a||_inf likewise
template <typename T, int DC>
__global__ void __launch_bounds__(512) hyper_solve_backward_kernel(HyperSolve p) {
    constexpr int DM = DC > 0 ? DC : HYPER_MAX_D;
    const int d = DC > 0 ? DC : p.d, D = d + 1;
    const int s = p.stages, h = p.h, w = p.w, nv = 2 * d + 2, m = w * (2 * d + 1);
    const int sf = (int)p.stage_floats, step_floats = step_length(p);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    const int G = (int)gridDim.x, groups = (p.B + warps - 1) / warps;
    const Offsets o = offsets(h, m);
    extern __shared__ float sm[];
    float* sets = sm;                                            // two steps' [stages][stage_floats] and scalars
    float* zs = sets + 2 * step_floats;                          // [2][stages][warps][d] stage inputs
    float* kz = zs + 2 * s * warps * d;                          // [stages][warps][d] stage cotangents
    float* kl = kz + s * warps * d;                              // [stages][warps]
    float* red = kl + s * warps;                                 // [warps][stages * nv]
    float* tot = red + warps * s * nv;                           // [stages * nv]
    float* ob = tot + s * nv;                                    // [stages * (2 d + 1)]
    float* hb = ob + s * (2 * d + 1);                            // h2bar [stages][h], h1bar [stages][h]
    float* tred = hb + 2 * s * h;                                // [blockDim]
    float* A2q = tred + blockDim.x;                              // Q16 of the second layer [h][h], where it is small
    float* A3q = A2q + (h <= kMaxKept ? h * h : 0);              // Q16 of the last layer's rows of weight set blockIdx.x [2 d + 1][h]
    T* ua = (T*)(A3q + (2 * d + 1) * h);                         // [2][stages][warps][w] units
    T* us = ua + (size_t)2 * s * warps * w;                      // [stages][warps][w] unit cotangents
    const T* traj = (const T*)p.traj;
    const bool dynamic = p.scaling == MPODE_SCALE_DYNAMIC, checked = p.scaling != MPODE_SCALE_NONE;
    const float inv_w = 1.f / (float)w;
    unsigned* counter = p.words;
    unsigned* err = p.words + 1;
    unsigned arrived = 0;                                        // barriers so far; the counter's target is that times G
    auto load = [&](int step) { load_step(p, step, sets + (step & 1) * step_floats); };
    auto scalars = [&](int step) -> const RkStepScalars& { return *(const RkStepScalars*)(sets + (step & 1) * step_floats + s * sf); };
    // the stages of step n for the samples of group g (Alg. 2, recompute): units and stage inputs into buffer n % 2
    auto recompute = [&](int n, int g) {
        const int smp = g * warps + warp, b = smp < p.B ? smp : p.B - 1;
        const RkStepScalars& sc = scalars(n);
        float y0[DM], K[RK_MAX_STAGES][DM], kl_unused;
#pragma unroll
        for (int i = 0; i < DM; ++i) y0[i] = i < d ? Low<T>::to_f(traj[((long long)n * p.B + b) * d + i]) : 0.f;
#pragma unroll
        for (int j = 0; j < RK_MAX_STAGES; ++j) {
            if (j < s) {
                float z[DM];
                stage_state<T, DM>(sc, j, y0, K, z);
                if (lane < d) {
                    float zl = z[0];
#pragma unroll
                    for (int i = 1; i < DM; ++i) zl = lane == i ? z[i] : zl;
                    zs[(((n & 1) * s + j) * warps + warp) * d + lane] = zl;
                }
                hyper_stage<T, DC>(sets + (n & 1) * step_floats + j * sf + 2 * h, w, d, lane, z, ua + ((size_t)((n & 1) * s + j) * warps + warp) * w,
                                   K[j], kl_unused);
            }
        }
    };

    // Alg. 2 initialisation: a <- dL/dy_N, g <- 0 (or the caller's partial), the initial scale
    bool bad = false;
    float amax = 0.f;
    for (int g = blockIdx.x; g < groups; g += G) {
        const int b = g * warps + warp;
        if (b < p.B && lane < D) {
            const float x = p.dLdyT[(long long)b * D + lane];
            p.a[(long long)b * D + lane] = x;
            bad |= Low<float>::nonfinite(x);
            amax = fmaxf(amax, fabsf(x));
        }
    }
    const long long P = (long long)o.c3 + m;
    if (!p.accumulate)
        for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < P; i += (long long)G * blockDim.x) p.g[i] = 0.f;
    // flag and norm of this attempt for everybody: called by all threads
    auto publish = [&](int slot, bool my_bad, float my_max) {
        warp_flag_or(p.words + 2 + slot, my_bad);
#pragma unroll
        for (int q = 16; q > 0; q >>= 1) my_max = fmaxf(my_max, __shfl_xor_sync(0xffffffffu, my_max, q));
        if (lane == 0 && my_max > 0.f) atomicMax(p.words + 6 + slot, __float_as_uint(my_max));      // non-negative floats order like their bits
    };
    if (h <= kMaxKept)
        for (int i = threadIdx.x; i < h * h; i += blockDim.x) A2q[i] = q16<T>(p.theta[o.A2 + i]);
    if ((int)blockIdx.x < w)
        for (int i = threadIdx.x; i < (2 * d + 1) * h; i += blockDim.x) A3q[i] = q16<T>(p.theta[o.A3 + (long long)set_row(blockIdx.x, i / h, w, d) * h + i % h]);
    int att = 0;                                                 // attempts so far; attempt 0 is the initialisation
    load(p.n_steps - 1);
    publish(0, bad, (amax <= 3.4028234e38f) ? amax : 0.f);
    grid_arrive(counter);
    ++arrived;
    if (!grid_wait(counter, arrived * G, err, p.wait_ns)) {
        if (blockIdx.x == 0 && threadIdx.x == 0) p.status[0] = MPODE_ERR_CUDA;
        return;
    }
    int e = p.e0;
    if (dynamic) {
        if (*(volatile unsigned*)(p.words + 2) != 0u) {
            if (blockIdx.x == 0 && threadIdx.x == 0) p.status[0] = MPODE_ERR_NONFINITE_INPUT;
            return;
        }
        if (p.e0_from_norm) e = initial_exponent(__uint_as_float(*(volatile unsigned*)(p.words + 6)), p.pbits);
    }

    int have_step = -1, have_group = -1;                         // whose units the step's buffers hold
    int next_step = -1;                                          // the step whose stages were recomputed ahead
    int retries = 0;
    bool overflow_seen = dynamic ? false : (*(volatile unsigned*)(p.words + 2) != 0u);
    const int k_lim = dynamic ? p.k_max : 1;
    for (int n = p.n_steps - 1; n >= 0; --n) {
        const RkStepScalars& sc = scalars(n);
        const int par = n & 1;
        cp_async_wait_all();
        __syncthreads();
        const float* set0 = sets + par * step_floats;
        int k_try = 0;
        bool accepted = false;
        float new_max = 0.f;
        while (k_try < k_lim) {
            ++k_try;
            ++att;
            const int slot = att & 3;
            bad = false;
            amax = 0.f;
            // ------------------------------------------------ group phase
            for (int g = blockIdx.x; g < groups; g += G) {
                __syncthreads();                                 // the group before is done with the buffers
                if (have_step != n || have_group != g) recompute(n, g);
                have_step = n; have_group = g;
                const int smp = g * warps + warp;
                const bool on = smp < p.B;
                const int b = on ? smp : p.B - 1;
                float vz[DM], psi[RK_MAX_STAGES][DM], al[DM];
#pragma unroll
                for (int i = 0; i < DM; ++i) {
                    al[i] = (on && i < d) ? p.a[(long long)b * D + i] : 0.f;
                    vz[i] = q16<T>(ldexpf(al[i], e));
                    bad |= q_bad<T>(vz[i]);
                }
                const float a_l = on ? p.a[(long long)b * D + d] : 0.f;
                const float vl = q16<T>(ldexpf(a_l, e));
                bad |= q_bad<T>(vl);
#pragma unroll
                for (int jr = 0; jr < RK_MAX_STAGES; ++jr) {
                    const int j = s - 1 - jr;
                    if (j >= 0) {
                        float kj[DM], ps[DM];
#pragma unroll
                        for (int i = 0; i < DM; ++i) {
                            float acc = sc.b[j] * vz[i];
#pragma unroll
                            for (int l = 0; l < RK_MAX_STAGES; ++l) {      // psi is kept by position: psi[q] belongs to stage s - 1 - q
                                const int st = s - 1 - l;
                                if (l < jr && sc.a[st][j] != 0.f) acc = fmaf(sc.ha[st][j], psi[l][i], acc);
                            }
                            kj[i] = i < d ? q16<T>(acc) : 0.f;
                            bad |= q_bad<T>(kj[i]);
                            ps[i] = 0.f;
                        }
                        const float klj = q16<T>(sc.b[j] * vl);
                        bad |= q_bad<T>(klj);
                        if (lane < d) {
                            float kv = kj[0];
#pragma unroll
                            for (int i = 1; i < DM; ++i) kv = lane == i ? kj[i] : kv;
                            kz[(j * warps + warp) * d + lane] = kv;
                        }
                        if (lane == 0) kl[j * warps + warp] = klj;
                        const float* W = set0 + j * sf + 2 * h;
                        const float* U = W + w * d + w;
                        const float* c = U + w * d;
                        const T* A = ua + ((size_t)(par * s + j) * warps + warp) * w;
                        T* Sb = us + ((size_t)j * warps + warp) * w;
#pragma unroll 4
                        for (int u = lane; u < w; u += 32) {
                            const float a = Low<T>::to_f(A[u]);
                            float ku = 0.f;
#pragma unroll
                            for (int i = 0; i < DM; ++i)
                                if (i < d) ku = fmaf(kj[i], U[u * d + i], ku);
                            // l' = -tr: the trace's unit derivative -2 a c_j / w meets the cotangent -kappa_l
                            const float abar = fmaf(klj * (2.f * inv_w) * c[u], a, ku * inv_w);
                            const T sq = Low<T>::from_f(on ? abar * (1.f - a * a) : 0.f);
                            bad |= Low<T>::nonfinite(sq);
                            Sb[u] = sq;
                            const float sbar = Low<T>::to_f(sq);
#pragma unroll
                            for (int i = 0; i < DM; ++i)
                                if (i < d) ps[i] = fmaf(sbar, W[u * d + i], ps[i]);
                        }
#pragma unroll
                        for (int i = 0; i < DM; ++i) {
                            psi[jr][i] = i < d ? q16<T>(warp_sum(ps[i])) : 0.f;
                            bad |= q_bad<T>(psi[jr][i]);
                        }
                    }
                }
                // the adjoint this attempt would leave; taken over when the attempt is accepted
                if (on) {
                    const float coef = ldexpf(sc.h, -e);
#pragma unroll
                    for (int i = 0; i < DM; ++i) {
                        if (i < d) {
                            float da = 0.f;
#pragma unroll
                            for (int q = 0; q < RK_MAX_STAGES; ++q)
                                if (q < s) da += psi[q][i];
                            float an = fmaf(coef, da, al[i]);
                            if (p.cot != nullptr) an += p.cot[((long long)n * p.B + b) * D + i];
                            amax = fmaxf(amax, fabsf(an));
                            if (lane == i) p.a_new[(long long)b * D + i] = an;
                        }
                    }
                    const float aln = a_l + (p.cot != nullptr ? p.cot[((long long)n * p.B + b) * D + d] : 0.f);
                    amax = fmaxf(amax, fabsf(aln));
                    if (lane == d) p.a_new[(long long)b * D + d] = aln;
                }
                __syncthreads();
                // this group's share of every weight set's cotangents: Wbar = sum sbar z, bbar = sum sbar, Ubar = sum a kappa_z / w,
                // cbar = -sum kappa_l (1 - a^2) / w, samples in ascending order
                const int n_smp = min(warps, p.B - g * warps);
                const bool first = g == (int)blockIdx.x;
                for (int q = threadIdx.x; q < s * w; q += blockDim.x) {
                    const int j = q / w, u = q - j * w;
                    float acc[2 * DM + 2];
#pragma unroll
                    for (int i = 0; i < 2 * DM + 2; ++i) acc[i] = 0.f;
#pragma unroll 4
                    for (int r = 0; r < n_smp; ++r) {
                        const float a = Low<T>::to_f(ua[((size_t)(par * s + j) * warps + r) * w + u]);
                        const float sbar = Low<T>::to_f(us[((size_t)j * warps + r) * w + u]);
                        const float* zr = zs + ((par * s + j) * warps + r) * d;
                        const float* kr = kz + (j * warps + r) * d;
                        if constexpr (DC == 2) {
                            const float2 z2 = *reinterpret_cast<const float2*>(zr), k2 = *reinterpret_cast<const float2*>(kr);
                            acc[0] = fmaf(sbar, z2.x, acc[0]); acc[1] = fmaf(sbar, z2.y, acc[1]);
                            acc[DM + 1] = fmaf(a * inv_w, k2.x, acc[DM + 1]); acc[DM + 2] = fmaf(a * inv_w, k2.y, acc[DM + 2]);
                        } else {
#pragma unroll
                            for (int i = 0; i < DM; ++i)
                                if (i < d) {
                                    acc[i] = fmaf(sbar, zr[i], acc[i]);
                                    acc[DM + 1 + i] = fmaf(a * inv_w, kr[i], acc[DM + 1 + i]);
                                }
                        }
                        acc[DM] += sbar;
                        acc[2 * DM + 1] = fmaf(-kl[j * warps + r] * inv_w, 1.f - a * a, acc[2 * DM + 1]);
                    }
                    float* dst = p.part + (((long long)blockIdx.x * w + u) * s + j) * nv;
#pragma unroll
                    for (int i = 0; i < 2 * DM + 2; ++i) {
                        const int dense = i < DM ? i : (i == DM ? d : (i <= 2 * DM ? d + 1 + (i - DM - 1) : 2 * d + 1));
                        const bool used = i < DM ? i < d : (i == DM || i == 2 * DM + 1 || i - DM - 1 < d);
                        if (used) dst[dense] = first ? acc[i] : dst[dense] + acc[i];
                    }
                }
            }
            publish(slot, bad && checked, amax);
            grid_arrive(counter);
            ++arrived;
            if (n > 0) {                                         // the step before, while the others arrive
                if (k_try == 1) load(n - 1);
                if (groups <= G && (int)blockIdx.x < groups && next_step != n - 1) {
                    cp_async_wait_all();
                    __syncthreads();
                    recompute(n - 1, blockIdx.x);
                    next_step = n - 1;
                }
            }
            bool alive = grid_wait(counter, arrived * G, err, p.wait_ns);
            // ------------------------------------------------ set phase: weight sets blockIdx.x, blockIdx.x + G, ...
            bool bad2 = false;
            if (alive) {
                for (int u = blockIdx.x; u < w; u += G) {
                    for (int v0 = lane; v0 < s * nv; v0 += 32) {
                        float x = 0.f;
                        const int nb = groups < G ? groups : G;   // blocks that hold samples
#pragma unroll 16
                        for (int r = warp; r < nb; r += warps) x += __ldcg(p.part + ((long long)r * w + u) * s * nv + v0);
                        red[warp * s * nv + v0] = x;
                    }
                    __syncthreads();
                    for (int v0 = threadIdx.x; v0 < s * nv; v0 += blockDim.x) {
                        float x = 0.f;
                        for (int r = 0; r < warps; ++r) x += red[r * s * nv + v0];
                        tot[v0] = x;
                    }
                    __syncthreads();
                    for (int q = threadIdx.x; q < s * (2 * d + 1); q += blockDim.x) {      // the chain rule through c = U . W, then one rounding
                        const int j = q / (2 * d + 1), r = q - j * (2 * d + 1);
                        const float* W = set0 + j * sf + 2 * h;
                        const float* U = W + w * d + w;
                        const float* t = tot + j * nv;
                        const float cbar = t[2 * d + 1];
                        float v = r < d ? fmaf(cbar, U[u * d + r], t[r]) : (r == d ? t[d] : fmaf(cbar, W[u * d + r - d - 1], t[r]));
                        v = q16<T>(v);
                        bad2 |= q_bad<T>(v);
                        ob[q] = v;
                    }
                    __syncthreads();
                    // their part of the cotangent of h2, then the gradient of the last layer's rows that belong to weight set u
                    const bool kept = u == (int)blockIdx.x;
                    for (int q = threadIdx.x; q < s * h; q += blockDim.x) {
                        const int j = q / h, k = q - j * h;
                        float t = 0.f;
                        for (int r = 0; r < 2 * d + 1; ++r)
                            t = fmaf(kept ? A3q[r * h + k] : q16<T>(p.theta[o.A3 + (long long)set_row(u, r, w, d) * h + k]), ob[j * (2 * d + 1) + r], t);
                        p.tpart[(long long)u * s * h + q] = t;
                    }
                    for (int q = threadIdx.x; q < (2 * d + 1) * (h + 1); q += blockDim.x) {
                        const int r = q / (h + 1), k = q - r * (h + 1), row = set_row(u, r, w, d);
                        float x = 0.f;
                        for (int j = s - 1; j >= 0; --j) x = k < h ? fmaf(ob[j * (2 * d + 1) + r], set0[j * sf + h + k], x) : x + ob[j * (2 * d + 1) + r];
                        bad2 |= q_bad<T>(q16<T>(x));
                        p.dg[k < h ? o.A3 + (long long)row * h + k : o.c3 + row] = x;
                    }
                    __syncthreads();
                }
                warp_flag_or(p.words + 2 + slot, bad2 && checked);
            }
            grid_arrive(counter);
            ++arrived;
            const unsigned extra = p.starve && n == 0 && (int)blockIdx.x == G - 1 ? 1u : 0u;      // test: an arrival that never comes
            alive = grid_wait(counter, arrived * G + extra, err, p.wait_ns) && alive;
            if (!alive) {
                if (blockIdx.x == 0 && threadIdx.x == 0) p.status[0] = MPODE_ERR_CUDA;
                return;
            }
            if (blockIdx.x == 0 && threadIdx.x == 0) { p.words[2 + ((att + 2) & 3)] = 0u; p.words[6 + ((att + 2) & 3)] = 0u; }
            // ------------------------------------------------ the two hidden layers backwards, in every block
            bool bad3 = false;
            {
                const int sh = s * h, parts = sh <= (int)blockDim.x ? (int)blockDim.x / sh : 1;
                for (int q0 = 0; q0 < sh; q0 += blockDim.x) {
                    const int q = q0 + (int)threadIdx.x % min(sh, (int)blockDim.x), pc = (int)threadIdx.x / min(sh, (int)blockDim.x);
                    float t = 0.f;
                    if (q < sh && pc < parts) {
#pragma unroll 32
                        for (int u = pc; u < w; u += parts) t += __ldcg(p.tpart + (long long)u * sh + q);
                    }
                    __syncthreads();
                    tred[threadIdx.x] = t;
                    __syncthreads();
                    if (pc == 0 && q < sh) {
                        float x = 0.f;
                        for (int r = 0; r < parts; ++r) x += tred[r * min(sh, (int)blockDim.x) + q - q0];
                        const int j = q / h, k = q - j * h;
                        const float h2 = set0[j * sf + h + k];
                        const float v = q16<T>((1.f - h2 * h2) * x);
                        bad3 |= q_bad<T>(v);
                        hb[q] = v;
                    }
                }
                __syncthreads();
                for (int q = threadIdx.x; q < sh; q += blockDim.x) {
                    const int j = q / h, l = q - j * h;
                    float t = 0.f;
#pragma unroll 8
                    for (int k = 0; k < h; ++k) t = fmaf(h <= kMaxKept ? A2q[k * h + l] : q16<T>(p.theta[o.A2 + k * h + l]), hb[j * h + k], t);
                    const float h1 = set0[j * sf + l];
                    const float v = q16<T>((1.f - h1 * h1) * t);
                    bad3 |= q_bad<T>(v);
                    hb[sh + q] = v;
                }
                __syncthreads();
                // Gradients of A2 | c2 | A1 | c1, stages added last to first: block 0 forms them.  Are their roundings finite?  Every entry
                // is at most sum_j max |hbar_j| max(1, |tau_j|) (h1 and h2 lie in [-1, 1]); only if that bound does not fit the format do
                // the other blocks look at the entries too.
                float bound = 0.f;
                for (int j = 0; j < s; ++j) {
                    float m1 = 0.f;
                    for (int k = lane; k < h; k += 32) m1 = fmaxf(m1, fmaxf(fabsf(hb[j * h + k]), fabsf(hb[sh + j * h + k])));
#pragma unroll
                    for (int q = 16; q > 0; q >>= 1) m1 = fmaxf(m1, __shfl_xor_sync(0xffffffffu, m1, q));
                    bound += m1 * fmaxf(1.f, fabsf(sc.tau16[j]));
                }
                if (blockIdx.x == 0 || q_bad<T>(q16<T>(2.f * bound))) {
                    for (int q = threadIdx.x; q < h * h + 3 * h; q += blockDim.x) {
                        float x = 0.f;
                        int at;
                        if (q < h * h) {
                            const int k = q / h, l = q - k * h;
                            for (int j = s - 1; j >= 0; --j) x = fmaf(hb[j * h + k], set0[j * sf + l], x);
                            at = o.A2 + q;
                        } else {
                            const int k = (q - h * h) % h, what = (q - h * h) / h;
                            for (int j = s - 1; j >= 0; --j) x = what == 1 ? fmaf(hb[sh + j * h + k], sc.tau16[j], x) : x + hb[(what == 0 ? 0 : sh) + j * h + k];
                            at = what == 0 ? o.c2 + k : (what == 1 ? o.A1 + k : o.c1 + k);
                        }
                        bad3 |= q_bad<T>(q16<T>(x));
                        if (blockIdx.x == 0) p.dg[at] = x;
                    }
                }
            }
            const bool any_bad = __syncthreads_or(checked && (bad3 || *(volatile unsigned*)(p.words + 2 + slot) != 0u)) != 0;
            new_max = __uint_as_float(*(volatile unsigned*)(p.words + 6 + slot));
            if (!dynamic) overflow_seen |= any_bad;
            if (!dynamic || !any_bad) { accepted = true; break; }
            if (e > -100) --e;                                   // halve and retry
            ++retries;
        }
        if (blockIdx.x == 0 && threadIdx.x == 0) { p.log_exp[n] = e; p.log_attempts[n] = k_try; p.log_doubled[n] = 0; }
        if (!accepted) {
            if (blockIdx.x == 0 && threadIdx.x == 0) { p.status[0] = MPODE_ERR_SCALE_FAILED; p.status[1] = n; p.status[2] = retries; }
            return;
        }
        // high-precision updates with h / S: each thread takes back what it wrote itself
        const float coef = ldexpf(sc.h, -e);
        for (int g = blockIdx.x; g < groups; g += G) {
            const int b = g * warps + warp;
            if (b < p.B && lane < D) p.a[(long long)b * D + lane] = p.a_new[(long long)b * D + lane];
        }
        __syncwarp();                                            // a row is read by the whole warp next
        for (int u = blockIdx.x; u < w; u += G)
            for (int q = threadIdx.x; q < (2 * d + 1) * (h + 1); q += blockDim.x) {
                const int r = q / (h + 1), k = q - r * (h + 1);
                const int row = set_row(u, r, w, d);
                const long long at = k < h ? o.A3 + (long long)row * h + k : o.c3 + row;
                p.g[at] = fmaf(coef, p.dg[at], p.g[at]);
            }
        if (blockIdx.x == 0)
            for (int q = threadIdx.x; q < h * h + 3 * h; q += blockDim.x) {
                const int k = (q - h * h) % h, what = (q - h * h) / h;
                const int at = q < h * h ? o.A2 + q : (what == 0 ? o.c2 + k : (what == 1 ? o.A1 + k : o.c1 + k));
                p.g[at] = fmaf(coef, p.dg[at], p.g[at]);
            }
        if (n > 0 && next_step == n - 1) { have_step = n - 1; have_group = blockIdx.x; }
        if (dynamic && k_try == 1) {                             // growth test
            const double scaled = p.growth_rule == 0 ? ldexp((double)new_max, e) : (double)new_max;
            if (scaled <= ldexp(1.0, p.pbits - 1) && e < 100) {
                ++e;
                if (blockIdx.x == 0 && threadIdx.x == 0) p.log_doubled[n] = 1;
            }
        }
    }
    if (p.scaling == MPODE_SCALE_NONE_SAFE && overflow_seen) {   // Sec. 5: report the overflow through infinite gradients
        for (int g = blockIdx.x; g < groups; g += G) {
            const int b = g * warps + warp;
            if (b < p.B && lane < D) p.a[(long long)b * D + lane] = INFINITY;
        }
        for (int u = blockIdx.x; u < w; u += G)
            for (int q = threadIdx.x; q < (2 * d + 1) * (h + 1); q += blockDim.x) {
                const int r = q / (h + 1), k = q - r * (h + 1);
                const int row = set_row(u, r, w, d);
                p.g[k < h ? o.A3 + (long long)row * h + k : o.c3 + row] = INFINITY;
            }
        if (blockIdx.x == 0) {
            for (int q = threadIdx.x; q < o.A3; q += blockDim.x) p.g[q] = INFINITY;
            if (threadIdx.x == 0) p.status[0] = MPODE_WARN_NONFINITE_GRAD;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) p.status[2] = retries;
}

size_t backward_smem(mpode_dtype dt, int stages, int h, int w, int d, int warps) {
    const size_t sf = hyper_stage_floats(h, w, d), s = stages, nv = 2 * d + 2;
    const size_t fl = 2 * (s * sf + kScalarFloats) + 3 * s * warps * d + s * warps + warps * s * nv + s * nv + s * (2 * d + 1) + 2 * s * h + 32 * (size_t)warps + (h <= kMaxKept ? (size_t)h * h : 0) + (2 * d + 1) * (size_t)h;
    return fl * sizeof(float) + 3 * s * warps * w * low_size(dt);
}
constexpr size_t kSmemCap = 200 * 1024;

// samples a block takes at a time (one warp each): eight while that gives at most a block per SM, else sixteen; fewer where the
// units of so many samples do not fit shared memory
int backward_warps(mpode_dtype dt, int B, int stages, int h, int w, int d) {
    int warps = B > 8 * sm_count() ? 16 : 8;
    while (warps > 1 && backward_smem(dt, stages, h, w, d, warps) > kSmemCap) warps /= 2;
    return warps;
}

}  // namespace

bool hyper_solve_shape_ok(mpode_dtype dt, int h, int w, int d, int stages) {
    return hyper_shape_ok(h, w, d) && stages >= 1 && stages <= RK_MAX_STAGES && backward_smem(dt, stages, h, w, d, 1) <= kSmemCap;
}
// a row of partial sums for every block that holds samples (the fewer samples a block takes, the more of them: four stages need the most room)
size_t hyper_solve_part_floats(mpode_dtype dt, int B, int h, int w, int d) {
    const int warps = backward_warps(dt, B, RK_MAX_STAGES, h, w, d), groups = (B + warps - 1) / warps;
    return (size_t)(groups < sm_count() ? groups : sm_count()) * w * RK_MAX_STAGES * (2 * d + 2);
}
size_t hyper_solve_tpart_floats(int h, int w) { return (size_t)w * RK_MAX_STAGES * h; }

void launch_hyper_table(mpode_dtype dt, const float* theta, const RkStepScalars* scal, int n_steps, int stages, int h, int w, int d, float* table,
                        cudaStream_t st, long long* launches) {
    const size_t smem = (size_t)2 * RK_MAX_STAGES * h * sizeof(float);
    MPODE_DISPATCH_T(dt, T, (hyper_table_kernel<T><<<n_steps, 256, smem, st>>>(theta, scal, stages, h, w, d, table, (long long)hyper_stage_floats(h, w, d))));
    if (launches) ++*launches;
}

template <typename T, int DC>
static bool solve_forward_t(const HyperSolve& p, cudaStream_t st) {
    static bool attr[kMaxDevices] = {false};
    const int dev = current_device();
    if (!attr[dev]) {
        if (cudaFuncSetAttribute(hyper_solve_forward_kernel<T, DC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemCap) != cudaSuccess) return false;
        attr[dev] = true;
    }
    const size_t smem = 2 * ((size_t)p.stages * p.stage_floats + kScalarFloats) * sizeof(float);
    hyper_solve_forward_kernel<T, DC><<<(p.B + 7) / 8, 256, smem, st>>>(p);
    return true;
}

template <typename T, int DC>
static bool solve_backward_t(mpode_dtype dt, const HyperSolve& p, cudaStream_t st) {
    static bool attr[kMaxDevices] = {false};
    const int dev = current_device();
    if (!attr[dev]) {
        if (cudaFuncSetAttribute(hyper_solve_backward_kernel<T, DC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemCap) != cudaSuccess) return false;
        attr[dev] = true;
    }
    const int warps = backward_warps(dt, p.B, p.stages, p.h, p.w, p.d);
    const int groups = (p.B + warps - 1) / warps;
    // every weight set has an owner block: no more blocks than SMs (all resident: cooperative launch), and enough for the sets
    int blocks = groups > p.w ? groups : p.w;
    if (blocks > sm_count()) blocks = sm_count();
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3((unsigned)(32 * warps));
    cfg.dynamicSmemBytes = backward_smem(dt, p.stages, p.h, p.w, p.d, warps);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, hyper_solve_backward_kernel<T, DC>, p) == cudaSuccess;
}

bool launch_hyper_solve_forward(mpode_dtype dt, const HyperSolve& p, cudaStream_t st, long long* launches) {
    bool ok = false;
    if (p.d == 2) { MPODE_DISPATCH_T(dt, T, (ok = solve_forward_t<T, 2>(p, st))); }
    else { MPODE_DISPATCH_T(dt, T, (ok = solve_forward_t<T, 0>(p, st))); }
    if (ok && launches) ++*launches;
    return ok;
}

bool launch_hyper_solve_backward(mpode_dtype dt, const HyperSolve& p, cudaStream_t st, long long* launches) {
    bool ok = false;
    if (p.d == 2) { MPODE_DISPATCH_T(dt, T, (ok = solve_backward_t<T, 2>(dt, p, st))); }
    else { MPODE_DISPATCH_T(dt, T, (ok = solve_backward_t<T, 0>(dt, p, st))); }
    if (ok && launches) ++*launches;
    return ok;
}

}  // namespace mpode
