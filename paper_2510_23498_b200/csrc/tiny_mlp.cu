// Whole-solve kernels for very small dense velocities: see tiny_mlp.h.  Arithmetic and rounding points are those of the
// layer-by-layer path: operands rounded to the low format (Q16), products accumulated in fp32, one rounding per layer output /
// cotangent, activation derivatives from the rounded stored output.
//
// What bounds these kernels is the dependent chain of one sample: stages x layers x steps, each a tanh or softplus and a few
// multiply-adds.  Eight lanes share a sample: lane q has the hidden units q, q + 8, ... in registers and the lanes' sums meet in
// three shuffles.  The forward pass has nothing to exchange between samples and spreads over many small blocks.  The backward pass
// is one cluster of up to 16 blocks (the samples of a batch of 1024): per attempt the blocks' parameter sums, overflow flags and
// norms are exchanged through distributed shared memory behind one cluster barrier, and every block adds them up and takes Alg. 2's
// decision itself.  Measured (512 samples, 3 -> 32 -> 2, 10 RK4 steps, fp16 with dynamic scaling, 15 attempts): one block with a
// thread per sample took 457 us forward and 2611 us backward; these take 22 and 125 us.
#include "tiny_mlp.h"

#include <cooperative_groups.h>
#include <math.h>

#include "tensormap.h"

namespace mpode {
namespace {

namespace cg = cooperative_groups;

template <typename T> __device__ __forceinline__ float q16(float x) { return Low<T>::to_f(Low<T>::from_f(x)); }
template <typename T> __device__ __forceinline__ bool q_nonfinite(float rounded) { return Low<T>::nonfinite(Low<T>::from_f(rounded)); }

// sum of two low-format values, rounded once (the exact sum fits a double)
template <typename T> __device__ __forceinline__ float q16_sum(float a, float b);
template <> __device__ __forceinline__ float q16_sum<float>(float a, float b) { return (float)((double)a + (double)b); }
template <> __device__ __forceinline__ float q16_sum<__half>(float a, float b) { return __half2float(__double2half((double)a + (double)b)); }
template <> __device__ __forceinline__ float q16_sum<__nv_bfloat16>(float a, float b) {
    return __bfloat162float(__double2bfloat16((double)a + (double)b));
}

constexpr int kLanes = 8;                        // lanes that share a sample (the scalar example: one)

template <bool POLY> __device__ __forceinline__ float lanes_sum(float x) {
    if (!POLY) {
#pragma unroll
        for (int o = 1; o < kLanes; o <<= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    }
    return x;
}

// Q16(theta) as floats in shared memory, hidden index innermost and padded to 8 UH units with zeros (the eight lanes of a sample read
// eight neighbouring words): W1 [d][hp], time column [hp], b1 [hp], W2 [d][hp], b2 [d]
struct TinyWeights { float *W1, *wt, *b1, *W2, *b2; int hp; };
__host__ __device__ inline int tiny_weight_floats(int d, int hp) { return 2 * d * hp + 2 * hp + d; }

template <typename T, int UH, bool POLY>
__device__ void tiny_load_weights(const TinyParams& p, float* sm, TinyWeights& w) {
    const float* th = p.theta;
    const int hp = kLanes * UH;
    w.hp = hp;
    w.W1 = sm; w.wt = w.W1 + p.d * hp; w.b1 = w.wt + hp; w.W2 = w.b1 + hp; w.b2 = w.W2 + p.d * hp;
    if (POLY) {         // Q16(theta_1..3) at the start of the weight area
        if (threadIdx.x < 3) w.W1[threadIdx.x] = q16<T>(th[threadIdx.x]);
    } else {
        const int in1 = p.d + (p.time ? 1 : 0), n1 = p.h * in1, nb1 = p.bias ? p.h : 0, n2 = p.d * p.h;
        for (int i = threadIdx.x; i < p.d * hp; i += blockDim.x) {
            const int c = i / hp, n = i - c * hp;
            w.W1[i] = n < p.h ? q16<T>(th[n * in1 + c]) : 0.f;
            w.W2[i] = n < p.h ? q16<T>(th[n1 + nb1 + c * p.h + n]) : 0.f;
        }
        for (int n = threadIdx.x; n < hp; n += blockDim.x) {
            w.wt[n] = p.time && n < p.h ? q16<T>(th[n * in1 + p.d]) : 0.f;
            w.b1[n] = nb1 && n < p.h ? q16<T>(th[n1 + n]) : 0.f;
        }
        for (int c = threadIdx.x; c < p.d; c += blockDim.x) w.b2[c] = p.bias ? q16<T>(th[n1 + nb1 + n2 + c]) : 0.f;
    }
    __syncthreads();
}

// A lane's share of the weights: in registers where there are few, else read from shared memory at every use
template <int UH, int DM> struct LaneWeights {
    static constexpr bool kRegs = UH * (2 * DM + 2) <= 24;
    const TinyWeights& w;
    int q;
    float r1[kRegs ? UH : 1][kRegs ? DM : 1], r2[kRegs ? UH : 1][kRegs ? DM : 1], rt[kRegs ? UH : 1], rb[kRegs ? UH : 1];
    __device__ __forceinline__ LaneWeights(const TinyWeights& w_, int q_, int d) : w(w_), q(q_) {
        if constexpr (kRegs) {
#pragma unroll
            for (int i = 0; i < UH; ++i) {
#pragma unroll
                for (int c = 0; c < DM; ++c) {
                    r1[i][c] = c < d ? w.W1[c * w.hp + q + kLanes * i] : 0.f;
                    r2[i][c] = c < d ? w.W2[c * w.hp + q + kLanes * i] : 0.f;
                }
                rt[i] = w.wt[q + kLanes * i];
                rb[i] = w.b1[q + kLanes * i];
            }
        }
    }
    __device__ __forceinline__ float W1(int i, int c) const { if constexpr (kRegs) return r1[i][c]; else return w.W1[c * w.hp + q + kLanes * i]; }
    __device__ __forceinline__ float W2(int i, int c) const { if constexpr (kRegs) return r2[i][c]; else return w.W2[c * w.hp + q + kLanes * i]; }
    __device__ __forceinline__ float wt(int i) const { if constexpr (kRegs) return rt[i]; else return w.wt[q + kLanes * i]; }
    __device__ __forceinline__ float b1(int i) const { if constexpr (kRegs) return rb[i]; else return w.b1[q + kLanes * i]; }
};

// k = f(tau, Y): H = Q16(act(W1 [Y; tau] + b1)) (this lane's units), k = Q16(W2 H + b2) (every lane)
template <typename T, int UH, int DM, bool POLY>
__device__ __forceinline__ void tiny_eval(const TinyParams& p, const LaneWeights<UH, DM>& lw, float tau16, const float (&Y)[DM], float (&H)[UH], float (&k)[DM]) {
    if constexpr (POLY) {       // Example 1, one rounding per operation; lambda and t^2 are kept for the backward pass
        const float t2 = q16<T>(tau16 * tau16);
        const float lam = q16_sum<T>(q16_sum<T>(q16<T>(lw.w.W1[0] * t2), q16<T>(lw.w.W1[1] * tau16)), lw.w.W1[2]);
        H[0] = lam; H[1] = t2;
        k[0] = q16<T>(-lam * Y[0]);
    } else {
#pragma unroll
        for (int c = 0; c < DM; ++c) k[c] = 0.f;
#pragma unroll
        for (int i = 0; i < UH; ++i) {
            float z = 0.f;
#pragma unroll
            for (int c = 0; c < DM; ++c)
                if (c < p.d) z = fmaf(Y[c], lw.W1(i, c), z);
            z = fmaf(tau16, lw.wt(i), z + lw.b1(i));
            H[i] = q16<T>(act_fwd(p.act, z));
#pragma unroll
            for (int c = 0; c < DM; ++c)
                if (c < p.d) k[c] = fmaf(H[i], lw.W2(i, c), k[c]);
        }
#pragma unroll
        for (int c = 0; c < DM; ++c) k[c] = c < p.d ? q16<T>(lanes_sum<POLY>(k[c]) + lw.w.b2[c]) : 0.f;
    }
}

// All stages of one step from the stored low-precision state ybar (Alg. 1 increment / Alg. 2 recompute)
template <typename T, int UH, int DM, bool POLY>
__device__ __forceinline__ void tiny_stages(const TinyParams& p, const LaneWeights<UH, DM>& lw, const RkStepScalars& sc, const float (&ybar)[DM],
                                            float (&Y)[RK_MAX_STAGES][DM], float (&H)[RK_MAX_STAGES][UH], float (&K)[RK_MAX_STAGES][DM]) {
#pragma unroll
    for (int j = 0; j < RK_MAX_STAGES; ++j) {
        if (j < p.stages) {
#pragma unroll
            for (int c = 0; c < DM; ++c) {
                float acc = ybar[c];
#pragma unroll
                for (int l = 0; l < RK_MAX_STAGES; ++l)
                    if (l < j && sc.ha[j][l] != 0.f) acc = fmaf(sc.ha[j][l], K[l][c], acc);
                Y[j][c] = j == 0 ? ybar[c] : q16<T>(acc);
            }
            tiny_eval<T, UH, DM, POLY>(p, lw, sc.tau16[j], Y[j], H[j], K[j]);
        }
    }
}

constexpr int kScalarWords = sizeof(RkStepScalars) / sizeof(float);

template <typename T, int UH, int DM, bool POLY>
__global__ void __launch_bounds__(64) tiny_forward_kernel(TinyParams p) {
    extern __shared__ float sm[];                // weights, then two steps' scalars
    TinyWeights w;
    tiny_load_weights<T, UH, POLY>(p, sm, w);
    float* scs = sm + tiny_weight_floats(p.d, kLanes * UH);
    constexpr int LP = POLY ? 1 : kLanes;
    const int gt = blockIdx.x * blockDim.x + threadIdx.x, smp = gt / LP, q = gt % LP;
    const bool on = smp < p.B;
    const int b = on ? smp : p.B - 1;            // lanes past the batch compute along (the shuffles want whole warps), store nothing
    const LaneWeights<UH, DM> lw(w, q, p.d);
    T* traj = (T*)p.traj;
    float y[DM], ybar[DM], Y[RK_MAX_STAGES][DM], H[RK_MAX_STAGES][UH], K[RK_MAX_STAGES][DM];
#pragma unroll
    for (int c = 0; c < DM; ++c) {
        y[c] = c < p.d ? p.y0[(long long)b * p.d + c] : 0.f;
        const T v = Low<T>::from_f(y[c]);
        if (c < p.d && on && q == 0) traj[(long long)b * p.d + c] = v;
        ybar[c] = Low<T>::to_f(v);
    }
    if (threadIdx.x < kScalarWords) scs[threadIdx.x] = ((const float*)p.scal)[threadIdx.x];
    for (int i = 0; i < p.n_steps; ++i) {
        __syncthreads();
        float next = 0.f;                        // the next step's scalars travel while this step runs
        const bool fetch = i + 1 < p.n_steps && threadIdx.x < kScalarWords;
        if (fetch) next = ((const float*)(p.scal + i + 1))[threadIdx.x];
        const RkStepScalars& sc = *(const RkStepScalars*)(scs + (i & 1) * kScalarWords);
        tiny_stages<T, UH, DM, POLY>(p, lw, sc, ybar, Y, H, K);
#pragma unroll
        for (int c = 0; c < DM; ++c) {
            float acc = 0.f;
#pragma unroll
            for (int j = 0; j < RK_MAX_STAGES; ++j)
                if (j < p.stages) acc = fmaf(sc.hb[j], K[j][c], acc);
            y[c] += p.round_increment ? sc.h * q16<T>(acc) : acc;
            const T v = Low<T>::from_f(y[c]);
            if (c < p.d && on && q == 0) traj[((long long)(i + 1) * p.B + b) * p.d + c] = v;
            ybar[c] = Low<T>::to_f(v);
        }
        if (fetch) scs[((i + 1) & 1) * kScalarWords + threadIdx.x] = next;
    }
    if (on && q == 0) {
#pragma unroll
        for (int c = 0; c < DM; ++c)
            if (c < p.d) p.yT[(long long)b * p.d + c] = y[c];
    }
}

// S_N = 2^floor(-log2(u_L m)) in integer arithmetic (u_L = 2^-pbits, m = f 2^E with f in [0.5, 1))
__device__ __forceinline__ int tiny_initial_exponent(float m, int pbits) {
    if (m == 0.f) return 0;
    int E;
    const float f = frexpf(m, &E);
    const int e = pbits - ((f > 0.5f) ? E : E - 1);
    return e < -100 ? -100 : (e > 100 ? 100 : e);
}

// THREADS: 256 (a batch of up to 512 is a cluster of 16, and a thread has all the registers it wants) or 512
template <typename T, int UH, int DM, bool POLY, int THREADS>
__global__ void __launch_bounds__(THREADS, 1) tiny_backward_kernel(TinyParams p) {
    extern __shared__ float sm[];
    cg::cluster_group cl = cg::this_cluster();
    const int n_ctas = (int)gridDim.x, rank = (int)blockIdx.x;      // one cluster: the whole grid
    TinyWeights w;
    const int in1 = p.d + (p.time ? 1 : 0);
    const int n1 = p.h * in1, nb1 = p.bias ? p.h : 0, n2 = p.d * p.h, nb2 = p.bias ? p.d : 0;
    const int P = POLY ? 3 : n1 + nb1 + n2 + nb2;
    const bool want_dt = p.tprime != nullptr;
    const int P3 = P + (want_dt ? 3 : 0);      // behind the parameters: dt, dh and Phi^T a of the step, summed over the batch alike
    const int o_b1 = n1, o_w2 = n1 + nb1, o_b2 = n1 + nb1 + n2;
    const int nwarps = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float* scs = sm + tiny_weight_floats(p.d, kLanes * UH);            // [2] steps' scalars
    float* part = scs + 2 * kScalarWords;                              // [nwarps][P3] per-warp sums
    float* wmax = part + (size_t)nwarps * P3;                          // [32] per-warp norms
    float* xch = wmax + 32;                                            // [2][P3 + 2] what the blocks exchange: sums, norm, flag
    float* dgs = xch + 2 * (P3 + 2);                                   // [P3 + 2] the sums over all blocks
    tiny_load_weights<T, UH, POLY>(p, sm, w);

    constexpr int LP = POLY ? 1 : kLanes;
    const int gt = blockIdx.x * blockDim.x + threadIdx.x, smp = gt / LP, q = gt % LP;
    const bool active = smp < p.B;
    const int b = active ? smp : p.B - 1;
    const LaneWeights<UH, DM> lw(w, q, p.d);
    const T* traj = (const T*)p.traj;
    const bool dynamic = p.scaling == MPODE_SCALE_DYNAMIC, checked = p.scaling != MPODE_SCALE_NONE;
    // The blocks' norms and flags (and, with `sums`, the parameter sums in `part`) meet: afterwards dgs holds the totals, dgs[P3] the
    // norm, and the return value is whether any flag was raised or a total does not fit the low format.  One cluster barrier: the
    // exchange area alternates, and a block is at the next barrier only after it has read this one.
    int round = 0;
    auto exchange = [&](bool bad, float m, bool sums) -> bool {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (lane == 0) wmax[warp] = m;
        const int blk_bad = __syncthreads_or(bad);
        float* x = xch + (round & 1) * (P3 + 2);
        if (sums)
            for (int i = threadIdx.x; i < P3; i += blockDim.x) {
                float t = 0.f;
                for (int ww = 0; ww < nwarps; ++ww) t += part[(size_t)ww * P3 + i];
                x[i] = t;
            }
        if (threadIdx.x == blockDim.x - 1) {
            float mm = wmax[0];
            for (int ww = 1; ww < nwarps; ++ww) mm = fmaxf(mm, wmax[ww]);
            x[P3] = mm;
            x[P3 + 1] = blk_bad ? 1.f : 0.f;
        }
        cl.sync();
        bool any = false;
        for (int i = (sums ? 0 : P3) + threadIdx.x; i < P3 + 2; i += blockDim.x) {
            float t = 0.f;
#pragma unroll 4
            for (int r = 0; r < n_ctas; ++r) {
                const float v = *cl.map_shared_rank(x + i, r);
                t = i < P3 ? t + v : fmaxf(t, v);
            }
            dgs[i] = t;
            if (i == P3 + 1) any |= t != 0.f;
            else if (i < P + (want_dt ? 2 : 0)) any |= q_nonfinite<T>(q16<T>(t));      // are Q16(dg), Q16(dt), Q16(dh) finite?
        }
        ++round;
        return __syncthreads_or(any) != 0;
    };

    float a[DM];
    bool in_bad = false;
    float amax = 0.f;
#pragma unroll
    for (int c = 0; c < DM; ++c) {
        a[c] = active && c < p.d ? p.dLdyT[(long long)b * p.d + c] : 0.f;
        in_bad |= Low<float>::nonfinite(a[c]);
        amax = fmaxf(amax, fabsf(a[c]));
    }
    int e = p.e0;
    if (dynamic) {
        if (exchange(in_bad, amax, false)) {
            if (rank == 0 && threadIdx.x == 0) p.status[0] = MPODE_ERR_NONFINITE_INPUT;
            cl.sync();
            return;
        }
        if (p.e0_from_norm) e = tiny_initial_exponent(dgs[P3], p.pbits);
    }
    if (!p.accumulate && rank == 0)
        for (int i = threadIdx.x; i < P; i += blockDim.x) p.g[i] = 0.f;
    if (threadIdx.x < kScalarWords) scs[((p.n_steps - 1) & 1) * kScalarWords + threadIdx.x] = ((const float*)(p.scal + p.n_steps - 1))[threadIdx.x];
    __syncthreads();

    float Y[RK_MAX_STAGES][DM], H[RK_MAX_STAGES][UH], K[RK_MAX_STAGES][DM], psi[RK_MAX_STAGES][DM];
    // per stage: the cotangent of the layer-1 pre-activation and of the stage derivative (the parameter gradients are formed from
    // them after the stage loop)
    float DZ[RK_MAX_STAGES][UH], KAP[RK_MAX_STAGES][DM];
    int retries = 0, overflow_seen = 0;
    const int s = p.stages;
    const int k_lim = dynamic ? p.k_max : 1;
    bool failed = false;
    float ybar[DM];
#pragma unroll
    for (int c = 0; c < DM; ++c) ybar[c] = c < p.d ? Low<T>::to_f(traj[((long long)(p.n_steps - 1) * p.B + b) * p.d + c]) : 0.f;

    for (int i = p.n_steps - 1; i >= 0; --i) {
        const RkStepScalars& sc = *(const RkStepScalars*)(scs + (i & 1) * kScalarWords);
        tiny_stages<T, UH, DM, POLY>(p, lw, sc, ybar, Y, H, K);        // recompute the increment
        // the step below: its state and scalars travel while this step runs
        float next_sc = 0.f;
        if (i > 0) {
            if (threadIdx.x < kScalarWords) next_sc = ((const float*)(p.scal + i - 1))[threadIdx.x];
#pragma unroll
            for (int c = 0; c < DM; ++c)
                if (c < p.d) ybar[c] = Low<T>::to_f(traj[((long long)(i - 1) * p.B + b) * p.d + c]);
        }
        float phi_a = 0.f;                                             // this sample's share of Phi^T a_{i+1} (adjoint before its update)
        if (want_dt) {
#pragma unroll
            for (int c = 0; c < DM; ++c) {
                float ph = 0.f;
#pragma unroll
                for (int j = 0; j < RK_MAX_STAGES; ++j)
                    if (j < s) ph = fmaf(sc.b[j], K[j][c], ph);
                if (p.round_increment) ph = q16<T>(ph);
                phi_a = fmaf(ph, a[c], phi_a);
            }
        }
        int k_try = 0;
        bool accepted = false;
        float a_new[DM];
        while (k_try < k_lim) {
            ++k_try;
            bool bad = false;
            float v[DM];
#pragma unroll
            for (int c = 0; c < DM; ++c) { v[c] = q16<T>(ldexpf(a[c], e)); bad |= q_nonfinite<T>(v[c]); }   // Q16(S a)
            float g_dt = 0.f, g_dh = 0.f;                              // this sample's dt and dh (Eq. (vjp))
            float g_p0 = 0.f, g_p1 = 0.f, g_p2 = 0.f;                  // scalar example: its three parameter cotangents
#pragma unroll
            for (int j = RK_MAX_STAGES - 1; j >= 0; --j) {
                if (j >= s) continue;
                float dtau = 0.f;                                      // cotangent of the stage time tau_j, this sample's share
#pragma unroll
                for (int c = 0; c < DM; ++c) {
                    float acc = sc.b[j] * v[c];
#pragma unroll
                    for (int l = 0; l < RK_MAX_STAGES; ++l)
                        if (l > j && l < s && sc.ha[l][j] != 0.f) acc = fmaf(sc.ha[l][j], psi[l][c], acc);
                    KAP[j][c] = q16<T>(acc);
                    bad |= q_nonfinite<T>(KAP[j][c]);
                }
                if constexpr (POLY) {   // psi = Q16(-lambda kappa); cotangent of lambda and of the three parameters, each product rounded
                    const float lam = H[j][0], t2 = H[j][1];
                    const float ps = q16<T>(-lam * KAP[j][0]);
                    const float dlam = q16<T>(-Y[j][0] * KAP[j][0]);
                    const float d1 = q16<T>(dlam * t2), d2 = q16<T>(dlam * sc.tau16[j]);
                    bad |= q_nonfinite<T>(ps) | q_nonfinite<T>(dlam) | q_nonfinite<T>(d1) | q_nonfinite<T>(d2);
                    psi[j][0] = ps;
                    g_p0 += d1; g_p1 += d2; g_p2 += dlam;
                    if (want_dt) {      // d lambda / d tau = 2 theta_1 tau + theta_2, operation by operation
                        const float dt2 = q16<T>(dlam * w.W1[0]);
                        const float dts = q16_sum<T>(q16<T>(dt2 * q16<T>(2.f * sc.tau16[j])), q16<T>(dlam * w.W1[1]));
                        bad |= q_nonfinite<T>(dt2) | q_nonfinite<T>(dts);
                        g_dt += dts;
                        float dhs = sc.c[j] * dts;
#pragma unroll
                        for (int l = 0; l < RK_MAX_STAGES; ++l)
                            if (l < j && sc.a[j][l] != 0.f) dhs = fmaf(sc.a[j][l], ps * K[l][0], dhs);
                        g_dh += dhs;
                    }
                } else {
                    // last layer: dX = W2^T kappa (dW2 += kappa H^T and db2 += kappa follow after the stage loop)
#pragma unroll
                    for (int c = 0; c < DM; ++c) psi[j][c] = 0.f;
#pragma unroll
                    for (int u = 0; u < UH; ++u) {
                        float dx = 0.f;
#pragma unroll
                        for (int c = 0; c < DM; ++c)
                            if (c < p.d) dx = fmaf(KAP[j][c], lw.W2(u, c), dx);
                        const float dz = q16<T>(act_deriv_from_output(p.act, H[j][u]) * dx);
                        bad |= q_nonfinite<T>(dz);
                        DZ[j][u] = dz;
#pragma unroll
                        for (int c = 0; c < DM; ++c)
                            if (c < p.d) psi[j][c] = fmaf(dz, lw.W1(u, c), psi[j][c]);
                        dtau = fmaf(dz, lw.wt(u), dtau);
                    }
#pragma unroll
                    for (int c = 0; c < DM; ++c) {
                        psi[j][c] = c < p.d ? q16<T>(lanes_sum<POLY>(psi[j][c])) : 0.f;
                        bad |= q_nonfinite<T>(psi[j][c]);
                    }
                    if (want_dt) {      // tau_j = t_i + c_j h and Y_j = ybar + h sum_l a_jl k_l both depend on the grid
                        dtau = lanes_sum<POLY>(dtau);
                        g_dt += dtau;
                        float dhs = sc.c[j] * dtau;
#pragma unroll
                        for (int l = 0; l < RK_MAX_STAGES; ++l) {
                            if (l >= j || sc.a[j][l] == 0.f) continue;
                            float dot = 0.f;
#pragma unroll
                            for (int c = 0; c < DM; ++c) dot = fmaf(psi[j][c], K[l][c], dot);
                            dhs = fmaf(sc.a[j][l], dot, dhs);
                        }
                        g_dh += dhs;
                    }
                }
            }
            // the adjoint this attempt would leave
            const float coef = ldexpf(sc.h, -e);
            float m = 0.f;
#pragma unroll
            for (int c = 0; c < DM; ++c) {
                float da = 0.f;
#pragma unroll
                for (int j = RK_MAX_STAGES - 1; j >= 0; --j)
                    if (j < s) da += psi[j][c];
                a_new[c] = fmaf(coef, da, a[c]);
                if (p.cot != nullptr && active && c < p.d) a_new[c] += p.cot[((long long)i * p.B + b) * p.d + c];     // w_i dR/dy_i
                m = fmaxf(m, fabsf(a_new[c]));
            }
            // This lane's share of its units' parameter gradients (the stages added last to first), summed over the batch: the warp's
            // samples by shuffles, then warps and blocks in ascending order in exchange()
            auto to_part = [&](int i2, float x, bool mine) {
#pragma unroll
                for (int o = 16; o >= LP; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
                if (lane < LP && mine) part[(size_t)warp * P3 + i2] = x;
            };
            const float keep = active ? 1.f : 0.f;                     // lanes past the batch count nothing
            if constexpr (POLY) {
                to_part(0, keep * g_p0, true); to_part(1, keep * g_p1, true); to_part(2, keep * g_p2, true);
            } else {
#pragma unroll
                for (int u = 0; u < UH; ++u) {
                    const int n = q + kLanes * u;
                    const bool mine = n < p.h;
                    float x;
#pragma unroll
                    for (int c = 0; c < DM; ++c) {
                        if (c >= p.d) continue;
                        x = 0.f;                                       // dW1 = dZ Y^T
#pragma unroll
                        for (int j = RK_MAX_STAGES - 1; j >= 0; --j)
                            if (j < s) x = fmaf(DZ[j][u], Y[j][c], x);
                        to_part(n * in1 + c, keep * x, mine);
                        x = 0.f;                                       // dW2 = kappa H^T
#pragma unroll
                        for (int j = RK_MAX_STAGES - 1; j >= 0; --j)
                            if (j < s) x = fmaf(KAP[j][c], H[j][u], x);
                        to_part(o_w2 + c * p.h + n, keep * x, mine);
                    }
                    if (p.time) {                                      // the time column: tau_j dZ
                        x = 0.f;
#pragma unroll
                        for (int j = RK_MAX_STAGES - 1; j >= 0; --j)
                            if (j < s) x = fmaf(sc.tau16[j], DZ[j][u], x);
                        to_part(n * in1 + p.d, keep * x, mine);
                    }
                    if (nb1) {
                        x = 0.f;
#pragma unroll
                        for (int j = RK_MAX_STAGES - 1; j >= 0; --j)
                            if (j < s) x += DZ[j][u];
                        to_part(o_b1 + n, keep * x, mine);
                    }
                }
                if (nb2) {
#pragma unroll
                    for (int c = 0; c < DM; ++c) {                     // db2 = kappa: the same in the eight lanes
                        if (c >= p.d) continue;
                        float x = 0.f;
#pragma unroll
                        for (int j = RK_MAX_STAGES - 1; j >= 0; --j)
                            if (j < s) x += KAP[j][c];
                        to_part(o_b2 + c, keep * x, q == 0);
                    }
                }
            }
            if (want_dt) { to_part(P, keep * g_dt, q == 0); to_part(P + 1, keep * g_dh, q == 0); to_part(P + 2, keep * phi_a, q == 0); }
            const bool any_bad = exchange(bad && active, active ? m : 0.f, true);
            if (!checked) { accepted = true; break; }
            if (!dynamic) { overflow_seen |= any_bad; accepted = true; break; }
            if (!any_bad) { accepted = true; break; }
            if (e > -100) --e;                                         // halve and retry
            ++retries;
        }
        if (rank == 0 && threadIdx.x == 0) { p.log_exp[i] = e; p.log_attempts[i] = k_try; p.log_doubled[i] = 0; }
        if (!accepted) {
            if (rank == 0 && threadIdx.x == 0) { p.status[0] = MPODE_ERR_SCALE_FAILED; p.status[1] = i; p.status[2] = retries; }
            failed = true;
            break;
        }
        // high-precision updates with h / S
        const float coef = ldexpf(sc.h, -e);
#pragma unroll
        for (int c = 0; c < DM; ++c) a[c] = a_new[c];
        if (rank == 0) {
            for (int i2 = threadIdx.x; i2 < P; i2 += blockDim.x) p.g[i2] = fmaf(coef, dgs[i2], p.g[i2]);
            if (want_dt && threadIdx.x == 0) {                         // Alg. 2: the two t' updates
                const float dts = dgs[P], dhs = dgs[P + 1], ph = dgs[P + 2];
                p.tprime[i] = p.tprime[i] + coef * (dts - dhs) - ph;
                p.tprime[i + 1] = p.tprime[i + 1] + coef * dhs + ph;
            }
        }
        if (dynamic && k_try == 1) {                                   // growth test
            const double scaled = p.growth_rule == 0 ? ldexp((double)dgs[P3], e) : (double)dgs[P3];
            if (scaled <= ldexp(1.0, p.pbits - 1) && e < 100) {
                ++e;
                if (rank == 0 && threadIdx.x == 0) p.log_doubled[i] = 1;
            }
        }
        if (i > 0 && threadIdx.x < kScalarWords) scs[((i - 1) & 1) * kScalarWords + threadIdx.x] = next_sc;
        __syncthreads();                                               // scalars are in place, dgs is free
    }
    if (!failed) {
        if (p.scaling == MPODE_SCALE_NONE_SAFE && overflow_seen) {
#pragma unroll
            for (int c = 0; c < DM; ++c) a[c] = INFINITY;
            if (rank == 0) {
                for (int i2 = threadIdx.x; i2 < P; i2 += blockDim.x) p.g[i2] = INFINITY;
                if (want_dt)
                    for (int i2 = threadIdx.x; i2 <= p.n_steps; i2 += blockDim.x) p.tprime[i2] = INFINITY;
                if (threadIdx.x == 0) p.status[0] = MPODE_WARN_NONFINITE_GRAD;
            }
        }
        if (rank == 0 && threadIdx.x == 0) p.status[2] = retries;
        if (active && q == 0) {
#pragma unroll
            for (int c = 0; c < DM; ++c)
                if (c < p.d) p.a[(long long)b * p.d + c] = a[c];
        }
    }
    cl.sync();                                                         // no block leaves while another reads its shared memory
}

template <typename T, int UH, int DM, bool POLY>
void forward_t(const TinyParams& p, cudaStream_t st) {
    const int per = 64 / (POLY ? 1 : kLanes);
    const size_t smem = (size_t)(tiny_weight_floats(p.d, kLanes * UH) + 2 * kScalarWords) * sizeof(float);
    tiny_forward_kernel<T, UH, DM, POLY><<<(p.B + per - 1) / per, 64, smem, st>>>(p);
}

template <typename T, int UH, int DM, bool POLY, int THREADS>
bool backward_t(const TinyParams& p, cudaStream_t st) {
    const int total = p.B * (POLY ? 1 : kLanes);
    int threads = total < THREADS ? (total + 31) / 32 * 32 : THREADS;
    if (threads < 64) threads = 64;                                    // a step's scalars are fetched a word per thread
    const int blocks = (total + threads - 1) / threads;                // at most 16: TINY_MAX_B * 8 / 512
    const int P3 = (POLY ? 3 : p.h * (p.d + (p.time ? 1 : 0)) + (p.bias ? p.h : 0) + p.d * p.h + (p.bias ? p.d : 0)) + 3;
    const size_t smem = (size_t)(tiny_weight_floats(p.d, kLanes * UH) + 2 * kScalarWords + (threads / 32) * P3 + 32 + 3 * (P3 + 2)) * sizeof(float);
    static bool attr[kMaxDevices] = {false};
    const int dev = current_device();
    if (!attr[dev]) {
        if (cudaFuncSetAttribute(tiny_backward_kernel<T, UH, DM, POLY, THREADS>, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024) != cudaSuccess ||
            cudaFuncSetAttribute(tiny_backward_kernel<T, UH, DM, POLY, THREADS>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
            return false;
        attr[dev] = true;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)blocks; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, tiny_backward_kernel<T, UH, DM, POLY, THREADS>, p) == cudaSuccess;
}

// the smallest variant that holds the sizes: hidden units per lane (4, 8) and state width (2, 4, 8); the scalar example has its own
template <typename T, bool BWD>
bool launch_t(const TinyParams& p, cudaStream_t st) {
    const bool wide = p.B * (p.poly ? 1 : kLanes) > 16 * 256;      // more samples than a cluster of 16 narrow blocks takes
#define MPODE_TINY(UH, DM, POLY)                                     \
    do {                                                             \
        if (BWD) return wide ? backward_t<T, UH, DM, POLY, 512>(p, st) : backward_t<T, UH, DM, POLY, 256>(p, st); \
        forward_t<T, UH, DM, POLY>(p, st);                           \
        return true;                                                 \
    } while (0)
    if (p.poly) MPODE_TINY(2, 1, true);
    if (p.h <= 32) {
        if (p.d <= 2) MPODE_TINY(4, 2, false);
        if (p.d <= 4) MPODE_TINY(4, 4, false);
        MPODE_TINY(4, 8, false);
    }
    if (p.d <= 2) MPODE_TINY(8, 2, false);
    if (p.d <= 4) MPODE_TINY(8, 4, false);
    MPODE_TINY(8, 8, false);
#undef MPODE_TINY
}

}  // namespace

bool tiny_mlp_supported(int B, int d, int h, int n_layers, int p) {
    return n_layers == 2 && d >= 1 && d <= TINY_MAX_D && h >= 1 && h <= TINY_MAX_H && B >= 1 && B <= TINY_MAX_B && p <= TINY_MAX_P;
}

bool launch_tiny_forward(mpode_dtype dt, const TinyParams& p, cudaStream_t st, long long* launches) {
    const bool ok = dt == MPODE_BF16 ? launch_t<__nv_bfloat16, false>(p, st) : (dt == MPODE_F16 ? launch_t<__half, false>(p, st) : launch_t<float, false>(p, st));
    if (ok && launches) ++*launches;
    return ok;
}

bool launch_tiny_backward(mpode_dtype dt, const TinyParams& p, cudaStream_t st, long long* launches) {
    const bool ok = dt == MPODE_BF16 ? launch_t<__nv_bfloat16, true>(p, st) : (dt == MPODE_F16 ? launch_t<__half, true>(p, st) : launch_t<float, true>(p, st));
    if (ok && launches) ++*launches;
    return ok;
}

}  // namespace mpode
