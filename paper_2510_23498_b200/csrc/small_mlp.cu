// Row-local kernels for small dense velocities.  Samples are independent through the time loop, so a block
// takes 16 (or 32) of them through the whole forward solve, or through the backward chain of several steps, without talking to any
// other block: a layer is one contraction [16 x K] x [K x N] whose activations never leave the SM (the weights come from L2 through a
// ring of buffers in shared memory), and the next layer starts after a block barrier.  What bounds this is the chain of layers, not bytes or tensor rate:
// a tcgen05 tile needs 128 rows (64 at half rate) and a hand-over between its epilogue and the next tile's operands, about 8 us per
// layer in rk_fused.cu, while mma.sync fragments of 16 rows spread the batch over the SMs and hand over in registers and shared memory.
// float32 runs the same program on the CUDA cores, 8 rows to a block: 12 us an evaluation of 96 K weights, 3.2 of them multiply-adds at full
// rate; two warps a scheduler do not hide the operands' latency.  16-bit networks whose weights fit the SM run in resident_mlp.cu.
// Weight gradients reduce over the whole batch: the chain keeps every layer input and cotangent of its steps in memory (L2), and a
// second launch forms them (small_wgrad.cu).
// Measured (training pass, before: rk_fused.cu): MLP 128-256-256-128 (128 K weights), 200 samples, 8 RK4 steps, bf16 1.65 -> 1.03 ms; MLP
// 64-256-256-64, 1024 samples, 16 RK4 steps, float32 5.7 -> 3.4 ms since a lane has four columns.
#include "small_mlp.h"

#include "profiler.h"
#include "tc_ptx.cuh"
#include "tensormap.h"

namespace mpode {
using namespace tc;
namespace {

constexpr int kWarps = 8, kThreads = 32 * kWarps;      // working warps; one more warp streams the weights
constexpr int kPassCols = 256, kUnitBytes = 16384;

template <typename T> __device__ __forceinline__ float lowf(T x) { return Low<T>::to_f(x); }
template <typename T> __device__ __forceinline__ float q16(float x) { return Low<T>::to_f(Low<T>::from_f(x)); }

// two neighbouring elements of a row, moved as one word
template <typename T> struct Pair { using W = uint32_t; };
template <> struct Pair<float> { using W = float2; };
template <typename T> __device__ __forceinline__ typename Pair<T>::W pack_w(float a, float b) {
    if constexpr (sizeof(T) == 4) return make_float2(a, b); else return cvt_pack<T>(a, b);
}
template <typename T> __device__ __forceinline__ T low_of(typename Pair<T>::W w) {
    if constexpr (sizeof(T) == 4) return w.x; else return from_bits<T>((unsigned short)(w & 0xFFFFu));
}
template <typename T> __device__ __forceinline__ T high_of(typename Pair<T>::W w) {
    if constexpr (sizeof(T) == 4) return w.y; else return from_bits<T>((unsigned short)(w >> 16));
}
template <typename T> __device__ __forceinline__ float lo_w(typename Pair<T>::W w) { return lowf(low_of<T>(w)); }
template <typename T> __device__ __forceinline__ float hi_w(typename Pair<T>::W w) { return lowf(high_of<T>(w)); }
// rows of a block: 16 per row tile of the matrix instructions; float32 runs on the CUDA cores with 8
template <typename T, int MT> constexpr int kRows = (sizeof(T) == 4 ? 8 : 16) * MT;


template <typename T> __device__ __forceinline__ float act_f(int act, float z) {
    if constexpr (sizeof(T) == 4) return act_fwd(act, z);
    switch (act) {
        case MPODE_ACT_SOFTPLUS: return fast_act<MPODE_ACT_SOFTPLUS>(z);
        case MPODE_ACT_RELU: return fast_act<MPODE_ACT_RELU>(z);
        case MPODE_ACT_TANH: return fast_act<MPODE_ACT_TANH>(z);
        default: return z;
    }
}
template <typename T> __device__ __forceinline__ float act_df(int act, float h) {
    if constexpr (sizeof(T) == 4) return act_deriv_from_output(act, h);
    switch (act) {
        case MPODE_ACT_SOFTPLUS: return fast_act_deriv<MPODE_ACT_SOFTPLUS>(h);
        case MPODE_ACT_RELU: return fast_act_deriv<MPODE_ACT_RELU>(h);
        case MPODE_ACT_TANH: return fast_act_deriv<MPODE_ACT_TANH>(h);
        default: return 1.f;
    }
}

__host__ __device__ inline int k32(int w) { return (w + 31) / 32; }

// ---------------------------------------------------------------- weights in fragment order, biases
struct PackJob { long long first[2 * SMALL_MAX_L + 1]; };      // first 16-byte group of each (layer, direction)
template <typename T>
__global__ void __launch_bounds__(256) small_pack_kernel(const __grid_constant__ SmallMlp p, const __grid_constant__ PackJob job) {
    chain_begin();
    const long long n = job.first[2 * p.L];
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        int q = 0;
        while (i >= job.first[q + 1]) ++q;
        const int l = q >> 1, back = q & 1;
        // [pass of 32 column tiles][32 of the reduction][tile][lane]
        const int r = (int)(i - job.first[q]), lane = r & 31;
        const int kp = k32(back ? p.wp[l + 1] : p.wp[l]), tiles = (back ? p.wp[l] : p.wp[l + 1]) / 8;
        const int pass = (r >> 5) / (32 * kp), in_pass = tiles - 32 * pass < 32 ? tiles - 32 * pass : 32, rr = (r >> 5) - pass * 32 * kp;
        const int kk = rr / in_pass, tile = pass * 32 + rr % in_pass;
        const int in_full = p.wr[l] + ((p.time && l == 0) ? 1 : 0);
        uint32_t w[4];
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            float v[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int k = kk * 32 + (g >> 1) * 16 + (g & 1) * 8 + 2 * (lane & 3) + h, c = tile * 8 + (lane >> 2);
                const int out = back ? k : c, in = back ? c : k;
                v[h] = out < p.wr[l + 1] && in < p.wr[l] ? p.theta[p.woff[l] + (long long)out * in_full + in] : 0.f;
            }
            w[g] = cvt_pack<T>(v[0], v[1]);
        }
        (back ? p.wb[l] : p.wf[l])[r] = make_uint4(w[0], w[1], w[2], w[3]);
    }
    if (blockIdx.x == 0) {
        for (int l = 0; l < p.L; ++l)
            for (int c = threadIdx.x; c < p.wp[l + 1]; c += blockDim.x) {
                const bool on = c < p.wr[l + 1];
                if (p.bias) ((T*)p.b16[l])[c] = Low<T>::from_f(on ? p.theta[p.boff[l] + c] : 0.f);
                if (p.time && l == 0) ((T*)p.wt16)[c] = Low<T>::from_f(on ? p.theta[p.woff[0] + (long long)c * (p.wr[0] + 1) + p.wr[0]] : 0.f);
            }
    }
}

// float32: forward [inputs][outputs], backward [outputs][inputs], zero in the padding
__global__ void __launch_bounds__(256) small_pack_f32_kernel(const __grid_constant__ SmallMlp p, const __grid_constant__ PackJob job) {
    chain_begin();
    const long long n = job.first[2 * p.L];
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        int q = 0;
        while (i >= job.first[q + 1]) ++q;
        // [pass of 256 columns][reduction][column]
        const int l = q >> 1, back = q & 1, r = (int)(i - job.first[q]);
        const int N = back ? p.wp[l] : p.wp[l + 1], K = back ? p.wp[l + 1] : p.wp[l];
        const int pass = r / (kPassCols * K), in_pass = N - kPassCols * pass < kPassCols ? N - kPassCols * pass : kPassCols, rr = r - pass * kPassCols * K;
        const int k = rr / in_pass, c = pass * kPassCols + rr % in_pass;
        const int out = back ? k : c, in = back ? c : k;
        const int in_full = p.wr[l] + ((p.time && l == 0) ? 1 : 0);
        ((float*)(back ? p.wb[l] : p.wf[l]))[r] = out < p.wr[l + 1] && in < p.wr[l] ? p.theta[p.woff[l] + (long long)out * in_full + in] : 0.f;
    }
    if (blockIdx.x == 0) {
        for (int l = 0; l < p.L; ++l)
            for (int c = threadIdx.x; c < p.wp[l + 1]; c += blockDim.x) {
                const bool on = c < p.wr[l + 1];
                if (p.bias) ((float*)p.b16[l])[c] = on ? p.theta[p.boff[l] + c] : 0.f;
                if (p.time && l == 0) ((float*)p.wt16)[c] = on ? p.theta[p.woff[0] + (long long)c * (p.wr[0] + 1) + p.wr[0]] : 0.f;
            }
    }
}

// ---------------------------------------------------------------- the weights on their way through shared memory
// The order in which a block needs the weights is fixed, so one thread streams them ahead of the arithmetic: bulk copies of at most
// 16 KB (32 of the reduction for up to 32 column tiles; in float32 16 rows of up to 256 columns) through a ring of buffers, across layer
// and stage boundaries.  (Loaded by the warps themselves, even 16 loads ahead, each unit cost an L2 round trip of half a microsecond.)
// Every wait is bounded.  A thread whose wait has given up waits no more (the producer issues no more) and runs on to its end, the error
// word tells the host, and the producer leaves last: a block does not end while copies into its shared memory are on their way.
struct Ring {
    uint64_t *full, *empty;
    unsigned char* buf;
    int n, s;
    uint32_t phase;
    bool lost;
    unsigned* err;
    unsigned long long wait_ns;
    bool laps;                 // whether every buffer has been used
    __device__ __forceinline__ void next() { if (++s == n) { s = 0; phase ^= 1u; laps = true; } }
    __device__ __forceinline__ unsigned char* stage() const { return buf + s * kUnitBytes; }
};
__device__ __forceinline__ void work_sync() { asm volatile("bar.sync 1, 256;" ::: "memory"); }      // the working warps

__device__ __forceinline__ void ring_wait(Ring& r) {
    if (!mbar_try_wait(&r.full[r.s], r.phase) && !r.lost) r.lost = !mbar_wait_long(&r.full[r.s], r.phase, r.err, 4u, r.wait_ns);
}
__device__ __forceinline__ void stream_units(Ring& r, const unsigned char* src, int bytes) {
    if (!r.lost) r.lost = !mbar_wait(&r.empty[r.s], r.phase ^ 1u, r.err, 1u, r.wait_ns);
    if (r.lost) return;
    mbar_arrive_expect_tx(&r.full[r.s], (uint32_t)bytes);
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_u32(r.stage())), "l"(src), "r"(bytes),
                 "r"(smem_u32(&r.full[r.s])) : "memory");
    r.next();
}
// the producer's last act: what it has issued lands (the last fill of every buffer that has been filled)
__device__ __forceinline__ void ring_drain(const Ring& r) {
    for (int q = 0; q < r.n; ++q) {
        const bool this_lap = q < r.s;
        if (this_lap || r.laps) mbar_wait(&r.full[q], this_lap ? r.phase : r.phase ^ 1u, r.err, 2u, r.wait_ns);
    }
}
// one contraction's weights: reduction K, N columns
template <typename T> __device__ __forceinline__ void stream_layer(Ring& r, const uint4* W, int K, int N) {
    const unsigned char* src = (const unsigned char*)W;
    for (int c = 0; c < N; c += kPassCols) {
        const int cols = min(kPassCols, N - c);
        if constexpr (sizeof(T) == 4) {
            for (int k = 0; k < K; k += 16) { const int b = min(16, K - k) * cols * 4; stream_units(r, src, b); src += b; }
        } else {
            const int b = cols * 64;
            for (int k = 0; k < k32(K); ++k) { stream_units(r, src, b); src += b; }
        }
    }
}

// ---------------------------------------------------------------- one contraction of a block's rows
// C[16 MT][8 tiles] = A[16 MT][32 kp] W, A in shared memory (row length lda), W from the ring.  Warp w takes the column tiles w, w + 8, ...
// of a pass.  pre(g, q, row, col) runs before the reduction loop and requests what the epilogue needs from memory for piece q of column
// tile g; epi(g, q, row, col, c0, c1) gets two neighbouring columns.
constexpr int kNG = 4;
template <typename T, int MT, typename P, typename F>
__device__ __forceinline__ void rows_gemm(Ring& ring, const T* A, int lda, int kp, int tiles, P&& pre, F&& epi) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t a0 = smem_u32(A) + (uint32_t)(((lane & 15) * lda + (lane >> 4) * 8) * 2);
    for (int p0 = 0; p0 < tiles; p0 += 32) {
        const int in_pass = min(32, tiles - p0);
        float acc[MT][kNG][4];
#pragma unroll
        for (int g = 0; g < kNG; ++g)
            if (warp + kWarps * g < in_pass) {
#pragma unroll
                for (int q = 0; q < 2 * MT; ++q) pre(g, q, q * 8 + (lane >> 2), (p0 + warp + kWarps * g) * 8 + 2 * (lane & 3));
            }
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int g = 0; g < kNG; ++g)
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[m][g][i] = 0.f;
        for (int k = 0; k < kp; ++k) {
            uint32_t a[MT][2][4];
#pragma unroll
            for (int m = 0; m < MT; ++m) {
                ldm4(a0 + (uint32_t)((m * 16 * lda + k * 32) * 2), a[m][0]);
                ldm4(a0 + (uint32_t)((m * 16 * lda + k * 32 + 16) * 2), a[m][1]);
            }
            ring_wait(ring);
            const uint4* W = (const uint4*)ring.stage() + warp * 32 + lane;
            uint4 b[kNG];
#pragma unroll
            for (int g = 0; g < kNG; ++g)
                if (warp + kWarps * g < in_pass) b[g] = W[g * kWarps * 32];
            __syncwarp();
            if (lane == 0) mbar_arrive(&ring.empty[ring.s]);      // the fragments are in registers
            ring.next();
#pragma unroll
            for (int g = 0; g < kNG; ++g)
                if (warp + kWarps * g < in_pass) {
#pragma unroll
                    for (int m = 0; m < MT; ++m) mma_k16<T>(acc[m][g], a[m][0], b[g].x, b[g].y);
                }
#pragma unroll
            for (int g = 0; g < kNG; ++g)
                if (warp + kWarps * g < in_pass) {
#pragma unroll
                    for (int m = 0; m < MT; ++m) mma_k16<T>(acc[m][g], a[m][1], b[g].z, b[g].w);
                }
        }
#pragma unroll
        for (int g = 0; g < kNG; ++g)
            if (warp + kWarps * g < in_pass) {
                const int col = (p0 + warp + kWarps * g) * 8 + 2 * (lane & 3);
#pragma unroll
                for (int m = 0; m < MT; ++m) {
                    epi(g, 2 * m, m * 16 + (lane >> 2), col, acc[m][g][0], acc[m][g][1]);
                    epi(g, 2 * m + 1, m * 16 + (lane >> 2) + 8, col, acc[m][g][2], acc[m][g][3]);
                }
            }
    }
}

// Shared memory of a block: two activation buffers (row length lda, zero behind the layer's width up to a multiple of 32), the stage
// derivatives, stage cotangents, state and seed of its rows and the fp32 state or adjoint (row length wp_0), two steps' scalars, the
// warps' sums of the time terms.
constexpr int kScalarWords = sizeof(RkStepScalars) / sizeof(float);
template <typename T> struct SmallSmem {
    T *act0, *ks, *ps, *yb, *vv;
    float *a, *scs, *red, *scratch;
    int lda, R, dp, d, half, pairs;
    __device__ SmallSmem(const SmallMlp& p, unsigned char* base, int rows) : R(rows), dp(p.wp[0]), d(p.wr[0]) {
        int kp = 0;
        for (int l = 0; l <= p.L; ++l) kp = max(kp, k32(p.wp[l]));
        lda = kp * 32 + 8;
        half = dp / 2; pairs = R * half;
        act0 = (T*)base;
        ks = act0 + 2 * R * lda; ps = ks + p.stages * R * dp; yb = ps + p.stages * R * dp; vv = yb + R * dp;
        a = (float*)(vv + R * dp);
        scs = a + R * dp;
        red = scs + 2 * kScalarWords;
        scratch = red + 3 * kWarps;
    }
    __device__ __forceinline__ T* act(int i) const { return act0 + i * R * lda; }
    __device__ __forceinline__ typename Pair<T>::W* w(T* x) const { return reinterpret_cast<typename Pair<T>::W*>(x); }
    __device__ __forceinline__ const RkStepScalars& scalars(int n) const { return *(const RkStepScalars*)(scs + (n & 1) * kScalarWords); }
};
template <typename T> size_t small_smem(const SmallMlp& p, int rows) {
    int kp = 0;
    for (int l = 0; l <= p.L; ++l) kp = k32(p.wp[l]) > kp ? k32(p.wp[l]) : kp;
    return (size_t)rows * sizeof(T) * (2 * (kp * 32 + 8) + (2 * p.stages + 2) * p.wp[0]) + (size_t)rows * p.wp[0] * 4 + (2 * kScalarWords + 3 * kWarps) * 4 +
           (sizeof(T) == 4 ? (size_t)kThreads * rows * 4 : 0);
}
// the ring behind the block's own shared memory: `n` buffers, then the barriers
__device__ __forceinline__ Ring make_ring(unsigned char* base, int n, unsigned* err, unsigned long long wait_ns) {
    Ring r;
    r.buf = base; r.n = n; r.s = 0; r.phase = 0; r.lost = r.laps = false; r.err = err; r.wait_ns = wait_ns;
    r.full = (uint64_t*)(base + n * kUnitBytes);
    r.empty = r.full + n;
    if (threadIdx.x == 0) {
        for (int i = 0; i < n; ++i) { mbar_init(&r.full[i], 1); mbar_init(&r.empty[i], kWarps); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    return r;
}
// a step's scalars travel to shared memory while the step before runs (asynchronous; wait with scalars_ready and a barrier)
template <typename T>
__device__ __forceinline__ void fetch_scalars(const SmallMlp& p, const SmallSmem<T>& sm, int n) {
    if (threadIdx.x < kScalarWords) {
        const float* src = (const float*)(p.scal + n) + threadIdx.x;
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(sm.scs + (n & 1) * kScalarWords + threadIdx.x)), "l"(src) : "memory");
    }
}
__device__ __forceinline__ void scalars_ready() { copies_done(); }

// float32 on the CUDA cores: a lane has four columns and all the block's rows, and a quarter of each unit's 16 reduction steps (8 lanes side
// by side share a quarter): 12 shared-memory reads of 16 bytes for 128 multiply-adds (16 rows: 20 for 256).  (One column a thread was 12 reads,
// 8 of 16 bytes, for 32, and bound by them.)  A warp covers 32 columns; where the pass has fewer than 256 the warps that are left
// share out the units.  The quarters meet by shuffles, each lane keeping a quarter of the rows, the warps' shares in shared memory; sums are
// added in a fixed order.
template <int MT, typename P, typename F>
__device__ __forceinline__ void rows_gemm_f32(Ring& ring, const SmallSmem<float>& sm, const float* A, int K, int N, P&& pre, F&& epi) {
    constexpr int R = kRows<float, MT>, Q = R / 4;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, kg = lane >> 3;
    for (int c0 = 0; c0 < N; c0 += kPassCols) {
        const int cols = min(kPassCols, N - c0);
        int cw = 1;                                               // warps side by side; the others of the 8 take other units
        while (cw * 32 < cols) cw *= 2;
        const int kw = kWarps / cw, mine = warp / cw, col = (warp % cw) * 32 + (lane & 7) * 4;
        const bool on = col < cols;                               // (widths are multiples of 8)
        const int row0 = (kg >> 1) * (R / 2) + (kg & 1) * Q;      // the rows this lane keeps
        if (kw == 1 && on) {
#pragma unroll
            for (int g = 0; g < 2; ++g)
#pragma unroll
                for (int q = 0; q < Q; ++q) pre(g, q, row0 + q, c0 + col + 2 * g);
        }
        float acc[R][4];
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[r][i] = 0.f;
        int turn = 0;
        for (int k = 0; k < K; k += 16) {
            ring_wait(ring);
            if (turn == mine && on && k + 4 * kg < K) {           // (K is a multiple of 8)
                const float* w = (const float*)ring.stage() + (size_t)(4 * kg) * cols + col;
                float4 wv[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) wv[q] = *reinterpret_cast<const float4*>(w + (size_t)q * cols);
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const float4 a = *reinterpret_cast<const float4*>(A + r * sm.lda + k + 4 * kg);
                    const float av[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        acc[r][0] = fmaf(av[q], wv[q].x, acc[r][0]);
                        acc[r][1] = fmaf(av[q], wv[q].y, acc[r][1]);
                        acc[r][2] = fmaf(av[q], wv[q].z, acc[r][2]);
                        acc[r][3] = fmaf(av[q], wv[q].w, acc[r][3]);
                    }
                }
            }
            if (++turn == kw) turn = 0;
            __syncwarp();
            if (lane == 0) mbar_arrive(&ring.empty[ring.s]);
            ring.next();
        }
        float v[Q][4];
        {
            float h[R / 2][4];
#pragma unroll
            for (int r = 0; r < R / 2; ++r)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float send = (kg & 2) ? acc[r][i] : acc[r + R / 2][i];
                    h[r][i] = ((kg & 2) ? acc[r + R / 2][i] : acc[r][i]) + __shfl_xor_sync(0xffffffffu, send, 16);
                }
#pragma unroll
            for (int r = 0; r < Q; ++r)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float send = (kg & 1) ? h[r][i] : h[r + Q][i];
                    v[r][i] = ((kg & 1) ? h[r + Q][i] : h[r][i]) + __shfl_xor_sync(0xffffffffu, send, 8);
                }
        }
        if (kw == 1) {
            if (on) {
#pragma unroll
                for (int g = 0; g < 2; ++g)
#pragma unroll
                    for (int q = 0; q < Q; ++q) epi(g, q, row0 + q, c0 + col + 2 * g, v[q][2 * g], v[q][2 * g + 1]);
            }
            continue;
        }
        const int ct = cw * 32;
        if (c0 > 0) work_sync();
#pragma unroll
        for (int q = 0; q < Q; ++q) *reinterpret_cast<float4*>(sm.scratch + ((size_t)(mine * R + row0 + q) * ct + col)) = make_float4(v[q][0], v[q][1], v[q][2], v[q][3]);
        work_sync();
        const int hc = ct / 2;
        for (int i = threadIdx.x; i < R * hc; i += kThreads) {
            const int r = i / hc, c = 2 * (i - r * hc);
            if (c >= cols) continue;
            pre(0, 0, r, c0 + c);
            float2 u = make_float2(0.f, 0.f);
            for (int q = 0; q < kw; ++q) {
                const float2 x = *reinterpret_cast<const float2*>(sm.scratch + (size_t)(q * R + r) * ct + c);
                u.x += x.x; u.y += x.y;
            }
            epi(0, 0, r, c0 + c, u.x, u.y);
        }
    }
}

// C[rows][N] = A[rows][K] W: A one of the activation buffers, W the next weights of the ring
template <typename T, int MT, typename P, typename F>
__device__ __forceinline__ void block_gemm(Ring& ring, const SmallSmem<T>& sm, const T* A, int K, int N, P&& pre, F&& epi) {
    if constexpr (sizeof(T) == 4) rows_gemm_f32<MT>(ring, sm, A, K, N, pre, epi);
    else rows_gemm<T, MT>(ring, A, sm.lda, k32(K), N / 8, pre, epi);
}

// zeros behind a layer's width, up to the next multiple of 32 columns
template <typename T>
__device__ __forceinline__ void zero_tail(T* act, int lda, int R, int w) {
    const int pad = k32(w) * 32 - w;
    if (pad == 0) return;
    for (int i = threadIdx.x; i < R * pad; i += kThreads) act[(i / pad) * lda + w + i % pad] = Low<T>::from_f(0.f);
}

// All stages of one step for the rows r0 .. r0 + R - 1 from the state in sm.yb: k_j into sm.ks; with KEEP every layer input into the
// slabs (slot `slot`).  `skip_last`: the last stage's derivative is not wanted.
template <typename T, int MT, bool KEEP>
__device__ __forceinline__ void small_stages(const SmallMlp& p, Ring& ring, const SmallSmem<T>& sm, const RkStepScalars& sc, int r0, int slot, bool skip_last) {
    using W = typename Pair<T>::W;
    const int R = kRows<T, MT>, dp = sm.dp;
    for (int j = 0; j < p.stages; ++j) {
        float ha[RK_MAX_STAGES - 1];
#pragma unroll
        for (int l = 0; l < RK_MAX_STAGES - 1; ++l) ha[l] = l < j ? sc.ha[j][l] : 0.f;
        T* x0 = KEEP ? (T*)p.xs[0] + ((long long)(slot * p.stages + j) * p.B + r0) * dp : nullptr;
        for (int i = threadIdx.x; i < sm.pairs; i += kThreads) {
            const int r = i / sm.half, c = 2 * (i - r * sm.half);
            W q = sm.w(sm.yb)[i];
            if (j > 0) {
                float v0 = lo_w<T>(q), v1 = hi_w<T>(q);
#pragma unroll
                for (int l = 0; l < RK_MAX_STAGES - 1; ++l)
                    if (l < j && ha[l] != 0.f) {
                        const W k = sm.w(sm.ks)[l * sm.pairs + i];
                        v0 = fmaf(ha[l], lo_w<T>(k), v0);
                        v1 = fmaf(ha[l], hi_w<T>(k), v1);
                    }
                q = pack_w<T>(v0, v1);
            }
            *(W*)(sm.act(0) + r * sm.lda + c) = q;
            if (KEEP && r0 + r < p.B) *(W*)(x0 + r * dp + c) = q;
        }
        zero_tail(sm.act(0), sm.lda, R, dp);
        work_sync();
        const float tau = sc.tau16[j];
        for (int l = 0; l < p.L; ++l) {
            const bool last = l == p.L - 1;
            if (last && skip_last && j == p.stages - 1) break;
            const int N = p.wp[l + 1];
            const W* b16 = p.bias ? (const W*)p.b16[l] : nullptr;
            const W* wt = p.time && l == 0 ? (const W*)p.wt16 : nullptr;
            T* dst = last ? sm.ks + j * R * dp : sm.act((l + 1) & 1);
            const int ld = last ? dp : sm.lda;
            T* keep = KEEP && !last ? (T*)p.xs[l + 1] + ((long long)(slot * p.stages + j) * p.B + r0) * N : nullptr;
            float2 bv[kNG];
            block_gemm<T, MT>(
                ring, sm, sm.act(l & 1), p.wp[l], N,
                [&](int g, int q, int, int c) {
                    if (q != 0) return;               // the same for every row
                    bv[g] = make_float2(0.f, 0.f);
                    if (b16 != nullptr) { const W w = __ldg(b16 + c / 2); bv[g] = make_float2(lo_w<T>(w), hi_w<T>(w)); }
                    if (wt != nullptr) { const W w = __ldg(wt + c / 2); bv[g].x = fmaf(tau, lo_w<T>(w), bv[g].x); bv[g].y = fmaf(tau, hi_w<T>(w), bv[g].y); }
                },
                [&](int g, int, int r, int c, float v0, float v1) {
                    v0 += bv[g].x; v1 += bv[g].y;
                    if (!last) { v0 = act_f<T>(p.act, v0); v1 = act_f<T>(p.act, v1); }
                    const W w = pack_w<T>(v0, v1);
                    *(W*)(dst + r * ld + c) = w;
                    if (KEEP && !last && r0 + r < p.B) *(W*)(keep + (long long)r * N + c) = w;
                });
            if (!last) zero_tail(dst, sm.lda, R, N);
            work_sync();
        }
    }
}

template <typename T, int MT>
__global__ void __launch_bounds__(kThreads + 32, 1) small_forward_kernel(const __grid_constant__ SmallMlp p) {
    chain_begin();
    using W = typename Pair<T>::W;
    extern __shared__ __align__(16) unsigned char smem[];
    const int R = kRows<T, MT>, r0 = blockIdx.x * R;
    Ring ring = make_ring(smem, p.ring, p.err, p.wait_ns);
    if (threadIdx.x >= kThreads) {
        if (threadIdx.x == kThreads) {
            for (int n = 0; n < p.n_steps * p.stages; ++n)
                for (int l = 0; l < p.L; ++l) stream_layer<T>(ring, p.wf[l], p.wp[l], p.wp[l + 1]);
            ring_drain(ring);
        }
        return;
    }
    const SmallSmem<T> sm(p, smem + p.ring * (kUnitBytes + 16), R);
    const int d = sm.d, dp = sm.dp;
    T* traj = (T*)p.traj;
    fetch_scalars(p, sm, 0);
    for (int i = threadIdx.x; i < R * dp; i += kThreads) {
        const int r = i / dp, c = i - r * dp;
        const bool on = r0 + r < p.B && c < d;
        const float y = on ? p.y0[(long long)(r0 + r) * d + c] : 0.f;
        const T q = Low<T>::from_f(y);
        sm.yb[i] = q;
        sm.a[i] = y;
        if (on) traj[(long long)(r0 + r) * d + c] = q;
    }
    for (int n = 0; n < p.n_steps; ++n) {
        scalars_ready();
        work_sync();
        if (n + 1 < p.n_steps) fetch_scalars(p, sm, n + 1);
        const RkStepScalars& sc = sm.scalars(n);
        small_stages<T, MT, false>(p, ring, sm, sc, r0, 0, false);
        float hb[RK_MAX_STAGES];
#pragma unroll
        for (int j = 0; j < RK_MAX_STAGES; ++j) hb[j] = j < p.stages ? sc.hb[j] : 0.f;
        const float h = sc.h;
        T* tn = traj + ((long long)(n + 1) * p.B + r0) * d;
        for (int i = threadIdx.x; i < sm.pairs; i += kThreads) {
            const int r = i / sm.half, c = 2 * (i - r * sm.half);
            float v0 = 0.f, v1 = 0.f;
#pragma unroll
            for (int j = 0; j < RK_MAX_STAGES; ++j)
                if (j < p.stages) {
                    const W k = sm.w(sm.ks)[j * sm.pairs + i];
                    v0 = fmaf(hb[j], lo_w<T>(k), v0);
                    v1 = fmaf(hb[j], hi_w<T>(k), v1);
                }
            float2 y = reinterpret_cast<float2*>(sm.a)[i];
            y.x += p.round_increment ? h * q16<T>(v0) : v0;
            y.y += p.round_increment ? h * q16<T>(v1) : v1;
            reinterpret_cast<float2*>(sm.a)[i] = y;
            const W q = pack_w<T>(y.x, y.y);
            sm.w(sm.yb)[i] = q;
            if (r0 + r < p.B && c < d) {
                if ((d & 1) == 0) *(W*)(tn + r * d + c) = q;
                else {
                    tn[r * d + c] = low_of<T>(q);
                    if (c + 1 < d) tn[r * d + c + 1] = high_of<T>(q);
                }
            }
        }
    }
    work_sync();
    for (int i = threadIdx.x; i < R * d; i += kThreads) {
        const int r = i / d, c = i - r * d;
        if (r0 + r < p.B) p.yT[(long long)r0 * d + i] = sm.a[r * dp + c];
    }
}

// The backward chain of `count` steps for a block's rows: recompute, seed, stage cotangents and layer cotangents; with commit also the
// adjoint update, after which the next step follows at once.  Without commit (dynamic scaling: one step per launch, the update waits for
// the finiteness decision) psi_j goes to memory.  With tpart also the block's share of the step's time terms: Phi^T a with
// Phi = sum_j b_j k_j, dt = sum_j dtau_j and dh = sum_j (c_j dtau_j + sum_{l<j} a_jl <psi_j, k_l>), dtau_j = <dZ_1, w_t>.
template <typename T, int MT>
__global__ void __launch_bounds__(kThreads + 32, 1) small_backward_kernel(const __grid_constant__ SmallMlp p) {
    chain_begin();
    using W = typename Pair<T>::W;
    extern __shared__ __align__(16) unsigned char smem[];
    const int R = kRows<T, MT>, r0 = blockIdx.x * R;
    Ring ring = make_ring(smem, p.ring, p.err, p.wait_ns);
    if (threadIdx.x >= kThreads) {
        if (threadIdx.x == kThreads) {
            for (int s = 0; s < p.count; ++s) {
                if (p.recompute)
                    for (int j = 0; j < p.stages; ++j)
                        for (int l = 0; l < p.L; ++l)      // (the last stage's derivative only for the time terms)
                            if (!(l == p.L - 1 && j == p.stages - 1 && p.tpart == nullptr)) stream_layer<T>(ring, p.wf[l], p.wp[l], p.wp[l + 1]);
                if (p.vjp)
                    for (int j = 0; j < p.stages; ++j) {
                        for (int l = p.L - 1; l >= 0; --l) stream_layer<T>(ring, p.wb[l], p.wp[l + 1], p.wp[l]);
                        ring.lost |= p.starve != 0;      // test of the waits: the rest of the weights never comes
                    }
            }
            ring_drain(ring);
        }
        return;
    }
    const SmallSmem<T> sm(p, smem + p.ring * (kUnitBytes + 16), R);
    const int d = sm.d, dp = sm.dp;
    const T* traj = (const T*)p.traj;
    const float lim = low_limit<T>();
    const int e = p.e_dev != nullptr ? *p.e_dev : p.e;
    const bool want_t = p.tpart != nullptr;
    bool bad = false;
    fetch_scalars(p, sm, p.step_hi);
    if (p.vjp) {
        for (int i = threadIdx.x; i < R * dp; i += kThreads) {
            const int r = i / dp, c = i - r * dp;
            sm.a[i] = r0 + r < p.B && c < d ? p.a[(long long)(r0 + r) * d + c] : 0.f;
        }
    }
    for (int s = 0; s < p.count; ++s) {
        const int n = p.step_hi - s;
        scalars_ready();
        work_sync();
        if (s + 1 < p.count) fetch_scalars(p, sm, n - 1);
        const RkStepScalars& sc = sm.scalars(n);
        float t_phi = 0.f, t_dt = 0.f, t_dh = 0.f;
        if (p.recompute) {
            const T* tn = traj + ((long long)n * p.B + r0) * d;
            for (int i = threadIdx.x; i < R * dp; i += kThreads) {
                // (rows behind the batch follow the last one with zero adjoint: from y = 0 they could overflow where no sample does)
                const int r = i / dp, c = i - r * dp, row = r0 + r < p.B ? r : p.B - 1 - r0;
                sm.yb[i] = c < d ? tn[row * d + c] : Low<T>::from_f(0.f);
            }
            work_sync();
            small_stages<T, MT, true>(p, ring, sm, sc, r0, s, !want_t);
        }
        if (!p.vjp) continue;
        for (int i = threadIdx.x; i < sm.pairs; i += kThreads) {       // seed Q16(S a)
            const float2 a = reinterpret_cast<const float2*>(sm.a)[i];
            const float v0 = ldexpf(a.x, e), v1 = ldexpf(a.y, e);
            bad |= !(fabsf(v0) < lim) | !(fabsf(v1) < lim);
            sm.w(sm.vv)[i] = pack_w<T>(v0, v1);
            if (want_t) {
                float p0 = 0.f, p1 = 0.f;
                for (int j = 0; j < p.stages; ++j) {
                    const W k = sm.w(sm.ks)[j * sm.pairs + i];
                    p0 = fmaf(sc.b[j], lo_w<T>(k), p0);
                    p1 = fmaf(sc.b[j], hi_w<T>(k), p1);
                }
                t_phi = fmaf(p0, a.x, fmaf(p1, a.y, t_phi));
            }
        }
        for (int j = p.stages - 1; j >= 0; --j) {
            // kappa_j = Q16(b_j v + sum_{l > j} (h a_lj) psi_l): each thread reads what it wrote itself, or what a barrier lies behind
            float ha[RK_MAX_STAGES];
#pragma unroll
            for (int l = 1; l < RK_MAX_STAGES; ++l) ha[l] = l > j && l < p.stages ? sc.ha[l][j] : 0.f;
            const float bj = sc.b[j], cj = sc.c[j];
            float dtau = 0.f;
            T* kap = (T*)p.zs[p.L] + ((long long)(s * p.stages + j) * p.B + r0) * dp;
            const W* wt = want_t && p.time ? (const W*)p.wt16 : nullptr;
            for (int i = threadIdx.x; i < sm.pairs; i += kThreads) {
                const int r = i / sm.half, c = 2 * (i - r * sm.half);
                const W v = sm.w(sm.vv)[i];
                float v0 = bj * lo_w<T>(v), v1 = bj * hi_w<T>(v);
#pragma unroll
                for (int l = 1; l < RK_MAX_STAGES; ++l)
                    if (ha[l] != 0.f) {
                        const W q = sm.w(sm.ps)[l * sm.pairs + i];
                        v0 = fmaf(ha[l], lo_w<T>(q), v0);
                        v1 = fmaf(ha[l], hi_w<T>(q), v1);
                    }
                bad |= !(fabsf(v0) < lim) | !(fabsf(v1) < lim);
                const W q = pack_w<T>(v0, v1);
                *(W*)(sm.act(0) + r * sm.lda + c) = q;
                if (r0 + r < p.B) *(W*)(kap + r * dp + c) = q;
                if (p.L == 1 && wt != nullptr) {
                    const W w = __ldg(wt + c / 2);
                    dtau = fmaf(lo_w<T>(q), lo_w<T>(w), fmaf(hi_w<T>(q), hi_w<T>(w), dtau));
                }
            }
            zero_tail(sm.act(0), sm.lda, R, dp);
            work_sync();
            int cur = 0;
            for (int l = p.L - 1; l >= 0; --l, cur ^= 1) {
                const int N = p.wp[l];
                const long long at = ((long long)(s * p.stages + j) * p.B + r0) * N;
                const T* H = l > 0 ? (const T*)p.xs[l] + at : nullptr;
                T* Z = l > 0 ? (T*)p.zs[l] + at : (p.commit ? nullptr : (T*)p.psi[j] + (long long)r0 * dp);
                T* dst = l > 0 ? sm.act(cur ^ 1) : sm.ps + j * R * dp;
                const int ld = l > 0 ? sm.lda : dp;
                W hw[kNG][2 * MT];
                block_gemm<T, MT>(
                    ring, sm, sm.act(cur), p.wp[l + 1], N,
                    [&](int g, int q, int r, int c) {      // the stored layer outputs whose activation derivative multiplies the result
                        hw[g][q] = l > 0 && r0 + r < p.B ? *(const W*)(H + (long long)r * N + c) : W{};
                    },
                    [&](int g, int q, int r, int c, float v0, float v1) {
                        if (l > 0) {
                            v0 *= act_df<T>(p.act, lo_w<T>(hw[g][q]));
                            v1 *= act_df<T>(p.act, hi_w<T>(hw[g][q]));
                        }
                        bad |= !(fabsf(v0) < lim) | !(fabsf(v1) < lim);
                        const W w = pack_w<T>(v0, v1);
                        *(W*)(dst + r * ld + c) = w;
                        if (Z != nullptr && r0 + r < p.B) *(W*)(Z + (long long)r * N + c) = w;
                        if (l == 1 && wt != nullptr) {
                            const W t = __ldg(wt + c / 2);
                            dtau = fmaf(lo_w<T>(w), lo_w<T>(t), fmaf(hi_w<T>(w), hi_w<T>(t), dtau));
                        }
                    });
                if (l > 0) zero_tail(dst, sm.lda, R, N);
                work_sync();
            }
            if (want_t) {
                t_dt += dtau;
                t_dh = fmaf(cj, dtau, t_dh);
                for (int l = 0; l < j; ++l) {
                    const float ajl = sc.a[j][l];
                    if (ajl == 0.f) continue;
                    float dot = 0.f;
                    for (int i = threadIdx.x; i < sm.pairs; i += kThreads) {
                        const W q = sm.w(sm.ps)[j * sm.pairs + i], k = sm.w(sm.ks)[l * sm.pairs + i];
                        dot = fmaf(lo_w<T>(q), lo_w<T>(k), fmaf(hi_w<T>(q), hi_w<T>(k), dot));
                    }
                    t_dh = fmaf(ajl, dot, t_dh);
                }
            }
        }
        if (p.commit) {      // a <- a + (h / S) sum_j psi_j (+ running cost)
            const float coef = ldexpf(sc.h, -e);
            for (int i = threadIdx.x; i < sm.pairs; i += kThreads) {
                float d0 = 0.f, d1 = 0.f;
#pragma unroll
                for (int j = RK_MAX_STAGES - 1; j >= 0; --j)
                    if (j < p.stages) {
                        const W q = sm.w(sm.ps)[j * sm.pairs + i];
                        d0 += lo_w<T>(q);
                        d1 += hi_w<T>(q);
                    }
                float2 a = reinterpret_cast<float2*>(sm.a)[i];
                a.x = fmaf(coef, d0, a.x); a.y = fmaf(coef, d1, a.y);
                if (p.cot != nullptr) {
                    const int r = i / sm.half, c = 2 * (i - r * sm.half);
                    const float* ct = p.cot + ((long long)n * p.B + r0 + r) * d + c;
                    if (r0 + r < p.B && c < d) a.x += ct[0];
                    if (r0 + r < p.B && c + 1 < d) a.y += ct[1];
                }
                reinterpret_cast<float2*>(sm.a)[i] = a;
            }
        }
        if (want_t) {      // lanes by shuffles, warps in ascending order
            const int warp = threadIdx.x >> 5;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                t_phi += __shfl_xor_sync(0xffffffffu, t_phi, o);
                t_dt += __shfl_xor_sync(0xffffffffu, t_dt, o);
                t_dh += __shfl_xor_sync(0xffffffffu, t_dh, o);
            }
            if ((threadIdx.x & 31) == 0) { sm.red[warp] = t_phi; sm.red[kWarps + warp] = t_dt; sm.red[2 * kWarps + warp] = t_dh; }
            work_sync();
            if (threadIdx.x < 3) {
                float x = 0.f;
                for (int w = 0; w < kWarps; ++w) x += sm.red[threadIdx.x * kWarps + w];
                p.tpart[((long long)s * gridDim.x + blockIdx.x) * 3 + threadIdx.x] = x;
            }
        }
    }
    if (p.commit) {
        work_sync();
        for (int i = threadIdx.x; i < R * d; i += kThreads) {
            const int r = i / d, c = i - r * d;
            if (r0 + r < p.B) p.a[(long long)r0 * d + i] = sm.a[r * dp + c];
        }
    }
    warp_flag_or(p.flag, bad);
}

// The time terms of the chunk's steps: the blocks' shares added in a fixed order; values {Phi^T a, dt, dh} of the last step to tvals, and
// with tprime the two t' updates of Alg. 2 per step.  Q16(dt), Q16(dh) join the finiteness test.
template <typename T>
__global__ void __launch_bounds__(96) small_time_kernel(SmallMlp p, int blocks) {
    chain_begin();
    __shared__ float v[3];
    const int q = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int s = 0; s < p.count; ++s) {
        float x = 0.f;
        for (int b = lane; b < blocks; b += 32) x += p.tpart[((long long)s * blocks + b) * 3 + q];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        __syncthreads();
        if (lane == 0) v[q] = x;
        __syncthreads();
        if (threadIdx.x != 0) continue;
        const float phi = v[0], dt = v[1], dh = v[2];
        if (p.flag != nullptr && (Low<T>::nonfinite(Low<T>::from_f(dt)) || Low<T>::nonfinite(Low<T>::from_f(dh)))) atomicOr(p.flag, 1u);
        if (p.tvals != nullptr) { p.tvals[0] = phi; p.tvals[1] = dt; p.tvals[2] = dh; }
        if (p.tprime != nullptr) {
            const int n = p.step_hi - s;
            p.tprime[n] = p.tprime[n] + p.coef[s] * (dt - dh) - phi;
            p.tprime[n + 1] = p.tprime[n + 1] + p.coef[s] * dh + phi;
        }
    }
}

constexpr int kSmemCap = 220 * 1024;
// ring buffers that fit beside the block's own shared memory: eight (128 KB ahead) at most, two at least
template <typename T> int ring_buffers(const SmallMlp& p, int rows) {
    const int left = kSmemCap - (int)small_smem<T>(p, rows), n = left / (kUnitBytes + 16);
    return n > 8 ? 8 : n;
}
template <typename K>
bool allow_smem(K kernel, bool (&done)[kMaxDevices]) {
    const int dev = current_device();
    if (!done[dev]) {
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemCap) != cudaSuccess) { cudaGetLastError(); return false; }
        done[dev] = true;
    }
    return true;
}

// row tiles per block: one (16 rows, in float32 8) while that is at most one block per SM, else two (half the weight traffic per row)
int rows_tiles(mpode_dtype dt, int B) {
    const int r = dt == MPODE_F32 ? 8 : 16;
    return (B + r - 1) / r <= sm_count() ? 1 : 2;
}

template <typename T, int MT>
bool forward_t(const SmallMlp& p, cudaStream_t st) {
    static bool done[kMaxDevices] = {false};
    if (!allow_smem(small_forward_kernel<T, MT>, done)) return false;
    SmallMlp q = p;
    q.ring = ring_buffers<T>(p, kRows<T, MT>);
    if (q.ring < 2) return false;
    const int rows = kRows<T, MT>, blocks = (p.B + rows - 1) / rows;
    const size_t smem = small_smem<T>(p, rows) + q.ring * (kUnitBytes + 16);
    launch_chain(small_forward_kernel<T, MT>, dim3(blocks), dim3(kThreads + 32), smem, st, q);
    return true;
}
// (st null, `ready`: only makes the kernel ready for its launch)
template <typename T, int MT>
bool backward_t(const SmallMlp& p, cudaStream_t st, bool ready = false) {
    static bool done[kMaxDevices] = {false};
    if (!allow_smem(small_backward_kernel<T, MT>, done)) return false;
    SmallMlp q = p;
    q.ring = ring_buffers<T>(p, kRows<T, MT>);
    if (q.ring < 2) return false;
    if (ready) return true;
    const int rows = kRows<T, MT>, blocks = (p.B + rows - 1) / rows;
    const size_t smem = small_smem<T>(p, rows) + q.ring * (kUnitBytes + 16);
    launch_chain(small_backward_kernel<T, MT>, dim3(blocks), dim3(kThreads + 32), smem, st, q);
    return true;
}
}  // namespace

size_t small_pack_elems(mpode_dtype dt, int n, int k) {      // columns, reduction
    return dt == MPODE_F32 ? (size_t)n * k : (size_t)(n / 8) * k32(k) * 256;
}
size_t small_pack_bytes(mpode_dtype dt, int L, const int* wp) {
    size_t n = 0;
    for (int l = 0; l < L; ++l) n += small_pack_elems(dt, wp[l + 1], wp[l]) + small_pack_elems(dt, wp[l], wp[l + 1]);
    return n * low_size(dt);
}

// Shared memory draws the first line: a block's rows and three ring buffers have to fit (32-512-512-32 does; a state width of 256 or a hidden width of 1024 does not).  Then the
// weights, since every block streams all of them: training pass of 8 RK4 steps, ms here / other path (fused program; float32: layer by
// layer), bf16 at 200, 1000 and 2300 samples: 128-256-256-128 (128 K weights) 1.03 / 1.65, 1.24 / 1.71, 1.54 / 1.80; 64-384-384-64 (192 K)
// 1.47 / 1.71, 1.66 / 1.77, 1.97 / 1.92; 32-512-512-32 (288 K) 1.77 / 1.74, 2.03 / 1.79, 2.41 / 1.97.  float32 at 64, 500, 1024 and 2300: 64-256-256-64
// (96 K) 2.19 / 3.88, 2.50 / 4.16, 2.90 / 4.45, 5.06 / 6.35; 128-384-384-128 (240 K) 4.42 / 4.47, 4.80 / 5.12, 5.25 / 6.54, 8.93 / 10.5 (the forward pass
// of 64 samples alone 1.39 / 1.15, of 2300 2.17 / 2.75); 64-512-512-64 (320 K) 5.52 / 3.83, 5.98 / 5.15, 6.53 / 7.02, 11.3 / 11.2.  And the batch,
// at one block of two row tiles per SM: with a second round of blocks at 3000 samples, float32, 8.62 / 8.26 (96 K), 16.2 / 11.9 (240 K),
// 20.5 / 14.8 (320 K); the 16-bit forward pass at 4700 0.36 / 0.59 (128 K), 0.54 / 0.61 (192 K), at 8000 see below.
bool small_mlp_supported(mpode_dtype dt, int B, int L, const int* wp) {
    if (L < 1 || L > SMALL_MAX_L) return false;
    SmallMlp p{};
    p.L = L; p.stages = RK_MAX_STAGES;
    long long elems = 0;
    for (int l = 0; l <= L; ++l) { p.wp[l] = p.wr[l] = wp[l]; if (l < L) elems += (long long)wp[l] * wp[l + 1]; }
    if (dt == MPODE_F32) return ring_buffers<float>(p, 16) >= 3 && elems <= 256 * 1024 && B <= 16 * sm_count();
    return ring_buffers<__half>(p, 32) >= 3 && elems <= 160 * 1024 && B <= 32 * sm_count();
}

// The 16-bit backward pass stops at one row tile per SM: its weight gradients grow with the batch and run on the slower matrix
// instructions.  Training pass of 8 RK4 steps, bf16, ms here / tensor-core program (rk_fused.cu): 64-128-64 0.66 / 1.21 at 1000 samples,
// 0.97 / 1.23 at 2300, 1.50 / 1.24 at 4000; 112-336-112 1.46 / 1.52 at 2300, 2.28 / 1.70 at 4000; 128-256-256-128 1.54 / 1.90 at 2300,
// 2.45 / 2.02 at 4000.  The forward pass alone at 4000: 0.16 / 0.37, 0.33 / 0.46, 0.36 / 0.56; at 8000 0.29 / 0.37, 0.62 / 0.47, 0.69 / 0.64.
bool small_backward_supported(mpode_dtype dt, int B) { return dt == MPODE_F32 || rows_tiles(dt, B) == 1; }

int small_blocks(mpode_dtype dt, int B) {
    const int r = (dt == MPODE_F32 ? 8 : 16) * rows_tiles(dt, B);
    return (B + r - 1) / r;
}

void launch_small_pack(mpode_dtype dt, const SmallMlp& p, cudaStream_t st, long long* launches) {
    PackJob job{};
    const int unit = dt == MPODE_F32 ? 1 : 8;                // elements a thread writes
    for (int l = 0; l < p.L; ++l) {
        job.first[2 * l + 1] = job.first[2 * l] + (long long)small_pack_elems(dt, p.wp[l + 1], p.wp[l]) / unit;
        job.first[2 * l + 2] = job.first[2 * l + 1] + (long long)small_pack_elems(dt, p.wp[l], p.wp[l + 1]) / unit;
    }
    long long blocks = (job.first[2 * p.L] + 255) / 256;
    if (blocks > 148 * 4) blocks = 148 * 4;
    if (dt == MPODE_BF16) launch_chain(small_pack_kernel<__nv_bfloat16>, dim3((int)blocks), dim3(256), 0, st, p, job);
    else if (dt == MPODE_F16) launch_chain(small_pack_kernel<__half>, dim3((int)blocks), dim3(256), 0, st, p, job);
    else launch_chain(small_pack_f32_kernel, dim3((int)blocks), dim3(256), 0, st, p, job);
    if (launches) ++*launches;
}

bool launch_small_forward(mpode_dtype dt, const SmallMlp& p, cudaStream_t st, long long* launches) {
    const bool one = rows_tiles(dt, p.B) == 1;
    const bool ok = dt == MPODE_BF16 ? (one ? forward_t<__nv_bfloat16, 1>(p, st) : forward_t<__nv_bfloat16, 2>(p, st))
                  : dt == MPODE_F16  ? (one ? forward_t<__half, 1>(p, st) : forward_t<__half, 2>(p, st))
                                     : (one ? forward_t<float, 1>(p, st) : forward_t<float, 2>(p, st));
    if (ok && launches) ++*launches;
    if (ok && tl_counters) ++tl_counters->fused;
    return ok;
}

bool small_backward_ready(mpode_dtype dt, const SmallMlp& p) {
    if (!small_wgrad_ready(dt, p)) return false;
    if (dt == MPODE_F32) return rows_tiles(dt, p.B) == 1 ? backward_t<float, 1>(p, nullptr, true) : backward_t<float, 2>(p, nullptr, true);
    return dt == MPODE_BF16 ? backward_t<__nv_bfloat16, 1>(p, nullptr, true) : backward_t<__half, 1>(p, nullptr, true);
}

void launch_small_backward(mpode_dtype dt, const SmallMlp& p, cudaStream_t st, long long* launches) {
    if (dt == MPODE_BF16) backward_t<__nv_bfloat16, 1>(p, st);
    else if (dt == MPODE_F16) backward_t<__half, 1>(p, st);
    else if (rows_tiles(dt, p.B) == 1) backward_t<float, 1>(p, st);
    else backward_t<float, 2>(p, st);
    if (launches) ++*launches;
    if (tl_counters) ++tl_counters->fused;
}

void launch_small_time(mpode_dtype dt, const SmallMlp& p, int blocks, cudaStream_t st, long long* launches) {
    if (dt == MPODE_BF16) launch_chain(small_time_kernel<__nv_bfloat16>, dim3(1), dim3(96), 0, st, p, blocks);
    else if (dt == MPODE_F16) launch_chain(small_time_kernel<__half>, dim3(1), dim3(96), 0, st, p, blocks);
    else launch_chain(small_time_kernel<float>, dim3(1), dim3(96), 0, st, p, blocks);
    if (launches) ++*launches;
}

}  // namespace mpode
