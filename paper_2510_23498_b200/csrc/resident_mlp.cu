// Row-local kernels of small dense velocities (16-bit formats) whose weights fit the SM.  A block takes 8 rows per row tile through the
// whole forward solve, or through the backward chain of several steps, and keeps all weights in shared memory, one copy for both directions:
// a weight tile is the first operand of mma.sync (16 output features x 16 inputs), read as it lies for the forward pass and through
// transposing loads for the input gradient.  The rows are the second operand, 8 at a time, so that 1000 samples spread over 125 SMs.
// What bounds a layer is its latency: weights from shared memory (64 wide 8 KB, 200 wide 85 KB at 128 bytes a cycle), a chain of one
// matrix instruction per 16 inputs, the epilogue and one block barrier.  Everything elementwise between two layers (stage input, state
// update, seed, stage cotangent, adjoint update) is done by the thread that holds the values, in the epilogue of the last layer.  Warps
// beside the ones that carry the chain move layer inputs and cotangents to memory, or, where the parameter gradient fits their registers
// and no step's gradient has to be looked at, form it on the spot: then a pass of any number of steps is one launch and a sum over blocks.
#include "resident_mlp.h"

#include "profiler.h"
#include "tc_ptx.cuh"
#include "tensormap.h"

namespace mpode {
using namespace tc;
namespace {

constexpr int kCap = 227 * 1024;                   // shared memory of a block
constexpr int kPieces = 8;                         // pieces of the parameter gradient per warp
constexpr int kPieceWarps = 8;
constexpr int kScalarWords = sizeof(RkStepScalars) / sizeof(float);

__host__ __device__ inline int up16(int w) { return (w + 15) / 16 * 16; }
// warps that carry the chain: 16 features each, one tile per warp up to 256 features
inline int chain_warps(int L, const int* wp) {
    int m = 0;
    for (int l = 0; l <= L; ++l) m = wp[l] > m ? wp[l] : m;
    return m <= 128 ? 8 : 16;
}

template <typename T> __device__ __forceinline__ float lo_of(uint32_t w) { return Low<T>::to_f(from_bits<T>((unsigned short)(w & 0xFFFFu))); }
template <typename T> __device__ __forceinline__ float hi_of(uint32_t w) { return Low<T>::to_f(from_bits<T>((unsigned short)(w >> 16))); }

template <typename T> __device__ __forceinline__ void mma_k16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1);
template <> __device__ __forceinline__ void mma_k16<__half>(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
template <> __device__ __forceinline__ void mma_k16<__nv_bfloat16>(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
template <typename T> __device__ __forceinline__ void mma_k8(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t b0);
template <> __device__ __forceinline__ void mma_k8<__half>(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t b0) {
    asm("mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a0), "r"(a1), "r"(b0));
}
template <> __device__ __forceinline__ void mma_k8<__nv_bfloat16>(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t b0) {
    asm("mma.sync.aligned.m16n8k8.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a0), "r"(a1), "r"(b0));
}
__device__ __forceinline__ void ldm4(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldm4_t(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldm2_t(uint32_t addr, uint32_t& r0, uint32_t& r1) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];" : "=r"(r0), "=r"(r1) : "r"(addr) : "memory");
}
__device__ __forceinline__ void stm2_t(uint32_t addr, uint32_t r0, uint32_t r1) {
    asm volatile("stmatrix.sync.aligned.m8n8.x2.trans.shared.b16 [%0], {%1,%2};" ::"r"(addr), "r"(r0), "r"(r1) : "memory");
}
__device__ __forceinline__ void copy16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void copies_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }

template <typename T> __device__ __forceinline__ float act16(int act, float z) {
    switch (act) {
        case MPODE_ACT_SOFTPLUS: return fast_act<MPODE_ACT_SOFTPLUS>(z);
        case MPODE_ACT_RELU: return fast_act<MPODE_ACT_RELU>(z);
        case MPODE_ACT_TANH: return fast_act<MPODE_ACT_TANH>(z);
        default: return z;
    }
}
template <typename T> __device__ __forceinline__ float act16_d(int act, float h) {
    switch (act) {
        case MPODE_ACT_SOFTPLUS: return fast_act_deriv<MPODE_ACT_SOFTPLUS>(h);
        case MPODE_ACT_RELU: return fast_act_deriv<MPODE_ACT_RELU>(h);
        case MPODE_ACT_TANH: return fast_act_deriv<MPODE_ACT_TANH>(h);
        default: return 1.f;
    }
}

// ---------------------------------------------------------------- the image of the weights
// Layer l: up16(outputs) rows of sw[l] elements (an odd number of 16-byte pieces: eight rows of a matrix load hit eight bank groups),
// zero in the padding; behind all layers the rounded biases and the rounded time column as floats.
template <typename T>
__global__ void __launch_bounds__(256) resident_pack_kernel(const __grid_constant__ ResidentMlp p) {
    chain_begin();
    const SmallMlp& s = p.s;
    const int step = (int)(gridDim.x * blockDim.x), first = (int)(blockIdx.x * blockDim.x + threadIdx.x);
    for (int l = 0; l < s.L; ++l) {
        const int ld = p.g.sw[l], n = up16(s.wp[l + 1]) * ld, in_full = s.wr[l] + ((s.time && l == 0) ? 1 : 0);
        T* dst = (T*)p.image + p.g.w_at[l];
        for (int i = first; i < n; i += step) {
            const int out = i / ld, in = i - out * ld;
            dst[i] = Low<T>::from_f(out < s.wr[l + 1] && in < s.wr[l] ? s.theta[s.woff[l] + (long long)out * in_full + in] : 0.f);
        }
        float* b = (float*)(p.image + (size_t)p.g.w_elems * sizeof(T)) + p.g.b_at[l];
        for (int c = first; c < up16(s.wp[l + 1]); c += step) {
            const bool on = c < s.wr[l + 1];
            b[c] = s.bias && on ? Low<T>::to_f(Low<T>::from_f(s.theta[s.boff[l] + c])) : 0.f;
            if (l == 0)
                ((float*)(p.image + (size_t)p.g.w_elems * sizeof(T)))[p.g.t_at + c] =
                    s.time && on ? Low<T>::to_f(Low<T>::from_f(s.theta[s.woff[0] + (long long)c * (s.wr[0] + 1) + s.wr[0]])) : 0.f;
        }
    }
}

// ---------------------------------------------------------------- shared memory
// Behind the image: the rows' buffers (R rows of sw[l] elements each), then the chain threads' slots and the steps' scalars.  Columns
// behind a width stay zero from the start to the end: tiles and copies write whole widths only, and the upper half of a tile that ends at a
// multiple of 8 is written as zeros.
inline ResidentBufs plan_bufs(const ResidentPlan& g, int L, int stages, int R, bool back) {
    ResidentBufs b;
    b.state = R * g.sw[0] * 2;
    int at = b.z0 = g.image_bytes;
    at += 2 * b.state;
    for (int l = 1; l < L; ++l) { b.z[l] = at; at += R * g.sw[l] * 2; }
    if (back) {
        b.x00 = at; at += 2 * b.state;
        for (int l = 0; l < L; ++l) { b.keep_at[l] = b.keep_stage; b.keep_stage += R * g.sw[l] * 2; }
        b.keep = at;
        at += b.keep_stage * stages;
    }
    b.slots = at + 32;      // (the last matrix load of an odd number of reduction steps reads 16 bytes past a row)
    return b;
}
// pieces of 8 inputs in a layer's parameter gradient; the bias and time columns are one more
__host__ __device__ inline int piece_columns(int inputs, bool sums) { return inputs / 8 + (sums ? 1 : 0); }
// [image][buffers][slots: `slots` words for each of the state tiles' threads][scalars of two steps][sums of the time terms]
inline size_t resident_smem(const ResidentPlan& g, int L, int wp0, int stages, int mt, bool back) {
    const int owners = up16(wp0) / 16 * 32;
    return plan_bufs(g, L, stages, 8 * mt, back).slots + (size_t)(back ? 2 : 1) * stages * 2 * mt * owners * 4 + 2 * kScalarWords * 4 + 3 * 16 * 4 + 16;
}

// One tile of 16 features for the block's 8 MT rows: acc[m][0, 1] = feature g of rows 2t, 2t + 1 (g = lane / 4, t = lane % 4), acc[m][2, 3]
// feature g + 8.  `w`: this lane's address in the weights, advanced by wstep per 16 of the reduction; `x`: in the rows' buffer.
template <typename T, int MT, bool BACK>
__device__ __forceinline__ void tile_product(float (&acc)[MT][4], uint32_t w, uint32_t wstep, uint32_t x, uint32_t xrow8, int ks) {
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[m][i] = 0.f;
    int k = 0;
    constexpr int G = MT <= 2 ? 4 : 2;      // reduction steps whose operands are requested together
#pragma unroll 1
    for (; k + G <= ks; k += G) {
        uint32_t a[G][4], b[G / 2][MT][4];
#pragma unroll
        for (int q = 0; q < G; ++q) {
            if (BACK) ldm4_t(w + q * wstep, a[q]); else ldm4(w + q * wstep, a[q]);
        }
#pragma unroll
        for (int q = 0; q < G / 2; ++q)
#pragma unroll
            for (int m = 0; m < MT; ++m) ldm4(x + q * 64 + m * xrow8, b[q][m]);
        w += G * wstep; x += G * 32;
#pragma unroll
        for (int q = 0; q < G; ++q)
#pragma unroll
            for (int m = 0; m < MT; ++m) mma_k16<T>(acc[m], a[q], b[q >> 1][m][2 * (q & 1)], b[q >> 1][m][2 * (q & 1) + 1]);
    }
#pragma unroll 1
    for (; k < ks; k += 2) {
        uint32_t a[2][4], b[MT][4];
#pragma unroll
        for (int m = 0; m < MT; ++m) ldm4(x + m * xrow8, b[m]);
        if (BACK) ldm4_t(w, a[0]); else ldm4(w, a[0]);
        if (k + 1 < ks) { if (BACK) ldm4_t(w + wstep, a[1]); else ldm4(w + wstep, a[1]); }
        w += 2 * wstep; x += 64;
#pragma unroll
        for (int m = 0; m < MT; ++m) mma_k16<T>(acc[m], a[0], b[m][0], b[m][1]);
        if (k + 1 < ks) {
#pragma unroll
            for (int m = 0; m < MT; ++m) mma_k16<T>(acc[m], a[1], b[m][2], b[m][3]);
        }
    }
}

// Everything a thread of the chain knows about its place
template <typename T, int MT>
struct Lane {
    int warp, lane, g, t;
    uint32_t xo8, xoff;                // lane's row and column offsets of matrix loads: rows' operand
    __device__ Lane() {
        warp = threadIdx.x >> 5; lane = threadIdx.x & 31; g = lane >> 2; t = lane & 3;
    }
    // rows' operand: row = lane % 8, 8 columns per group of 8 lanes
    __device__ __forceinline__ uint32_t x_at(uint32_t buf, int sx) const { return buf + (uint32_t)(((lane & 7) * sx + (lane >> 3) * 8) * 2); }
    __device__ __forceinline__ uint32_t w_fwd(uint32_t w, int sw, int f0) const { return w + (uint32_t)(((f0 + (lane & 15)) * sw + (lane >> 4) * 8) * 2); }
    __device__ __forceinline__ uint32_t w_bwd(uint32_t w, int sw, int f0) const {
        return w + (uint32_t)((((lane & 7) + (lane >> 4) * 8) * sw + f0 + ((lane >> 3) & 1) * 8) * 2);
    }
    // a tile's values as they lie in a rows' buffer: row = lane % 8, 8 columns for each of the two halves
    __device__ __forceinline__ uint32_t frag_at(uint32_t buf, int sx, int f0, int m) const {
        return buf + (uint32_t)(((m * 8 + (lane & 7)) * sx + f0 + ((lane >> 3) & 1) * 8) * 2);
    }
};

// the next layer's input of a tile (or the next stage's): packed pairs of rows, the half behind the width as zeros
template <int MT, typename P>
__device__ __forceinline__ void put_tile(const P& ln, uint32_t buf, int sx, int f0, int width, const uint32_t (&v)[MT][2]) {
#pragma unroll
    for (int m = 0; m < MT; ++m) stm2_t(ln.frag_at(buf, sx, f0, m), v[m][0], f0 + 8 < width ? v[m][1] : 0u);
}

// R rows of `width` elements between a rows' buffer and memory ([B][width], rows from r0), 16 bytes at a time
template <typename T>
__device__ __forceinline__ void rows_out(uint32_t buf, int sx, T* dst, int width, int R, int r0, int B, int tid, int threads) {
    const int per = width / 8, n = R * per;
    for (int i = tid; i < n; i += threads) {
        const int r = i / per, c = (i - r * per) * 8;
        if (r0 + r >= B) continue;
        const uint4 v = lds128(buf + (uint32_t)((r * sx + c) * 2));
        *reinterpret_cast<uint4*>(dst + (long long)(r0 + r) * width + c) = v;
    }
}
// the stored state: rows of d elements, of any parity
template <typename T>
__device__ __forceinline__ void state_out(uint32_t buf, int sx, T* dst, int d, int R, int r0, int B, int tid, int threads) {
    if ((d & 7) == 0) { rows_out<T>(buf, sx, dst, d, R, r0, B, tid, threads); return; }
    for (int i = tid; i < R * d; i += threads) {
        const int r = i / d, c = i - r * d;
        unsigned short v;
        asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(buf + (uint32_t)((r * sx + c) * 2)));
        if (r0 + r < B) reinterpret_cast<unsigned short*>(dst)[(long long)(r0 + r) * d + c] = v;
    }
}
template <typename T>
__device__ __forceinline__ void state_in(uint32_t buf, int sx, const T* src, int d, int R, int r0, int B, int tid, int threads) {
    if ((d & 7) == 0) {
        const int per = d / 8, n = R * per;
        for (int i = tid; i < n; i += threads) {
            const int r = i / per, c = (i - r * per) * 8;
            if (r0 + r < B) copy16(buf + (uint32_t)((r * sx + c) * 2), src + (long long)(r0 + r) * d + c);
        }
        return;
    }
    for (int i = tid; i < R * d; i += threads) {
        const int r = i / d, c = i - r * d;
        if (r0 + r < B) {
            const unsigned short v = reinterpret_cast<const unsigned short*>(src)[(long long)(r0 + r) * d + c];
            asm volatile("st.shared.u16 [%0], %1;" ::"r"(buf + (uint32_t)((r * sx + c) * 2)), "h"(v) : "memory");
        }
    }
}

// image into shared memory, buffers zeroed, first step's scalars
__device__ __forceinline__ void load_image(const ResidentMlp& p, unsigned char* smem) {
    for (int i = threadIdx.x; i < p.g.image_bytes / 16; i += blockDim.x) copy16(smem_u32(smem) + (uint32_t)i * 16u, p.image + (size_t)i * 16);
    for (int i = p.b.z0 + threadIdx.x * 16; i < p.b.slots; i += blockDim.x * 16) sts128(smem_u32(smem) + (uint32_t)i, 0u, 0u, 0u, 0u);
}
__device__ __forceinline__ void copy_scalars(float* dst, const RkStepScalars* src, int tid) {
    if (tid < kScalarWords) dst[tid] = ((const float*)src)[tid];
}

// A hidden layer: H = Q16(act(W x + b + tau w_t)) of the block's rows
template <typename T, int MT, int NW>
__device__ __forceinline__ void hidden_layer(const ResidentMlp& p, const Lane<T, MT>& ln, uint32_t wimg, const float* fl, int l, float tau, uint32_t in, uint32_t out) {
    const SmallMlp& s = p.s;
    const int K = up16(s.wp[l]) / 16, N = s.wp[l + 1], sx = p.g.sw[l];
    const uint32_t w = wimg + (uint32_t)p.g.w_at[l] * 2u, x = ln.x_at(in, sx);
    const bool time = s.time && l == 0;
    for (int f0 = ln.warp * 16; f0 < N; f0 += NW * 16) {
        float bA = fl[p.g.b_at[l] + f0 + ln.g], bB = fl[p.g.b_at[l] + f0 + 8 + ln.g];
        if (time) { bA = fmaf(tau, fl[p.g.t_at + f0 + ln.g], bA); bB = fmaf(tau, fl[p.g.t_at + f0 + 8 + ln.g], bB); }
        float acc[MT][4];
        tile_product<T, MT, false>(acc, ln.w_fwd(w, p.g.sw[l], f0), 32u, x, (uint32_t)(16 * sx), K);
        uint32_t v[MT][2];
#pragma unroll
        for (int m = 0; m < MT; ++m) {
            v[m][0] = cvt_pack<T>(act16<T>(s.act, acc[m][0] + bA), act16<T>(s.act, acc[m][1] + bA));
            v[m][1] = cvt_pack<T>(act16<T>(s.act, acc[m][2] + bB), act16<T>(s.act, acc[m][3] + bB));
        }
        put_tile<MT>(ln, out, p.g.sw[l + 1], f0, N, v);
    }
}

// ---------------------------------------------------------------- forward
template <typename T, int MT, int NW>
__global__ void __launch_bounds__(NW * 32 + 64, 1) resident_forward_kernel(const __grid_constant__ ResidentMlp p) {
    chain_begin();
    extern __shared__ __align__(16) unsigned char smem[];
    const SmallMlp& s = p.s;
    constexpr int R = 8 * MT;
    const int r0 = blockIdx.x * R, d = s.wr[0], L = s.L, S = s.stages;
    const uint32_t base = smem_u32(smem);
    auto z0_at = [&](int q) -> uint32_t { return base + (uint32_t)(p.b.z0 + q * p.b.state); };
    auto z_at = [&](int l) -> uint32_t { return base + (uint32_t)p.b.z[l]; };
    const int tiles0 = up16(s.wp[0]) / 16, owners = tiles0 * 32;
    uint32_t* slots = (uint32_t*)(smem + p.b.slots);
    float* scal = (float*)(slots + S * 2 * MT * owners);
    const float* fl = (const float*)(smem + (size_t)p.g.w_elems * sizeof(T));
    load_image(p, smem);
    copy_scalars(scal, s.scal, threadIdx.x);
    T* traj = (T*)s.traj;
    __syncthreads();
    if (threadIdx.x >= NW * 32) {          // scalars of the next step, the stored state of this one
        const int tid = threadIdx.x - NW * 32;
        copies_done();
        __syncthreads();
        int cur = 0;
        for (int n = 0; n < s.n_steps; ++n) {
            if (n + 1 < s.n_steps) copy_scalars(scal + ((n + 1) & 1) * kScalarWords, s.scal + n + 1, tid);
            for (int j = 0; j < S; ++j) {
                if (j == 0) state_out<T>(z0_at(cur), p.g.sw[0], traj + (long long)n * s.B * d, d, R, r0, s.B, tid, 64);
                for (int l = 0; l < L; ++l) __syncthreads();
                cur ^= 1;
            }
        }
        state_out<T>(z0_at(cur), p.g.sw[0], traj + (long long)s.n_steps * s.B * d, d, R, r0, s.B, tid, 64);
        return;
    }
    const Lane<T, MT> ln;
    const bool owner = ln.warp < tiles0;
    const int f0 = ln.warp * 16;
    uint32_t* ks = slots + threadIdx.x;            // k_j of this thread's values: word (2 MT j + 2 m + h) * owners
    float y[MT][4];
    uint32_t yb[MT][2];
    if (owner) {
#pragma unroll
        for (int m = 0; m < MT; ++m) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int r = r0 + m * 8 + 2 * ln.t + (i & 1), c = f0 + ln.g + (i >> 1) * 8;
                y[m][i] = r < s.B && c < d ? s.y0[(long long)r * d + c] : 0.f;
            }
            yb[m][0] = cvt_pack<T>(y[m][0], y[m][1]);
            yb[m][1] = cvt_pack<T>(y[m][2], y[m][3]);
        }
        put_tile<MT>(ln, z0_at(0), p.g.sw[0], f0, s.wp[0], yb);
    }
    copies_done();
    __syncthreads();
    int cur = 0;
    for (int n = 0; n < s.n_steps; ++n) {
        const RkStepScalars& sc = *(const RkStepScalars*)(scal + (n & 1) * kScalarWords);
        for (int j = 0; j < S; ++j) {
            const float tau = sc.tau16[j];
            for (int l = 0; l + 1 < L; ++l) {
                hidden_layer<T, MT, NW>(p, ln, base, fl, l, tau, l == 0 ? z0_at(cur) : z_at(l), z_at(l + 1));
                __syncthreads();
            }
            if (owner) {
                const int l = L - 1, K = up16(s.wp[l]) / 16, sx = p.g.sw[l];
                const bool last = j + 1 == S;
                // the terms of what follows that do not depend on this stage
                float v[MT][4];
#pragma unroll
                for (int m = 0; m < MT; ++m)
#pragma unroll
                    for (int i = 0; i < 4; ++i) v[m][i] = last ? 0.f : ((i & 1) ? hi_of<T>(yb[m][i >> 1]) : lo_of<T>(yb[m][i >> 1]));
                for (int q = 0; q < j; ++q) {
                    const float c = last ? sc.hb[q] : sc.ha[j + 1][q];
                    if (!last && c == 0.f) continue;
#pragma unroll
                    for (int m = 0; m < MT; ++m)
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const uint32_t k = ks[((q * MT + m) * 2 + h) * owners];
                            v[m][2 * h] = fmaf(c, lo_of<T>(k), v[m][2 * h]);
                            v[m][2 * h + 1] = fmaf(c, hi_of<T>(k), v[m][2 * h + 1]);
                        }
                }
                float bA = fl[p.g.b_at[l] + f0 + ln.g], bB = fl[p.g.b_at[l] + f0 + 8 + ln.g];
                if (s.time && l == 0) { bA = fmaf(tau, fl[p.g.t_at + f0 + ln.g], bA); bB = fmaf(tau, fl[p.g.t_at + f0 + 8 + ln.g], bB); }
                const float c = last ? sc.hb[j] : sc.ha[j + 1][j];
                float acc[MT][4];
                tile_product<T, MT, false>(acc, ln.w_fwd(base + (uint32_t)p.g.w_at[l] * 2u, p.g.sw[l], f0), 32u, ln.x_at(l == 0 ? z0_at(cur) : z_at(l), sx),
                                           (uint32_t)(16 * sx), K);
                uint32_t o[MT][2];
#pragma unroll
                for (int m = 0; m < MT; ++m) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const float b = h ? bB : bA;
                        const uint32_t k = cvt_pack<T>(acc[m][2 * h] + b, acc[m][2 * h + 1] + b);
                        ks[((j * MT + m) * 2 + h) * owners] = k;
                        if (last || c != 0.f) {
                            v[m][2 * h] = fmaf(c, lo_of<T>(k), v[m][2 * h]);
                            v[m][2 * h + 1] = fmaf(c, hi_of<T>(k), v[m][2 * h + 1]);
                        }
                        if (last) {
#pragma unroll
                            for (int i = 2 * h; i < 2 * h + 2; ++i) y[m][i] += s.round_increment ? sc.h * Low<T>::to_f(Low<T>::from_f(v[m][i])) : v[m][i];
                            yb[m][h] = cvt_pack<T>(y[m][2 * h], y[m][2 * h + 1]);
                        }
                        o[m][h] = last ? yb[m][h] : cvt_pack<T>(v[m][2 * h], v[m][2 * h + 1]);
                    }
                }
                put_tile<MT>(ln, z0_at(cur ^ 1), p.g.sw[0], f0, s.wp[0], o);
            }
            __syncthreads();
            cur ^= 1;
        }
    }
    if (owner) {
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int r = r0 + m * 8 + 2 * ln.t + (i & 1), c = f0 + ln.g + (i >> 1) * 8;
                if (r < s.B && c < d) s.yT[(long long)r * d + c] = y[m][i];
            }
    }
}

// ---------------------------------------------------------------- backward
// The chain of `count` steps (recompute, seed, stage and layer cotangents, with commit the adjoint update), as small_backward_kernel
// describes it; with REG the parameter gradient of the block's rows beside it, in the registers of eight warps, pieces of 16 x 8: a step's
// sums first, then g += (h / S) dg in float32.
template <typename T, int MT, int NW, bool REG>
__global__ void __launch_bounds__(NW * 32 + (REG ? kPieceWarps * 32 : 128), 1) resident_backward_kernel(const __grid_constant__ ResidentMlp p) {
    chain_begin();
    extern __shared__ __align__(16) unsigned char smem[];
    const SmallMlp& s = p.s;
    constexpr int R = 8 * MT;
    const int r0 = blockIdx.x * R, d = s.wr[0], L = s.L, S = s.stages, B = s.B;
    const uint32_t base = smem_u32(smem);
    auto z0_at = [&](int q) -> uint32_t { return base + (uint32_t)(p.b.z0 + q * p.b.state); };
    auto z_at = [&](int l) -> uint32_t { return base + (uint32_t)p.b.z[l]; };
    auto x00_at = [&](int q) -> uint32_t { return base + (uint32_t)(p.b.x00 + q * p.b.state); };
    auto keep_at = [&](int j, int l) -> uint32_t { return base + (uint32_t)(p.b.keep + j * p.b.keep_stage + p.b.keep_at[l]); };
    const int tiles0 = up16(s.wp[0]) / 16, owners = tiles0 * 32;
    uint32_t* slots = (uint32_t*)(smem + p.b.slots);
    float* scal = (float*)(slots + 2 * S * 2 * MT * owners);
    float* red = scal + 2 * kScalarWords;
    const float* fl = (const float*)(smem + (size_t)p.g.w_elems * sizeof(T));
    const T* traj = (const T*)s.traj;
    const bool want_t = s.tpart != nullptr;
    load_image(p, smem);
    copy_scalars(scal, s.scal + s.step_hi, threadIdx.x);
    __syncthreads();
    if (s.recompute) state_in<T>(x00_at(0), p.g.sw[0], traj + (long long)s.step_hi * B * d, d, R, r0, B, threadIdx.x, blockDim.x);
    else
        for (int j = 0; j < S; ++j)      // the layer outputs of a recompute launch
            for (int l = 1; l < L; ++l)
                state_in<T>(keep_at(j, l), p.g.sw[l], (const T*)s.xs[l] + (long long)j * B * s.wp[l], s.wp[l], R, r0, B, threadIdx.x,
                            blockDim.x);
    copies_done();
    __syncthreads();
    auto x0_of = [&](int st, int j) -> uint32_t { return j == 0 ? x00_at(st & 1) : keep_at(j, 0); };
    auto x_of = [&](int st, int j, int l) -> uint32_t { return l == 0 ? x0_of(st, j) : keep_at(j, l); };
    if (threadIdx.x >= NW * 32) {
        const int tid = threadIdx.x - NW * 32, threads = blockDim.x - NW * 32, warp = tid >> 5, lane = tid & 31;
        // REG: this warp's pieces, (layer, first output, first input or -1 for bias and time)
        int piece[kPieces] = {};      // layer << 20 | output << 10 | input, -1: none
        auto pl = [&](int i) { return piece[i] >> 20; };
        auto pm = [&](int i) { return piece[i] >> 10 & 0x3FF; };
        auto pn = [&](int i) { return (piece[i] & 0x3FF) == 0x3FF ? -1 : piece[i] & 0x3FF; };
        float acc[kPieces][4], tot[kPieces][4];
        if (REG) {
#pragma unroll
            for (int i = 0; i < kPieces; ++i) {
                piece[i] = -1;
                int id = warp + kPieceWarps * i;
                for (int l = 0; l < L && id >= 0; ++l) {
                    const int tm = up16(s.wp[l + 1]) / 16, tn = piece_columns(s.wp[l], s.bias || (s.time && l == 0));
                    if (id < tm * tn) piece[i] = l << 20 | (id / tn * 16) << 10 | (id % tn * 8 < s.wp[l] ? id % tn * 8 : 0x3FF);
                    id -= tm * tn;
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[i][q] = tot[i][q] = 0.f;
            }
        }
        for (int st = 0; st < s.count; ++st) {
            const int n = s.step_hi - st;
            copies_done();
            __syncthreads();
            if (st + 1 < s.count) {
                copy_scalars(scal + ((st + 1) & 1) * kScalarWords, s.scal + n - 1, tid);
                if (s.recompute) state_in<T>(x00_at((st + 1) & 1), p.g.sw[0], traj + (long long)(n - 1) * B * d, d, R, r0, B, tid, threads);
            }
            if (s.recompute) {
                for (int j = 0; j < S; ++j)
                    for (int l = 0; l < L; ++l) {
                        if (!REG) rows_out<T>(x_of(st, j, l), p.g.sw[l], (T*)s.xs[l] + (long long)(st * S + j) * B * s.wp[l], s.wp[l], R, r0, B, tid, threads);
                        if (l == L - 1 && j == S - 1 && !want_t) break;
                        __syncthreads();
                    }
            }
            if (!s.vjp) continue;
            const RkStepScalars& sc = *(const RkStepScalars*)(scal + (st & 1) * kScalarWords);
            int par = 0;
            for (int j = S - 1; j >= 0; --j, par ^= 1)
                for (int l = L - 1; l >= 0; --l) {
                    const uint32_t z = l == L - 1 ? z0_at(par) : z_at(l + 1);
                    const int sz = p.g.sw[l + 1];
                    if (!REG) {
                        rows_out<T>(z, sz, (T*)s.zs[l + 1] + (long long)(st * S + j) * B * s.wp[l + 1], s.wp[l + 1], R, r0, B, tid, threads);
                    } else {
                        const uint32_t x = x_of(st, j, l);
                        const int sx = p.g.sw[l];
                        uint32_t ones = 0u;      // column 0: ones, column 1: the rounded stage time
                        if ((lane >> 2) == 0) ones = cvt_pack<T>(1.f, 1.f);
                        else if ((lane >> 2) == 1 && s.time && l == 0) ones = cvt_pack<T>(sc.tau16[j], sc.tau16[j]);
#pragma unroll
                        for (int i = 0; i < kPieces; ++i) {
                            if (pl(i) != l) continue;
                            const int n0 = pn(i) < 0 ? 0 : pn(i);
                            if constexpr (MT == 1) {
                                uint32_t f[4];      // both halves of the outputs, then the inputs (twice)
                                const int q = lane >> 3;
                                ldm4_t(q < 2 ? z + (uint32_t)(((lane & 7) * sz + pm(i) + q * 8) * 2) : x + (uint32_t)(((lane & 7) * sx + n0) * 2), f);
                                mma_k8<T>(acc[i], f[0], f[1], pn(i) < 0 ? ones : f[2]);
                            } else {
                                static_assert(!REG || MT <= 2, "16 rows at most");
                                uint32_t a[4], b0, b1;
                                ldm4_t(z + (uint32_t)((((lane & 7) + (lane >> 4) * 8) * sz + pm(i) + ((lane >> 3) & 1) * 8) * 2), a);
                                ldm2_t(x + (uint32_t)((((lane & 7) + ((lane >> 3) & 1) * 8) * sx + n0) * 2), b0, b1);
                                mma_k16<T>(acc[i], a, pn(i) < 0 ? ones : b0, pn(i) < 0 ? ones : b1);
                            }
                        }
                    }
                    __syncthreads();
                }
            if (REG) {
                const float cf = ldexpf(sc.h, -s.e);
#pragma unroll
                for (int i = 0; i < kPieces; ++i)
#pragma unroll
                    for (int q = 0; q < 4; ++q) { tot[i][q] = fmaf(cf, acc[i][q], tot[i][q]); acc[i][q] = 0.f; }
            }
            if (want_t) __syncthreads();
        }
        if (REG) {
            float* out = p.partial + (long long)blockIdx.x * p.g.params;
#pragma unroll
            for (int i = 0; i < kPieces; ++i) {
                const int l = pl(i);
                if (l < 0) continue;
                const bool time = s.time && l == 0;
                const int in_full = s.wr[l] + (time ? 1 : 0);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int m = pm(i) + (lane >> 2) + (q >> 1) * 8, c = 2 * (lane & 3) + (q & 1);
                    if (m >= s.wr[l + 1]) continue;
                    if (pn(i) >= 0) { if (pn(i) + c < s.wr[l]) out[s.woff[l] + (long long)m * in_full + pn(i) + c] = tot[i][q]; }
                    else if (c == 0 && s.bias) out[s.boff[l] + m] = tot[i][q];
                    else if (c == 1 && time) out[s.woff[l] + (long long)m * in_full + s.wr[l]] = tot[i][q];
                }
            }
        }
        return;
    }
    // ---- the chain
    const Lane<T, MT> ln;
    const bool owner = ln.warp < tiles0;
    const int f0 = ln.warp * 16;
    uint32_t* ks = slots + threadIdx.x;                                // k_j and psi_j of this thread's values
    uint32_t* ps = ks + S * 2 * MT * owners;
    const float lim = OverflowLimit<T>::value();
    const int e = s.e_dev != nullptr ? *s.e_dev : s.e;
    bool bad = false;
    auto note = [&](float x, float yv) { bad |= !(fabsf(x) < lim) | !(fabsf(yv) < lim); };
    float a[MT][4];
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int r = r0 + m * 8 + 2 * ln.t + (i & 1), c = f0 + ln.g + (i >> 1) * 8;
            a[m][i] = owner && s.vjp && r < B && c < d ? s.a[(long long)r * d + c] : 0.f;
        }
    for (int st = 0; st < s.count; ++st) {
        const int n = s.step_hi - st;
        const RkStepScalars& sc = *(const RkStepScalars*)(scal + (st & 1) * kScalarWords);
        uint32_t vv[MT][2];
        float t_phi = 0.f, t_dt = 0.f, t_dh = 0.f;
        // seed Q16(S a); kappa_j = Q16(b_j v + sum_{l > j} (h a_lj) psi_l), into the rows' buffer of its parity
        auto put_kappa = [&](int j, int par, float& dtau) {
            float ha[RK_MAX_STAGES];
#pragma unroll
            for (int l = 1; l < RK_MAX_STAGES; ++l) ha[l] = l > j && l < S ? sc.ha[l][j] : 0.f;
            const float bj = sc.b[j];
            float wA = 0.f, wB = 0.f;
            if (want_t && L == 1 && s.time) { wA = fl[p.g.t_at + f0 + ln.g]; wB = fl[p.g.t_at + f0 + 8 + ln.g]; }
            uint32_t o[MT][2];
#pragma unroll
            for (int m = 0; m < MT; ++m)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float v0 = bj * lo_of<T>(vv[m][h]), v1 = bj * hi_of<T>(vv[m][h]);
#pragma unroll
                    for (int l = 1; l < RK_MAX_STAGES; ++l)
                        if (ha[l] != 0.f) {
                            const uint32_t q = ps[((l * MT + m) * 2 + h) * owners];
                            v0 = fmaf(ha[l], lo_of<T>(q), v0);
                            v1 = fmaf(ha[l], hi_of<T>(q), v1);
                        }
                    note(v0, v1);
                    o[m][h] = cvt_pack<T>(v0, v1);
                    const float wt = h ? wB : wA;
                    dtau = fmaf(lo_of<T>(o[m][h]), wt, fmaf(hi_of<T>(o[m][h]), wt, dtau));
                }
            put_tile<MT>(ln, z0_at(par), p.g.sw[0], f0, s.wp[0], o);
        };
        float dtau_k = 0.f;                // (one layer: of the cotangent in the buffer)
        if (s.vjp && owner) {
#pragma unroll
            for (int m = 0; m < MT; ++m)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float v0 = ldexpf(a[m][2 * h], e), v1 = ldexpf(a[m][2 * h + 1], e);
                    note(v0, v1);
                    vv[m][h] = cvt_pack<T>(v0, v1);
                }
            put_kappa(S - 1, 0, dtau_k);
        }
        __syncthreads();
        if (s.recompute) {
            uint32_t yb[MT][2];
            if (owner) {
#pragma unroll
                for (int m = 0; m < MT; ++m) ldm2_t(ln.frag_at(x00_at(st & 1), p.g.sw[0], f0, m), yb[m][0], yb[m][1]);
            }
            for (int j = 0; j < S; ++j) {
                const float tau = sc.tau16[j];
                for (int l = 0; l < L; ++l) {
                    const bool last = l == L - 1;
                    if (last && j == S - 1 && !want_t) break;
                    if (!last) {
                        hidden_layer<T, MT, NW>(p, ln, base, fl, l, tau, x_of(st, j, l), x_of(st, j, l + 1));
                    } else if (owner) {
                        const int K = up16(s.wp[l]) / 16, sx = p.g.sw[l];
                        const bool next = j + 1 < S;
                        float v[MT][4];
#pragma unroll
                        for (int m = 0; m < MT; ++m)
#pragma unroll
                            for (int i = 0; i < 4; ++i) v[m][i] = (i & 1) ? hi_of<T>(yb[m][i >> 1]) : lo_of<T>(yb[m][i >> 1]);
                        for (int q = 0; q < j && next; ++q) {
                            const float c = sc.ha[j + 1][q];
                            if (c == 0.f) continue;
#pragma unroll
                            for (int m = 0; m < MT; ++m)
#pragma unroll
                                for (int h = 0; h < 2; ++h) {
                                    const uint32_t k = ks[((q * MT + m) * 2 + h) * owners];
                                    v[m][2 * h] = fmaf(c, lo_of<T>(k), v[m][2 * h]);
                                    v[m][2 * h + 1] = fmaf(c, hi_of<T>(k), v[m][2 * h + 1]);
                                }
                        }
                        float bA = fl[p.g.b_at[l] + f0 + ln.g], bB = fl[p.g.b_at[l] + f0 + 8 + ln.g];
                        if (s.time && l == 0) { bA = fmaf(tau, fl[p.g.t_at + f0 + ln.g], bA); bB = fmaf(tau, fl[p.g.t_at + f0 + 8 + ln.g], bB); }
                        const float c = next ? sc.ha[j + 1][j] : 0.f;
                        float acc[MT][4];
                        tile_product<T, MT, false>(acc, ln.w_fwd(base + (uint32_t)p.g.w_at[l] * 2u, p.g.sw[l], f0), 32u, ln.x_at(x_of(st, j, l), sx), (uint32_t)(16 * sx), K);
                        uint32_t o[MT][2];
#pragma unroll
                        for (int m = 0; m < MT; ++m)
#pragma unroll
                            for (int h = 0; h < 2; ++h) {
                                const float b = h ? bB : bA;
                                const uint32_t k = cvt_pack<T>(acc[m][2 * h] + b, acc[m][2 * h + 1] + b);
                                ks[((j * MT + m) * 2 + h) * owners] = k;
                                if (c != 0.f) {
                                    v[m][2 * h] = fmaf(c, lo_of<T>(k), v[m][2 * h]);
                                    v[m][2 * h + 1] = fmaf(c, hi_of<T>(k), v[m][2 * h + 1]);
                                }
                                o[m][h] = cvt_pack<T>(v[m][2 * h], v[m][2 * h + 1]);
                            }
                        if (next) put_tile<MT>(ln, x0_of(st, j + 1), p.g.sw[0], f0, s.wp[0], o);
                    }
                    __syncthreads();
                }
            }
        }
        if (!s.vjp) continue;
        if (want_t && owner) {
#pragma unroll
            for (int m = 0; m < MT; ++m)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float p0 = 0.f, p1 = 0.f;
                    for (int j = 0; j < S; ++j) {
                        const uint32_t k = ks[((j * MT + m) * 2 + h) * owners];
                        p0 = fmaf(sc.b[j], lo_of<T>(k), p0);
                        p1 = fmaf(sc.b[j], hi_of<T>(k), p1);
                    }
                    t_phi = fmaf(p0, a[m][2 * h], fmaf(p1, a[m][2 * h + 1], t_phi));
                }
        }
        int par = 0;
        for (int j = S - 1; j >= 0; --j, par ^= 1) {
            float dtau = dtau_k;
            dtau_k = 0.f;
            for (int l = L - 1; l >= 0; --l) {
                const uint32_t z = l == L - 1 ? z0_at(par) : z_at(l + 1);
                const int K = up16(s.wp[l + 1]) / 16, sz = p.g.sw[l + 1], sw = p.g.sw[l];
                const uint32_t w = base + (uint32_t)p.g.w_at[l] * 2u, zx = ln.x_at(z, sz);
                if (l > 0) {
                    const int N = s.wp[l];
                    const uint32_t H = x_of(st, j, l);
                    for (int n0 = ln.warp * 16; n0 < N; n0 += NW * 16) {
                        uint32_t hv[MT][2];
#pragma unroll
                        for (int m = 0; m < MT; ++m) ldm2_t(ln.frag_at(H, sw, n0, m), hv[m][0], hv[m][1]);
                        float acc[MT][4];
                        tile_product<T, MT, true>(acc, ln.w_bwd(w, sw, n0), (uint32_t)(32 * sw), zx, (uint32_t)(16 * sz), K);
                        float wA = 0.f, wB = 0.f;
                        if (want_t && l == 1 && s.time) { wA = fl[p.g.t_at + n0 + ln.g]; wB = fl[p.g.t_at + n0 + 8 + ln.g]; }
                        uint32_t o[MT][2];
#pragma unroll
                        for (int m = 0; m < MT; ++m)
#pragma unroll
                            for (int h = 0; h < 2; ++h) {
                                const float v0 = acc[m][2 * h] * act16_d<T>(s.act, lo_of<T>(hv[m][h])), v1 = acc[m][2 * h + 1] * act16_d<T>(s.act, hi_of<T>(hv[m][h]));
                                note(v0, v1);
                                o[m][h] = cvt_pack<T>(v0, v1);
                                const float wt = h ? wB : wA;
                                if (want_t) dtau = fmaf(lo_of<T>(o[m][h]), wt, fmaf(hi_of<T>(o[m][h]), wt, dtau));
                            }
                        put_tile<MT>(ln, z_at(l), sw, n0, N, o);
                    }
                } else if (owner) {
                    float acc[MT][4];
                    tile_product<T, MT, true>(acc, ln.w_bwd(w, sw, f0), (uint32_t)(32 * sw), zx, (uint32_t)(16 * sz), K);
#pragma unroll
                    for (int m = 0; m < MT; ++m)
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            note(acc[m][2 * h], acc[m][2 * h + 1]);
                            const uint32_t q = cvt_pack<T>(acc[m][2 * h], acc[m][2 * h + 1]);
                            ps[((j * MT + m) * 2 + h) * owners] = q;
                            if (!s.commit) {
#pragma unroll
                                for (int i = 0; i < 2; ++i) {
                                    const int r = r0 + m * 8 + 2 * ln.t + i, c = f0 + ln.g + h * 8;
                                    if (r < B && c < s.wp[0]) reinterpret_cast<unsigned short*>(s.psi[j])[(long long)r * s.wp[0] + c] = (unsigned short)(i ? q >> 16 : q & 0xFFFFu);
                                }
                            }
                        }
                    if (j > 0) put_kappa(j - 1, par ^ 1, dtau_k);
                }
                __syncthreads();
            }
            if (want_t) {
                t_dt += dtau;
                t_dh = fmaf(sc.c[j], dtau, t_dh);
                if (owner)
                    for (int l = 0; l < j; ++l) {
                        const float ajl = sc.a[j][l];
                        if (ajl == 0.f) continue;
                        float dot = 0.f;
#pragma unroll
                        for (int m = 0; m < MT; ++m)
#pragma unroll
                            for (int h = 0; h < 2; ++h) {
                                const uint32_t q = ps[((j * MT + m) * 2 + h) * owners], k = ks[((l * MT + m) * 2 + h) * owners];
                                dot = fmaf(lo_of<T>(q), lo_of<T>(k), fmaf(hi_of<T>(q), hi_of<T>(k), dot));
                            }
                        t_dh = fmaf(ajl, dot, t_dh);
                    }
            }
        }
        if (s.commit && owner) {      // a <- a + (h / S) sum_j psi_j (+ running cost)
            const float coef = ldexpf(sc.h, -e);
#pragma unroll
            for (int m = 0; m < MT; ++m)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float d0 = 0.f, d1 = 0.f;
#pragma unroll
                    for (int j = RK_MAX_STAGES - 1; j >= 0; --j)
                        if (j < S) {
                            const uint32_t q = ps[((j * MT + m) * 2 + h) * owners];
                            d0 += lo_of<T>(q);
                            d1 += hi_of<T>(q);
                        }
                    a[m][2 * h] = fmaf(coef, d0, a[m][2 * h]);
                    a[m][2 * h + 1] = fmaf(coef, d1, a[m][2 * h + 1]);
                    if (s.cot != nullptr) {
#pragma unroll
                        for (int i = 0; i < 2; ++i) {
                            const int r = r0 + m * 8 + 2 * ln.t + i, c = f0 + ln.g + h * 8;
                            if (r < B && c < d) a[m][2 * h + i] += s.cot[((long long)n * B + r) * d + c];
                        }
                    }
                }
        }
        if (want_t) {      // lanes by shuffles, warps in ascending order
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                t_phi += __shfl_xor_sync(0xffffffffu, t_phi, o);
                t_dt += __shfl_xor_sync(0xffffffffu, t_dt, o);
                t_dh += __shfl_xor_sync(0xffffffffu, t_dh, o);
            }
            if (ln.lane == 0) { red[ln.warp] = t_phi; red[16 + ln.warp] = t_dt; red[32 + ln.warp] = t_dh; }
            __syncthreads();
            if (threadIdx.x < 3) {
                float x = 0.f;
                for (int w = 0; w < NW; ++w) x += red[threadIdx.x * 16 + w];
                s.tpart[((long long)st * gridDim.x + blockIdx.x) * 3 + threadIdx.x] = x;
            }
        }
    }
    if (s.vjp && s.commit && owner) {
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int r = r0 + m * 8 + 2 * ln.t + (i & 1), c = f0 + ln.g + (i >> 1) * 8;
                if (r < B && c < d) s.a[(long long)r * d + c] = a[m][i];
            }
    }
    warp_flag_or(s.flag, bad);
}

// out = beta out + the blocks' gradients, in ascending order
__global__ void __launch_bounds__(128) resident_reduce_kernel(const float* __restrict__ partial, int blocks, long long params, float beta, float* __restrict__ out) {
    chain_begin();
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= params) return;
    float v = 0.f;
#pragma unroll 16
    for (int b = 0; b < blocks; ++b) v += partial[b * params + i];
    out[i] = (beta != 0.f ? beta * out[i] : 0.f) + v;
}

template <typename K>
bool allow_cap(K kernel, bool (&done)[kMaxDevices]) {
    const int dev = current_device();
    if (!done[dev]) {
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kCap) != cudaSuccess) { cudaGetLastError(); return false; }
        done[dev] = true;
    }
    return true;
}
template <typename T, int MT, int NW>
bool forward_t(const ResidentMlp& p, cudaStream_t st) {
    static bool done[kMaxDevices] = {false};
    if (!allow_cap(resident_forward_kernel<T, MT, NW>, done)) return false;
    ResidentMlp q = p;
    q.b = plan_bufs(p.g, p.s.L, p.s.stages, 8 * MT, false);
    return launch_chain(resident_forward_kernel<T, MT, NW>, dim3(p.g.blocks_f), dim3(NW * 32 + 64), resident_smem(p.g, p.s.L, p.s.wp[0], p.s.stages, MT, false), st, q) == cudaSuccess;
}
template <typename T, int MT>
bool forward_t(const ResidentMlp& p, cudaStream_t st) {
    return chain_warps(p.s.L, p.s.wp) == 8 ? forward_t<T, MT, 8>(p, st) : forward_t<T, MT, 16>(p, st);
}
template <typename T>
bool forward_t(const ResidentMlp& p, cudaStream_t st) {
    return p.g.mt_f == 1 ? forward_t<T, 1>(p, st) : p.g.mt_f == 2 ? forward_t<T, 2>(p, st) : forward_t<T, 4>(p, st);
}
// (`ready`: only makes the kernel ready for its launch)
template <typename T, int MT, int NW, bool REG>
bool backward_t(const ResidentMlp& p, cudaStream_t st, bool ready) {
    static bool done[kMaxDevices] = {false};
    if (!allow_cap(resident_backward_kernel<T, MT, NW, REG>, done)) return false;
    if (ready) return true;
    ResidentMlp q = p;
    q.b = plan_bufs(p.g, p.s.L, p.s.stages, 8 * MT, true);
    return launch_chain(resident_backward_kernel<T, MT, NW, REG>, dim3(p.g.blocks_b), dim3(NW * 32 + (REG ? kPieceWarps * 32 : 128)),
                        resident_smem(p.g, p.s.L, p.s.wp[0], p.s.stages, MT, true), st, q) == cudaSuccess;
}
template <typename T>
bool backward_t(const ResidentMlp& p, cudaStream_t st, bool ready) {
    const bool narrow = chain_warps(p.s.L, p.s.wp) == 8, reg = p.partial != nullptr;
    if (p.g.mt_b == 1) return !narrow ? backward_t<T, 1, 16, false>(p, st, ready) : reg ? backward_t<T, 1, 8, true>(p, st, ready) : backward_t<T, 1, 8, false>(p, st, ready);
    return !narrow ? backward_t<T, 2, 16, false>(p, st, ready) : reg ? backward_t<T, 2, 8, true>(p, st, ready) : backward_t<T, 2, 8, false>(p, st, ready);
}

}  // namespace

ResidentPlan plan_resident(mpode_dtype dt, int B, int L, const int* wp, bool bias, bool time) {
    ResidentPlan g;
    if (dt == MPODE_F32 || L < 1 || L > SMALL_MAX_L || wp[0] > 256) return g;
    int floats = 0;
    for (int l = 0; l <= L; ++l) {
        if (wp[l] > 1000) return g;
        g.sw[l] = up16(wp[l]) + 8;
    }
    for (int l = 0; l < L; ++l) {
        g.w_at[l] = g.w_elems;
        g.w_elems += up16(wp[l + 1]) * g.sw[l];
        g.b_at[l] = floats;
        floats += up16(wp[l + 1]);
    }
    g.t_at = floats;
    floats += up16(wp[1]);
    g.image_bytes = (g.w_elems * 2 + floats * 4 + 15) / 16 * 16;
    const int sms = sm_count();
    auto tiles = [&](int most) { int mt = 1; while (mt < most && (B + 8 * mt - 1) / (8 * mt) > sms) mt *= 2; return mt; };
    g.mt_f = tiles(4); g.blocks_f = (B + 8 * g.mt_f - 1) / (8 * g.mt_f);
    g.mt_b = tiles(2); g.blocks_b = (B + 8 * g.mt_b - 1) / (8 * g.mt_b);
    g.forward = g.blocks_f <= sms && resident_smem(g, L, wp[0], RK_MAX_STAGES, g.mt_f, false) <= (size_t)kCap;
    g.backward = g.blocks_b <= sms && resident_smem(g, L, wp[0], RK_MAX_STAGES, g.mt_b, true) <= (size_t)kCap;
    int pieces = 0;
    for (int l = 0; l < L; ++l) pieces += up16(wp[l + 1]) / 16 * piece_columns(wp[l], bias || (time && l == 0));
    g.pieces = chain_warps(L, wp) == 8 && pieces <= kPieces * kPieceWarps ? pieces : 0;
    return g;
}

void launch_resident_pack(mpode_dtype dt, const ResidentMlp& p, cudaStream_t st, long long* launches) {
    int blocks = (p.g.w_elems + 255) / 256;
    if (blocks > 148 * 4) blocks = 148 * 4;
    if (dt == MPODE_BF16) launch_chain(resident_pack_kernel<__nv_bfloat16>, dim3(blocks), dim3(256), 0, st, p);
    else launch_chain(resident_pack_kernel<__half>, dim3(blocks), dim3(256), 0, st, p);
    if (launches) ++*launches;
}

bool launch_resident_forward(mpode_dtype dt, const ResidentMlp& p, cudaStream_t st, long long* launches) {
    const bool ok = dt == MPODE_BF16 ? forward_t<__nv_bfloat16>(p, st) : forward_t<__half>(p, st);
    if (ok && launches) ++*launches;
    if (ok && tl_counters) ++tl_counters->fused;
    return ok;
}

bool resident_backward_ready(mpode_dtype dt, const ResidentMlp& p) {
    return dt == MPODE_BF16 ? backward_t<__nv_bfloat16>(p, nullptr, true) : backward_t<__half>(p, nullptr, true);
}

void launch_resident_backward(mpode_dtype dt, const ResidentMlp& p, cudaStream_t st, long long* launches) {
    if (dt == MPODE_BF16) backward_t<__nv_bfloat16>(p, st, false);
    else backward_t<__half>(p, st, false);
    if (launches) ++*launches;
    if (tl_counters) ++tl_counters->fused;
}

void launch_resident_reduce(const ResidentMlp& p, cudaStream_t st, long long* launches) {
    launch_chain(resident_reduce_kernel, dim3((unsigned)((p.g.params + 127) / 128)), dim3(128), 0, st, (const float*)p.partial, p.g.blocks_b, p.g.params, p.s.beta, p.s.out);
    if (launches) ++*launches;
}

}  // namespace mpode
