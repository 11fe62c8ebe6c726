// Row-local kernels of small dense velocities (16-bit formats) whose weights fit the SM.  A block takes 8 rows per row tile through the
// whole forward solve, or through the backward chain of several steps, and keeps all weights in shared memory, one copy for both directions:
// a weight tile is the first operand of mma.sync (16 output features x 16 inputs), read as it lies for the forward pass and through
// transposing loads for the input gradient.  The rows are the second operand, 8 at a time, so that 1000 samples spread over 125 SMs.
// What bounds a layer is its latency: weights from shared memory (64 wide 8 KB, 200 wide 85 KB at 128 bytes a cycle), a chain of one
// matrix instruction per 16 inputs, the epilogue and one block barrier.  Everything elementwise between two layers (stage input, state
// update, seed, stage cotangent, adjoint update) is done by the thread that holds the values, in the epilogue of the last layer.  Warps
// beside the ones that carry the chain move layer inputs and cotangents to memory, or, where the parameter gradient fits their registers
// and no step's gradient has to be looked at, form it on the spot: then a pass of any number of steps is one launch and a sum over blocks.
// Measured, a layer (before: small_mlp.cu): one layer of 64 1.28 -> 0.29 us, 200-200 2.2 -> 0.94 us; training passes: linear equation 64 wide, 1024
// samples, 100 RK4 steps 2.97 -> 0.53 ms; MLP 72-200-200-72, 1000 samples, 16 RK4 steps, float16 dynamic 4.8 -> 2.3 ms (with small_wgrad.cu).
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
// rows and columns of a layer's weights in the image: whole reduction steps, of a single layer an even number of them
__host__ __device__ inline int image_width(int L, int w) { return L == 1 ? (w + 31) / 32 * 32 : up16(w); }
// warps that carry the chain: 16 features each, one tile per warp up to 256 features
inline int chain_warps(int L, const int* wp) {
    int m = 0;
    for (int l = 0; l <= L; ++l) m = wp[l] > m ? wp[l] : m;
    return m <= 128 ? 8 : 16;
}

template <typename T> __device__ __forceinline__ float lo_of(uint32_t w) { return Low<T>::to_f(from_bits<T>((unsigned short)(w & 0xFFFFu))); }
template <typename T> __device__ __forceinline__ float hi_of(uint32_t w) { return Low<T>::to_f(from_bits<T>((unsigned short)(w >> 16))); }


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
        const int ld = p.g.sw[l], n = image_width(s.L, s.wp[l + 1]) * ld, in_full = s.wr[l] + ((s.time && l == 0) ? 1 : 0);
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
// [image][buffers][slots: words of the state tiles' threads: k_j; forward y; backward psi_j, seed, adjoint][scalars of two steps][sums of the time terms]
inline size_t resident_smem(const ResidentPlan& g, int L, int wp0, int stages, int mt, bool back) {
    const int owners = up16(wp0) / 16 * 32;
    const int words = (back ? 4 * RK_MAX_STAGES + 6 : 2 * RK_MAX_STAGES + 4) * mt;
    return plan_bufs(g, L, stages, 8 * mt, back).slots + (size_t)words * owners * 4 + 2 * kScalarWords * 4 + 3 * 16 * 4 + 16;
}

// One tile of 16 features for the block's 8 MT rows: acc[m][0, 1] = feature g of rows 2t, 2t + 1 (g = lane / 4, t = lane % 4), acc[m][2, 3]
// feature g + 8.  `w`: this lane's address in the weights, advanced by wstep per 16 of the reduction; `x`: in the rows' buffer.  The operands
// of a group of kAhead reduction steps are requested while the group before is multiplied; the weights of the first group depend on nothing
// and are requested before the barrier that the rows are waited for with.  (Without the second set of registers a 208-long reduction took
// 918 cycles, 270 of them matrix instructions.)
constexpr int kAhead = 2;
template <int MT> struct Ops { uint32_t a[kAhead][4], b[MT][4]; };
template <int MT, bool BACK, int N = kAhead>
__device__ __forceinline__ void load_weights(Ops<MT>& o, uint32_t w, uint32_t wstep) {
#pragma unroll
    for (int q = 0; q < N; ++q) { if (BACK) ldm4_t(w + q * wstep, o.a[q]); else ldm4(w + q * wstep, o.a[q]); }
}
template <int MT>
__device__ __forceinline__ void load_rows(Ops<MT>& o, uint32_t x, uint32_t xrow8) {
#pragma unroll
    for (int m = 0; m < MT; ++m) ldm4(x + m * xrow8, o.b[m]);
}
template <typename T, int MT, int N = kAhead>
__device__ __forceinline__ void multiply(float (&acc)[MT][4], const Ops<MT>& o) {
#pragma unroll
    for (int q = 0; q < N; ++q)
#pragma unroll
        for (int m = 0; m < MT; ++m) mma_k16<T>(acc[m], o.a[q], o.b[m][2 * q], o.b[m][2 * q + 1]);
}
// Where a warp's product of a phase finds its operands.  Formed for the next phase at the start of this one, beside the matrix
// instructions: everything that belongs to a layer comes from the constant bank at an index.
struct Phase { uint32_t w, wstep, x, xrow8; int ks; bool on; };
template <int MT, bool BACK>
__device__ __forceinline__ void request_weights(Ops<MT>& o, const Phase& ph) {      // the first group's
    load_weights<MT, BACK, 1>(o, ph.w, ph.wstep);
    if (ph.ks > 1) { if (BACK) ldm4_t(ph.w + ph.wstep, o.a[1]); else ldm4(ph.w + ph.wstep, o.a[1]); }
}
// KS reduction steps as straight-line code: a branch costs as much as a matrix instruction here, where each scheduler has one or two warps
template <typename T, int MT, bool BACK, int KS>
__device__ __forceinline__ void product_steps(float (&acc)[MT][4], Ops<MT>& o, const Phase& ph) {
    load_rows<MT>(o, ph.x, ph.xrow8);
#pragma unroll
    for (int k = 0; k < KS; k += kAhead) {
        Ops<MT> nx;
        const uint32_t w = ph.w + (uint32_t)(k + kAhead) * ph.wstep, x = ph.x + (uint32_t)(k + kAhead) * 32u;
        if (k + 2 * kAhead <= KS) { load_weights<MT, BACK>(nx, w, ph.wstep); load_rows<MT>(nx, x, ph.xrow8); }
        else if (k + kAhead < KS) { load_weights<MT, BACK, 1>(nx, w, ph.wstep); load_rows<MT>(nx, x, ph.xrow8); }
        if (k + kAhead <= KS) multiply<T, MT>(acc, o); else multiply<T, MT, 1>(acc, o);
        if (k + kAhead < KS) o = nx;
    }
}
template <typename T, int MT, bool BACK>
__device__ __forceinline__ void tail_product(float (&acc)[MT][4], Ops<MT>& o, Phase q) {      // up to 16 steps, two at a time
#pragma unroll 1
    for (;;) {
        load_rows<MT>(o, q.x, q.xrow8);
        if (q.ks == 1) { multiply<T, MT, 1>(acc, o); return; }
        multiply<T, MT>(acc, o);
        if ((q.ks -= 2) <= 0) return;
        q.w += 2u * q.wstep; q.x += 64u;
        request_weights<MT, BACK>(o, q);
    }
}
template <typename T, int MT, bool BACK>
__device__ __forceinline__ void tile_product(float (&acc)[MT][4], Ops<MT>& o, const Phase& ph) {
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[m][i] = 0.f;
    switch (ph.ks) {
#define MPODE_STEPS(K) case K: product_steps<T, MT, BACK, K>(acc, o, ph); return;
        MPODE_STEPS(1) MPODE_STEPS(2) MPODE_STEPS(3) MPODE_STEPS(4) MPODE_STEPS(5) MPODE_STEPS(6) MPODE_STEPS(7) MPODE_STEPS(8)
        MPODE_STEPS(9) MPODE_STEPS(10) MPODE_STEPS(11) MPODE_STEPS(12) MPODE_STEPS(13) MPODE_STEPS(14) MPODE_STEPS(15) MPODE_STEPS(16)
#undef MPODE_STEPS
        default: break;
    }
    Phase q = ph;
#pragma unroll 1
    for (;;) {      // (wider than 256: 16 steps at a time)
        if (q.ks <= 16) { tail_product<T, MT, BACK>(acc, o, q); return; }
        product_steps<T, MT, BACK, 16>(acc, o, q);
        q.w += 16u * q.wstep; q.x += 512u; q.ks -= 16;
        request_weights<MT, BACK>(o, q);
    }
}

// Everything a thread of the chain knows about its place
template <typename T, int MT>
struct Lane {
    int warp, lane, g, t;
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
// Rows behind the batch take the last row's values: they are integrated along with zero adjoint, and from a state of their own (y = 0) they
// could overflow where no sample does, which zero cotangents turn into NaN (parameter gradients, time terms, overflow flag).
template <typename T>
__device__ __forceinline__ void state_in(uint32_t buf, int sx, const T* src, int d, int R, int r0, int B, int tid, int threads) {
    auto row = [&](int r) { return (long long)(r0 + r < B ? r0 + r : B - 1); };
    if ((d & 7) == 0) {
        const int per = d / 8, n = R * per;
        for (int i = tid; i < n; i += threads) {
            const int r = i / per, c = (i - r * per) * 8;
            copy16(buf + (uint32_t)((r * sx + c) * 2), src + row(r) * d + c);
        }
        return;
    }
    for (int i = tid; i < R * d; i += threads) {
        const int r = i / d, c = i - r * d;
        const unsigned short v = reinterpret_cast<const unsigned short*>(src)[row(r) * d + c];
        asm volatile("st.shared.u16 [%0], %1;" ::"r"(buf + (uint32_t)((r * sx + c) * 2)), "h"(v) : "memory");
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

// the phase of layer l on the rows in `in`: the layer itself, or its input gradient
template <typename T, int MT>
__device__ __forceinline__ Phase forward_phase(const ResidentMlp& p, const Lane<T, MT>& ln, uint32_t base, int l, uint32_t in) {
    const int sw = p.g.sw[l], f0 = ln.warp * 16;
    return Phase{ln.w_fwd(base + (uint32_t)p.g.w_at[l] * 2u, sw, f0), 32u, ln.x_at(in, sw), (uint32_t)(16 * sw), up16(p.s.wp[l]) / 16, f0 < p.s.wp[l + 1]};
}
template <typename T, int MT>
__device__ __forceinline__ Phase backward_phase(const ResidentMlp& p, const Lane<T, MT>& ln, uint32_t base, int l, uint32_t in) {
    const int sw = p.g.sw[l], sz = p.g.sw[l + 1], f0 = ln.warp * 16;
    return Phase{ln.w_bwd(base + (uint32_t)p.g.w_at[l] * 2u, sw, f0), (uint32_t)(32 * sw), ln.x_at(in, sz), (uint32_t)(16 * sz), up16(p.s.wp[l + 1]) / 16, f0 < p.s.wp[l]};
}

// A hidden layer: H = Q16(act(W x + b + tau w_t)) of the block's rows.
template <typename T, int MT, int NW>
__device__ __forceinline__ void hidden_layer(const ResidentMlp& p, const Lane<T, MT>& ln, const float* fl, int l, float tau, uint32_t out, Phase ph, Ops<MT>& ahead) {
    const SmallMlp& s = p.s;
    const int N = s.wp[l + 1], so = p.g.sw[l + 1], b = p.g.b_at[l];
#pragma unroll 1
    for (int f0 = ln.warp * 16; f0 < N; f0 += NW * 16) {
        float bA = fl[b + f0 + ln.g], bB = fl[b + f0 + 8 + ln.g];
        if (s.time && l == 0) { bA = fmaf(tau, fl[p.g.t_at + f0 + ln.g], bA); bB = fmaf(tau, fl[p.g.t_at + f0 + 8 + ln.g], bB); }
        if (f0 >= NW * 16) {
            ph.w += NW * 2 * ph.xrow8;       // (a row's features further by the rows of one tile per warp: 16 NW rows of 2 sw bytes)
            request_weights<MT, false>(ahead, ph);
        }
        float acc[MT][4];
        tile_product<T, MT, false>(acc, ahead, ph);
        uint32_t v[MT][2];
#pragma unroll
        for (int m = 0; m < MT; ++m) {
            v[m][0] = cvt_pack<T>(act16<T>(s.act, acc[m][0] + bA), act16<T>(s.act, acc[m][1] + bA));
            v[m][1] = cvt_pack<T>(act16<T>(s.act, acc[m][2] + bB), act16<T>(s.act, acc[m][3] + bB));
        }
        put_tile<MT>(ln, out, so, f0, N, v);
    }
}

// What the last layer's epilogue of stage j needs besides the product: the terms of the next stage's input (or, after the last stage, of the
// increment) that do not depend on this stage, and this stage's coefficient.
template <typename T, int MT>
struct StageTerms {
    float v[MT][4], c, bA, bB;
    bool on;
    // row: h a_{j+1, .} or h b_.; from the state or from zero
    __device__ __forceinline__ void start(const float* row, int j, bool sum, const uint32_t (&yb)[MT][2], const uint32_t* ks, int owners) {
        const float4 r = *reinterpret_cast<const float4*>(row);
        const float cq[RK_MAX_STAGES - 1] = {r.x, r.y, r.z};
        c = row[j];
        on = sum || c != 0.f;
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                float v0 = sum ? 0.f : lo_of<T>(yb[m][h]), v1 = sum ? 0.f : hi_of<T>(yb[m][h]);
#pragma unroll
                for (int q = 0; q < RK_MAX_STAGES - 1; ++q) {      // (no branches: a slot that is not wanted is read all the same)
                    const bool use = q < j && (sum || cq[q] != 0.f);
                    const uint32_t k = ks[((q * MT + m) * 2 + h) * owners];
                    const float w0 = fmaf(cq[q], lo_of<T>(k), v0), w1 = fmaf(cq[q], hi_of<T>(k), v1);
                    v0 = use ? w0 : v0;
                    v1 = use ? w1 : v1;
                }
                v[m][2 * h] = v0; v[m][2 * h + 1] = v1;
            }
    }
    // k_j of pair (m, h), rounded once; the terms with it
    __device__ __forceinline__ uint32_t stage(const float (&acc)[MT][4], int m, int h) {
        const float b = h ? bB : bA;
        const uint32_t k = cvt_pack<T>(acc[m][2 * h] + b, acc[m][2 * h + 1] + b);
        const float w0 = fmaf(c, lo_of<T>(k), v[m][2 * h]), w1 = fmaf(c, hi_of<T>(k), v[m][2 * h + 1]);
        v[m][2 * h] = on ? w0 : v[m][2 * h];
        v[m][2 * h + 1] = on ? w1 : v[m][2 * h + 1];
        return k;
    }
};

// ---------------------------------------------------------------- one layer
// A velocity of a single layer is the shortest chain: every phase is one product of up to 128 x 128 and the elementwise step behind it.  With
// one warp to a scheduler a phase is the sum of its instructions' latencies (the general code's 150 instructions: 1000 cycles), so the
// weights of a warp's tile stay in registers, for both directions, and nothing is left in a phase but matrix loads, matrix
// instructions, the epilogue and the barrier.  KS1: reduction steps, a multiple of two (the image is padded with zeros to it).
template <typename T, int MT, int KS1>
struct Linear {
    uint32_t w[KS1][4];
    template <bool BACK> __device__ __forceinline__ void load(uint32_t at, uint32_t wstep) {
#pragma unroll
        for (int k = 0; k < KS1; ++k) { if (BACK) ldm4_t(at + k * wstep, w[k]); else ldm4(at + k * wstep, w[k]); }
    }
    __device__ __forceinline__ void product(float (&acc)[MT][4], uint32_t x, uint32_t xrow8) const {
        uint32_t b[KS1 / 2][MT][4];
#pragma unroll
        for (int k = 0; k < KS1 / 2; ++k)
#pragma unroll
            for (int m = 0; m < MT; ++m) ldm4(x + k * 64 + m * xrow8, b[k][m]);
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[m][i] = 0.f;
#pragma unroll
        for (int k = 0; k < KS1; ++k)
#pragma unroll
            for (int m = 0; m < MT; ++m) mma_k16<T>(acc[m], w[k], b[k >> 1][m][2 * (k & 1)], b[k >> 1][m][2 * (k & 1) + 1]);
    }
};
// Y_{j+1} = Q16(ybar + sum_{l <= j} (h a_{j+1,l}) k_l): the terms with l < j, where the tableau has any
template <typename T, int MT>
__device__ __forceinline__ void earlier_terms(float (&v)[MT][4], const float* row, int j, const uint32_t* ks, int owners) {
    for (int q = 0; q < j; ++q) {
        const float c = row[q];
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
}

template <typename T, int MT, int KS1>
__device__ __forceinline__ void linear_forward(const ResidentMlp& p, uint32_t base, uint32_t* ks, const float* scal, const float* fl, int r0) {
    const SmallMlp& s = p.s;
    const Lane<T, MT> ln;
    const int d = s.wr[0], S = s.stages, sx = p.g.sw[0], tiles0 = up16(s.wp[0]) / 16, owners = tiles0 * 32, f0 = ln.warp * 16;
    const bool owner = ln.warp < tiles0, upper = f0 + 8 < s.wp[0], time = s.time != 0, alone = s.alone != 0;
    const uint32_t xrow8 = (uint32_t)(16 * sx), z0 = base + (uint32_t)p.b.z0;
    float y[MT][4], u[MT][4];
    uint32_t yb[MT][2];
    if (owner) {
#pragma unroll
        for (int m = 0; m < MT; ++m) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int r = r0 + m * 8 + 2 * ln.t + (i & 1), c = f0 + ln.g + (i >> 1) * 8;
                y[m][i] = r < s.B && c < d ? s.y0[(long long)r * d + c] : 0.f;
                u[m][i] = 0.f;
            }
            yb[m][0] = cvt_pack<T>(y[m][0], y[m][1]);
            yb[m][1] = cvt_pack<T>(y[m][2], y[m][3]);
        }
        put_tile<MT>(ln, z0, sx, f0, s.wp[0], yb);
    }
    copies_done();
    __syncthreads();
    Linear<T, MT, KS1> W;
    float b0 = 0.f, b1 = 0.f, t0 = 0.f, t1 = 0.f;
    if (owner) {
        W.template load<false>(ln.w_fwd(base, sx, f0), 32u);
        b0 = fl[f0 + ln.g]; b1 = fl[f0 + 8 + ln.g];
        t0 = fl[p.g.t_at + f0 + ln.g]; t1 = fl[p.g.t_at + f0 + 8 + ln.g];
    }
    const uint32_t x0 = ln.x_at(z0, sx), o0 = ln.frag_at(z0, sx, f0, 0);
    uint32_t cur = 0;      // offset of the buffer that holds the stage input
    for (int n = 0; n < s.n_steps; ++n) {
        const RkStepScalars& sc = *(const RkStepScalars*)(scal + (n & 1) * kScalarWords);
#pragma unroll
        for (int j = 0; j < RK_MAX_STAGES; ++j) {
            if (j >= S) break;
            const uint32_t nxt = (uint32_t)p.b.state - cur;
            if (owner) {
                const bool last = j + 1 == S;
                const float hb = sc.hb[j], c = sc.ha[j + 1 < RK_MAX_STAGES ? j + 1 : j][j];
                float acc[MT][4];
                W.product(acc, x0 + cur, xrow8);
                const float bA = time ? fmaf(sc.tau16[j], t0, b0) : b0, bB = time ? fmaf(sc.tau16[j], t1, b1) : b1;
                float v[MT][4];
                uint32_t k[MT][2];
#pragma unroll
                for (int m = 0; m < MT; ++m)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        k[m][h] = cvt_pack<T>(acc[m][2 * h] + (h ? bB : bA), acc[m][2 * h + 1] + (h ? bB : bA));
                        u[m][2 * h] = fmaf(hb, lo_of<T>(k[m][h]), u[m][2 * h]);
                        u[m][2 * h + 1] = fmaf(hb, hi_of<T>(k[m][h]), u[m][2 * h + 1]);
                        v[m][2 * h] = lo_of<T>(yb[m][h]);
                        v[m][2 * h + 1] = hi_of<T>(yb[m][h]);
                    }
                if (!last) {
                    if (!alone) {
                        earlier_terms<T, MT>(v, sc.ha[j + 1 < RK_MAX_STAGES ? j + 1 : j], j, ks, owners);
#pragma unroll
                        for (int m = 0; m < MT; ++m) { ks[((j * MT + m) * 2) * owners] = k[m][0]; ks[((j * MT + m) * 2 + 1) * owners] = k[m][1]; }
                    }
                    if (alone || c != 0.f) {
#pragma unroll
                        for (int m = 0; m < MT; ++m)
#pragma unroll
                            for (int i = 0; i < 4; ++i) v[m][i] = fmaf(c, (i & 1) ? hi_of<T>(k[m][i >> 1]) : lo_of<T>(k[m][i >> 1]), v[m][i]);
                    }
                } else {
#pragma unroll
                    for (int m = 0; m < MT; ++m)
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            y[m][i] += s.round_increment ? sc.h * Low<T>::to_f(Low<T>::from_f(u[m][i])) : u[m][i];
                            v[m][i] = y[m][i];
                            u[m][i] = 0.f;
                        }
                }
#pragma unroll
                for (int m = 0; m < MT; ++m) {
                    const uint32_t q0 = cvt_pack<T>(v[m][0], v[m][1]), q1 = cvt_pack<T>(v[m][2], v[m][3]);
                    if (last) { yb[m][0] = q0; yb[m][1] = q1; }
                    stm2_t(o0 + nxt + m * xrow8, q0, upper ? q1 : 0u);
                }
            }
            __syncthreads();
            cur = nxt;
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

// (no time terms: the general code has them)
template <typename T, int MT, int KS1>
__device__ __forceinline__ void linear_backward(const ResidentMlp& p, uint32_t base, uint32_t* ks, const float* scal, const float* fl, int r0) {
    const SmallMlp& s = p.s;
    const Lane<T, MT> ln;
    const int d = s.wr[0], S = s.stages, B = s.B, sx = p.g.sw[0], tiles0 = up16(s.wp[0]) / 16, owners = tiles0 * 32, f0 = ln.warp * 16;
    const bool owner = ln.warp < tiles0, upper = f0 + 8 < s.wp[0], time = s.time != 0, alone = s.alone != 0;
    const uint32_t xrow8 = (uint32_t)(16 * sx);
    uint32_t* ps = ks + RK_MAX_STAGES * 2 * MT * owners;
    const int e = s.e_dev != nullptr ? *s.e_dev : s.e;
    const float scale = ldexpf(1.f, e), unscale = ldexpf(1.f, -e);      // (|e| <= 100: products with them are what ldexp gives)
    uint32_t bad = 0u;
    Linear<T, MT, KS1> F, Bk;
    float b0 = 0.f, b1 = 0.f, t0 = 0.f, t1 = 0.f, a[MT][4];
    if (owner) {
        F.template load<false>(ln.w_fwd(base, sx, f0), 32u);
        Bk.template load<true>(ln.w_bwd(base, sx, f0), (uint32_t)(32 * sx));
        b0 = fl[f0 + ln.g]; b1 = fl[f0 + 8 + ln.g];
        t0 = fl[p.g.t_at + f0 + ln.g]; t1 = fl[p.g.t_at + f0 + 8 + ln.g];
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int r = r0 + m * 8 + 2 * ln.t + (i & 1), c = f0 + ln.g + (i >> 1) * 8;
                a[m][i] = s.vjp && r < B && c < d ? s.a[(long long)r * d + c] : 0.f;
            }
    }
    const uint32_t xl = ln.x_at(base, sx), ol = ln.frag_at(base, sx, f0, 0);      // + the buffer's offset
    for (int st = 0; st < s.count; ++st) {
        const int n = s.step_hi - st;
        const RkStepScalars& sc = *(const RkStepScalars*)(scal + (st & 1) * kScalarWords);
        const uint32_t x00 = (uint32_t)(p.b.x00 + (st & 1) * p.b.state);
        uint32_t vv[MT][2];
        if (s.vjp && owner) {              // seed Q16(S a); the last stage's cotangent Q16(b v)
            const float bj = sc.b[S - 1];
#pragma unroll
            for (int m = 0; m < MT; ++m) {
                uint32_t o[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    vv[m][h] = cvt_pack<T>(a[m][2 * h] * scale, a[m][2 * h + 1] * scale);
                    note_nonfinite<T>(vv[m][h], bad);
                    o[h] = cvt_pack<T>(bj * lo_of<T>(vv[m][h]), bj * hi_of<T>(vv[m][h]));
                    note_nonfinite<T>(o[h], bad);
                }
                stm2_t(ol + (uint32_t)p.b.z0 + m * xrow8, o[0], upper ? o[1] : 0u);
            }
        }
        __syncthreads();
        if (s.recompute) {
            uint32_t yb[MT][2];
            if (owner) {
#pragma unroll
                for (int m = 0; m < MT; ++m) ldm2_t(ol + x00 + m * xrow8, yb[m][0], yb[m][1]);
            }
#pragma unroll
            for (int j = 0; j + 1 < RK_MAX_STAGES; ++j) {
                if (j + 1 >= S) break;
                if (owner) {
                    const float c = sc.ha[j + 1][j];
                    float acc[MT][4];
                    F.product(acc, xl + (j == 0 ? x00 : (uint32_t)(p.b.keep + j * p.b.keep_stage)), xrow8);
                    const float bA = time ? fmaf(sc.tau16[j], t0, b0) : b0, bB = time ? fmaf(sc.tau16[j], t1, b1) : b1;
                    float v[MT][4];
                    uint32_t k[MT][2];
#pragma unroll
                    for (int m = 0; m < MT; ++m)
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            k[m][h] = cvt_pack<T>(acc[m][2 * h] + (h ? bB : bA), acc[m][2 * h + 1] + (h ? bB : bA));
                            v[m][2 * h] = lo_of<T>(yb[m][h]);
                            v[m][2 * h + 1] = hi_of<T>(yb[m][h]);
                        }
                    if (!alone) {
                        earlier_terms<T, MT>(v, sc.ha[j + 1], j, ks, owners);
#pragma unroll
                        for (int m = 0; m < MT; ++m) { ks[((j * MT + m) * 2) * owners] = k[m][0]; ks[((j * MT + m) * 2 + 1) * owners] = k[m][1]; }
                    }
                    if (alone || c != 0.f) {
#pragma unroll
                        for (int m = 0; m < MT; ++m)
#pragma unroll
                            for (int i = 0; i < 4; ++i) v[m][i] = fmaf(c, (i & 1) ? hi_of<T>(k[m][i >> 1]) : lo_of<T>(k[m][i >> 1]), v[m][i]);
                    }
#pragma unroll
                    for (int m = 0; m < MT; ++m)
                        stm2_t(ol + (uint32_t)(p.b.keep + (j + 1) * p.b.keep_stage) + m * xrow8, cvt_pack<T>(v[m][0], v[m][1]), upper ? cvt_pack<T>(v[m][2], v[m][3]) : 0u);
                }
                __syncthreads();
            }
        }
        if (!s.vjp) continue;
        float sum[MT][4];
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int i = 0; i < 4; ++i) sum[m][i] = 0.f;
        uint32_t z = (uint32_t)p.b.z0, zn = z + (uint32_t)p.b.state;
#pragma unroll
        for (int j = RK_MAX_STAGES - 1; j >= 0; --j) {
            if (j >= S) continue;
            if (owner) {
                const int jp = j > 0 ? j - 1 : 0;
                const float bj = sc.b[jp], cj = sc.ha[j][jp];
                float acc[MT][4];
                Bk.product(acc, xl + z, xrow8);
#pragma unroll
                for (int m = 0; m < MT; ++m) {
                    uint32_t o[2];
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const uint32_t q = cvt_pack<T>(acc[m][2 * h], acc[m][2 * h + 1]);
                        note_nonfinite<T>(q, bad);
                        sum[m][2 * h] += lo_of<T>(q);
                        sum[m][2 * h + 1] += hi_of<T>(q);
                        if (!alone) ps[((j * MT + m) * 2 + h) * owners] = q;
                        if (!s.commit) {
#pragma unroll
                            for (int i = 0; i < 2; ++i) {
                                const int r = r0 + m * 8 + 2 * ln.t + i, c = f0 + ln.g + h * 8;
                                if (r < B && c < s.wp[0]) reinterpret_cast<unsigned short*>(s.psi[j])[(long long)r * s.wp[0] + c] = (unsigned short)(i ? q >> 16 : q & 0xFFFFu);
                            }
                        }
                        if (j > 0) {
                            float v0 = bj * lo_of<T>(vv[m][h]), v1 = bj * hi_of<T>(vv[m][h]);
                            if (alone || cj != 0.f) { v0 = fmaf(cj, lo_of<T>(q), v0); v1 = fmaf(cj, hi_of<T>(q), v1); }
                            if (!alone) {
                                for (int l = j + 1; l < S; ++l) {
                                    const float c = sc.ha[l][jp];
                                    if (c == 0.f) continue;
                                    const uint32_t w = ps[((l * MT + m) * 2 + h) * owners];
                                    v0 = fmaf(c, lo_of<T>(w), v0);
                                    v1 = fmaf(c, hi_of<T>(w), v1);
                                }
                            }
                            o[h] = cvt_pack<T>(v0, v1);
                            note_nonfinite<T>(o[h], bad);
                        }
                    }
                    if (j > 0) stm2_t(ol + zn + m * xrow8, o[0], upper ? o[1] : 0u);
                }
            }
            __syncthreads();
            const uint32_t w = z; z = zn; zn = w;
        }
        if (s.commit && owner) {      // a <- a + (h / S) sum_j psi_j (+ running cost)
            const float coef = sc.h * unscale;
#pragma unroll
            for (int m = 0; m < MT; ++m)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    a[m][i] = fmaf(coef, sum[m][i], a[m][i]);
                    const int r = r0 + m * 8 + 2 * ln.t + (i & 1), c = f0 + ln.g + (i >> 1) * 8;
                    if (s.cot != nullptr && r < B && c < d) a[m][i] += s.cot[((long long)n * B + r) * d + c];
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
    warp_flag_or(s.flag, any_nonfinite(bad));
}

// ---------------------------------------------------------------- forward
template <typename T, int MT, int NW, int KS1>
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
    float* scal = (float*)(slots + (2 * RK_MAX_STAGES + 4) * MT * owners);
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
    if constexpr (KS1 > 0) { linear_forward<T, MT, KS1>(p, base, slots + threadIdx.x, scal, fl, r0); return; }
    const Lane<T, MT> ln;
    const bool owner = ln.warp < tiles0;
    const int f0 = ln.warp * 16;
    uint32_t* ks = slots + threadIdx.x;            // k_j of this thread's values: word (2 MT j + 2 m + h) * owners
    float* ys = (float*)(ks + RK_MAX_STAGES * 2 * MT * owners);      // y: word (4 m + i) * owners
    uint32_t yb[MT][2];
    if (owner) {
#pragma unroll
        for (int m = 0; m < MT; ++m) {
            float y[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int r = r0 + m * 8 + 2 * ln.t + (i & 1), c = f0 + ln.g + (i >> 1) * 8;
                y[i] = r < s.B && c < d ? s.y0[(long long)r * d + c] : 0.f;
                ys[(4 * m + i) * owners] = y[i];
            }
            yb[m][0] = cvt_pack<T>(y[0], y[1]);
            yb[m][1] = cvt_pack<T>(y[2], y[3]);
        }
        put_tile<MT>(ln, z0_at(0), p.g.sw[0], f0, s.wp[0], yb);
    }
    copies_done();
    __syncthreads();
    int cur = 0;
    Ops<MT> ahead;
    const float bias0 = owner ? fl[p.g.b_at[L - 1] + f0 + ln.g] : 0.f, bias1 = owner ? fl[p.g.b_at[L - 1] + f0 + 8 + ln.g] : 0.f;
    Phase ph = forward_phase(p, ln, base, 0, z0_at(0));
    if (ph.on) request_weights<MT, false>(ahead, ph);
    for (int n = 0; n < s.n_steps; ++n) {
        const RkStepScalars& sc = *(const RkStepScalars*)(scal + (n & 1) * kScalarWords);
#pragma unroll 1
        for (int j = 0; j < S; ++j) {
            const float tau = sc.tau16[j];
#pragma unroll 1
            for (int l = 0; l + 1 < L; ++l) {
                const Phase nx = forward_phase(p, ln, base, l + 1, z_at(l + 1));
                hidden_layer<T, MT, NW>(p, ln, fl, l, tau, z_at(l + 1), ph, ahead);
                ph = nx;
                if (ph.on) request_weights<MT, false>(ahead, ph);
                __syncthreads();
            }
            const Phase nx = forward_phase(p, ln, base, 0, z0_at(cur ^ 1));
            if (owner) {
                const bool last = j + 1 == S;
                StageTerms<T, MT> w;
                w.start(last ? sc.hb : sc.ha[j + 1], j, last, yb, ks, owners);
                w.bA = bias0; w.bB = bias1;
                if (s.time && L == 1) { w.bA = fmaf(tau, fl[p.g.t_at + f0 + ln.g], w.bA); w.bB = fmaf(tau, fl[p.g.t_at + f0 + 8 + ln.g], w.bB); }
                float acc[MT][4];
                tile_product<T, MT, false>(acc, ahead, ph);
                uint32_t o[MT][2];
#pragma unroll
                for (int m = 0; m < MT; ++m)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const uint32_t k = w.stage(acc, m, h);
                        if (!last) {
                            ks[((j * MT + m) * 2 + h) * owners] = k;
                        } else {
#pragma unroll
                            for (int i = 2 * h; i < 2 * h + 2; ++i) {
                                const float y = ys[(4 * m + i) * owners] + (s.round_increment ? sc.h * Low<T>::to_f(Low<T>::from_f(w.v[m][i])) : w.v[m][i]);
                                ys[(4 * m + i) * owners] = w.v[m][i] = y;
                            }
                        }
                        o[m][h] = cvt_pack<T>(w.v[m][2 * h], w.v[m][2 * h + 1]);
                        if (last) yb[m][h] = o[m][h];
                    }
                put_tile<MT>(ln, z0_at(cur ^ 1), p.g.sw[0], f0, s.wp[0], o);
            }
            ph = nx;
            if (ph.on) request_weights<MT, false>(ahead, ph);
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
                if (r < s.B && c < d) s.yT[(long long)r * d + c] = ys[(4 * m + i) * owners];
            }
    }
}

// ---------------------------------------------------------------- backward
// The chain of `count` steps (recompute, seed, stage and layer cotangents, with commit the adjoint update), as small_backward_kernel
// describes it; with REG the parameter gradient of the block's rows beside it, in the registers of eight warps, pieces of 16 x 8: a step's
// sums first, then g += (h / S) dg in float32.
template <typename T, int MT, int NW, bool REG, int KS1>
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
    float* scal = (float*)(slots + (4 * RK_MAX_STAGES + 6) * MT * owners);
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
        uint32_t off[kPieces], off2[kPieces];      // this lane's offsets in the rows' buffers of outputs and inputs
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
                const int l = piece[i] < 0 ? 0 : pl(i), m0 = pm(i), n0 = piece[i] < 0 || pn(i) < 0 ? 0 : pn(i), sz = p.g.sw[l + 1], sx = p.g.sw[l];
                off[i] = (uint32_t)(MT == 1 ? ((lane >> 4) == 0 ? (lane & 7) * sz + m0 + (lane >> 3) * 8 : (lane & 7) * sx + n0)
                                            : ((lane & 7) + (lane >> 4) * 8) * sz + m0 + ((lane >> 3) & 1) * 8) * 2u;
                off2[i] = (uint32_t)(((lane & 7) + ((lane >> 3) & 1) * 8) * sx + n0) * 2u;
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
                        uint32_t ones = 0u;      // column 0: ones, column 1: the rounded stage time
                        if ((lane >> 2) == 0) ones = cvt_pack<T>(1.f, 1.f);
                        else if ((lane >> 2) == 1 && s.time && l == 0) ones = cvt_pack<T>(sc.tau16[j], sc.tau16[j]);
                        const uint32_t at = MT == 2 || (lane >> 4) == 0 ? z : x;
#pragma unroll
                        for (int i = 0; i < kPieces; ++i) {
                            if (pl(i) != l) continue;
                            const bool cols = pn(i) >= 0;
                            if constexpr (MT == 1) {
                                uint32_t f[4];      // both halves of the outputs, then the inputs (twice)
                                ldm4_t(at + off[i], f);
                                mma_k8<T>(acc[i], f[0], f[1], cols ? f[2] : ones);
                            } else {
                                static_assert(!REG || MT <= 2, "16 rows at most");
                                uint32_t a[4], b0, b1;
                                ldm4_t(at + off[i], a);
                                ldm2_t(x + off2[i], b0, b1);
                                mma_k16<T>(acc[i], a, cols ? b0 : ones, cols ? b1 : ones);
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
    if constexpr (KS1 > 0) { linear_backward<T, MT, KS1>(p, base, slots + threadIdx.x, scal, fl, r0); return; }
    // ---- the chain
    const Lane<T, MT> ln;
    const bool owner = ln.warp < tiles0;
    const int f0 = ln.warp * 16;
    uint32_t* ks = slots + threadIdx.x;                                // k_j and psi_j of this thread's values
    uint32_t* ps = ks + RK_MAX_STAGES * 2 * MT * owners;
    uint32_t* vs = ps + RK_MAX_STAGES * 2 * MT * owners;                           // seed: word (2 m + h) * owners
    float* as = (float*)(vs + 2 * MT * owners);                        // adjoint: word (4 m + i) * owners
    const int e = s.e_dev != nullptr ? *s.e_dev : s.e;
    const float scale = ldexpf(1.f, e), unscale = ldexpf(1.f, -e);      // (|e| <= 100: products with them are what ldexp gives)
    uint32_t bad = 0u;
    if (owner && s.vjp) {
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int r = r0 + m * 8 + 2 * ln.t + (i & 1), c = f0 + ln.g + (i >> 1) * 8;
                as[(4 * m + i) * owners] = r < B && c < d ? s.a[(long long)r * d + c] : 0.f;
            }
    }
    Ops<MT> ahead;
    const float bias0 = owner ? fl[p.g.b_at[L - 1] + f0 + ln.g] : 0.f, bias1 = owner ? fl[p.g.b_at[L - 1] + f0 + 8 + ln.g] : 0.f;
    Phase ph;
    // what follows a phase: the operands' place is settled at its start, the weights are requested at its end
    auto first_back = [&](int par) { return backward_phase(p, ln, base, L - 1, z0_at(par)); };
    auto take = [&](const Phase& nx, bool back) {
        ph = nx;
        if (ph.on) { if (back) request_weights<MT, true>(ahead, ph); else request_weights<MT, false>(ahead, ph); }
    };
    const bool evaluates = s.recompute && (S > 1 || L > 1 || want_t);      // whether anything is evaluated before the vector-Jacobian product
    for (int st = 0; st < s.count; ++st) {
        const int n = s.step_hi - st;
        const RkStepScalars& sc = *(const RkStepScalars*)(scal + (st & 1) * kScalarWords);
        float t_phi = 0.f, t_dt = 0.f, t_dh = 0.f;
        float dtau_k = 0.f;                // (one layer: of the stage cotangent in the buffer)
        auto put_kappa = [&](int par, uint32_t (&o)[MT][2]) {
            if (want_t && L == 1 && s.time) {
                const float wA = fl[p.g.t_at + f0 + ln.g], wB = fl[p.g.t_at + f0 + 8 + ln.g];
#pragma unroll
                for (int m = 0; m < MT; ++m)
#pragma unroll
                    for (int h = 0; h < 2; ++h) dtau_k = fmaf(lo_of<T>(o[m][h]), h ? wB : wA, fmaf(hi_of<T>(o[m][h]), h ? wB : wA, dtau_k));
            }
            put_tile<MT>(ln, z0_at(par), p.g.sw[0], f0, s.wp[0], o);
        };
        if (s.vjp && owner) {              // seed Q16(S a); the last stage's cotangent Q16(b v)
            uint32_t o[MT][2];
            const float bj = sc.b[S - 1];
#pragma unroll
            for (int m = 0; m < MT; ++m)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const uint32_t v = cvt_pack<T>(as[(4 * m + 2 * h) * owners] * scale, as[(4 * m + 2 * h + 1) * owners] * scale);
                    note_nonfinite<T>(v, bad);
                    vs[(2 * m + h) * owners] = v;
                    const float k0 = bj * lo_of<T>(v), k1 = bj * hi_of<T>(v);
                    o[m][h] = cvt_pack<T>(k0, k1);
                    note_nonfinite<T>(o[m][h], bad);
                }
            put_kappa(0, o);
        }
        if (evaluates) take(forward_phase(p, ln, base, 0, x00_at(st & 1)), false); else take(first_back(0), true);
        __syncthreads();
        if (s.recompute) {
#pragma unroll 1
            for (int j = 0; j < S; ++j) {
                const float tau = sc.tau16[j];
                const bool next = j + 1 < S, eval = next || want_t;      // (the last stage's derivative is wanted for the time terms alone)
#pragma unroll 1
                for (int l = 0; l + 1 < L; ++l) {
                    const bool back = l + 2 == L && !eval;
                    const Phase nx = back ? first_back(0) : forward_phase(p, ln, base, l + 1, keep_at(j, l + 1));
                    hidden_layer<T, MT, NW>(p, ln, fl, l, tau, keep_at(j, l + 1), ph, ahead);
                    take(nx, back);
                    __syncthreads();
                }
                if (!eval) break;
                // with one layer nothing of the last stage is evaluated
                const bool back = !next || (L == 1 && j + 2 == S && !want_t);
                const Phase nx = back ? first_back(0) : forward_phase(p, ln, base, 0, keep_at(j + 1, 0));
                if (owner) {
                    StageTerms<T, MT> w;
                    uint32_t yb[MT][2];
#pragma unroll
                    for (int m = 0; m < MT; ++m) ldm2_t(ln.frag_at(x00_at(st & 1), p.g.sw[0], f0, m), yb[m][0], yb[m][1]);
                    w.start(next ? sc.ha[j + 1] : sc.hb, j, false, yb, ks, owners);
                    w.bA = bias0; w.bB = bias1;
                    if (s.time && L == 1) { w.bA = fmaf(tau, fl[p.g.t_at + f0 + ln.g], w.bA); w.bB = fmaf(tau, fl[p.g.t_at + f0 + 8 + ln.g], w.bB); }
                    float acc[MT][4];
                    tile_product<T, MT, false>(acc, ahead, ph);
                    uint32_t o[MT][2];
#pragma unroll
                    for (int m = 0; m < MT; ++m)
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            ks[((j * MT + m) * 2 + h) * owners] = w.stage(acc, m, h);
                            o[m][h] = cvt_pack<T>(w.v[m][2 * h], w.v[m][2 * h + 1]);
                        }
                    if (next) put_tile<MT>(ln, keep_at(j + 1, 0), p.g.sw[0], f0, s.wp[0], o);
                }
                take(nx, back);
                __syncthreads();
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
                    t_phi = fmaf(p0, as[(4 * m + 2 * h) * owners], fmaf(p1, as[(4 * m + 2 * h + 1) * owners], t_phi));
                }
        }
#pragma unroll 1
        for (int j = S - 1; j >= 0; --j) {
            const int par = (S - 1 - j) & 1;
            float dtau = dtau_k;
            dtau_k = 0.f;
#pragma unroll 1
            for (int l = L - 1; l >= 1; --l) {
                const Phase nx = backward_phase(p, ln, base, l - 1, z_at(l));
                const int N = s.wp[l], sw = p.g.sw[l];
                const uint32_t H = keep_at(j, l);
#pragma unroll 1
                for (int n0 = ln.warp * 16; n0 < N; n0 += NW * 16) {
                    if (n0 >= NW * 16) {
                        ph.w += NW * 32;
                        request_weights<MT, true>(ahead, ph);
                    }
                    uint32_t hv[MT][2];
#pragma unroll
                    for (int m = 0; m < MT; ++m) ldm2_t(ln.frag_at(H, sw, n0, m), hv[m][0], hv[m][1]);
                    float acc[MT][4];
                    tile_product<T, MT, true>(acc, ahead, ph);
                    uint32_t o[MT][2];
#pragma unroll
                    for (int m = 0; m < MT; ++m)
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const float v0 = acc[m][2 * h] * act16_d<T>(s.act, lo_of<T>(hv[m][h])), v1 = acc[m][2 * h + 1] * act16_d<T>(s.act, hi_of<T>(hv[m][h]));
                            o[m][h] = cvt_pack<T>(v0, v1);
                            note_nonfinite<T>(o[m][h], bad);
                        }
                    if (want_t && l == 1 && s.time) {
                        const float wA = fl[p.g.t_at + n0 + ln.g], wB = fl[p.g.t_at + n0 + 8 + ln.g];
#pragma unroll
                        for (int m = 0; m < MT; ++m)
#pragma unroll
                            for (int h = 0; h < 2; ++h) dtau = fmaf(lo_of<T>(o[m][h]), h ? wB : wA, fmaf(hi_of<T>(o[m][h]), h ? wB : wA, dtau));
                    }
                    put_tile<MT>(ln, z_at(l), sw, n0, N, o);
                }
                take(nx, true);
                __syncthreads();
            }
            const Phase nx = first_back(par ^ 1);
            if (owner) {
                // psi_j; then kappa_{j-1} = Q16(b_{j-1} v + sum_{l >= j} (h a_{l,j-1}) psi_l)
                float cl[RK_MAX_STAGES], bj = 0.f, cj = 0.f;
#pragma unroll
                for (int l = 2; l < RK_MAX_STAGES; ++l) cl[l] = j > 0 && l > j && l < S ? sc.ha[l][j - 1] : 0.f;
                if (j > 0) { bj = sc.b[j - 1]; cj = sc.ha[j][j - 1]; }
                float acc[MT][4];
                tile_product<T, MT, true>(acc, ahead, ph);
                uint32_t o[MT][2];
#pragma unroll
                for (int m = 0; m < MT; ++m)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const uint32_t q = cvt_pack<T>(acc[m][2 * h], acc[m][2 * h + 1]);
                        note_nonfinite<T>(q, bad);
                        ps[((j * MT + m) * 2 + h) * owners] = q;
                        if (!s.commit) {
#pragma unroll
                            for (int i = 0; i < 2; ++i) {
                                const int r = r0 + m * 8 + 2 * ln.t + i, c = f0 + ln.g + h * 8;
                                if (r < B && c < s.wp[0]) reinterpret_cast<unsigned short*>(s.psi[j])[(long long)r * s.wp[0] + c] = (unsigned short)(i ? q >> 16 : q & 0xFFFFu);
                            }
                        }
                        if (j > 0) {
                            const uint32_t v = vs[(2 * m + h) * owners];
                            float v0 = bj * lo_of<T>(v), v1 = bj * hi_of<T>(v);
                            const float u0 = fmaf(cj, lo_of<T>(q), v0), u1 = fmaf(cj, hi_of<T>(q), v1);
                            v0 = cj != 0.f ? u0 : v0;
                            v1 = cj != 0.f ? u1 : v1;
#pragma unroll
                            for (int l = 2; l < RK_MAX_STAGES; ++l) {
                                const uint32_t u = ps[((l * MT + m) * 2 + h) * owners];
                                const float w0 = fmaf(cl[l], lo_of<T>(u), v0), w1 = fmaf(cl[l], hi_of<T>(u), v1);
                                v0 = cl[l] != 0.f ? w0 : v0;
                                v1 = cl[l] != 0.f ? w1 : v1;
                            }
                            o[m][h] = cvt_pack<T>(v0, v1);
                            note_nonfinite<T>(o[m][h], bad);
                        }
                    }
                if (j > 0) put_kappa(par ^ 1, o);
            }
            if (j > 0) take(nx, true);
            __syncthreads();
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
            const float coef = sc.h * unscale;
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
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        float v = fmaf(coef, i ? d1 : d0, as[(4 * m + 2 * h + i) * owners]);
                        const int r = r0 + m * 8 + 2 * ln.t + i, c = f0 + ln.g + h * 8;
                        if (s.cot != nullptr && r < B && c < d) v += s.cot[((long long)n * B + r) * d + c];
                        as[(4 * m + 2 * h + i) * owners] = v;
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
                if (r < B && c < d) s.a[(long long)r * d + c] = as[(4 * m + i) * owners];
            }
    }
    warp_flag_or(s.flag, any_nonfinite(bad));
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
template <typename T, int MT, int NW, int KS1>
bool forward_t(const ResidentMlp& p, cudaStream_t st) {
    static bool done[kMaxDevices] = {false};
    if (!allow_cap(resident_forward_kernel<T, MT, NW, KS1>, done)) return false;
    ResidentMlp q = p;
    q.b = plan_bufs(p.g, p.s.L, p.s.stages, 8 * MT, false);
    return launch_chain(resident_forward_kernel<T, MT, NW, KS1>, dim3(p.g.blocks_f), dim3(NW * 32 + 64), resident_smem(p.g, p.s.L, p.s.wp[0], p.s.stages, MT, false), st, q) ==
           cudaSuccess;
}
template <typename T, int MT>
bool forward_t(const ResidentMlp& p, cudaStream_t st) {
    if (p.s.L == 1 && p.s.wp[0] <= 128) {
        const int w = image_width(1, p.s.wp[0]);
        return w == 32 ? forward_t<T, MT, 8, 2>(p, st) : w == 64 ? forward_t<T, MT, 8, 4>(p, st) : w == 96 ? forward_t<T, MT, 8, 6>(p, st) : forward_t<T, MT, 8, 8>(p, st);
    }
    if (chain_warps(p.s.L, p.s.wp) == 8) return forward_t<T, MT, 8, 0>(p, st);
    if constexpr (MT <= 2) return forward_t<T, MT, 16, 0>(p, st); else return false;
}
template <typename T>
bool forward_t(const ResidentMlp& p, cudaStream_t st) {
    return p.g.mt_f == 1 ? forward_t<T, 1>(p, st) : p.g.mt_f == 2 ? forward_t<T, 2>(p, st) : forward_t<T, 4>(p, st);
}
// (`ready`: only makes the kernel ready for its launch)
template <typename T, int MT, int NW, bool REG, int KS1>
bool backward_t(const ResidentMlp& p, cudaStream_t st, bool ready) {
    static bool done[kMaxDevices] = {false};
    if (!allow_cap(resident_backward_kernel<T, MT, NW, REG, KS1>, done)) return false;
    if (ready) return true;
    ResidentMlp q = p;
    q.b = plan_bufs(p.g, p.s.L, p.s.stages, 8 * MT, true);
    return launch_chain(resident_backward_kernel<T, MT, NW, REG, KS1>, dim3(p.g.blocks_b), dim3(NW * 32 + (REG ? kPieceWarps * 32 : 128)),
                        resident_smem(p.g, p.s.L, p.s.wp[0], p.s.stages, MT, true), st, q) == cudaSuccess;
}
template <typename T, int MT, bool REG>
bool backward_t(const ResidentMlp& p, cudaStream_t st, bool ready) {
    if (p.s.L == 1 && p.s.wp[0] <= 128) {
        const int w = image_width(1, p.s.wp[0]);
        bool ok = true;
        if (p.s.tpart == nullptr) {
            ok = w == 32 ? backward_t<T, MT, 8, REG, 2>(p, st, ready) : w == 64 ? backward_t<T, MT, 8, REG, 4>(p, st, ready)
               : w == 96 ? backward_t<T, MT, 8, REG, 6>(p, st, ready) : false;
            if constexpr (!REG)      // (97 wide and more have 91 pieces at least, and registers hold 64)
                if (w == 128) ok = backward_t<T, MT, 8, REG, 8>(p, st, ready);
        }
        if (p.s.tpart == nullptr && !ready) return ok;
        return ok && backward_t<T, MT, 8, REG, 0>(p, st, ready);      // the time terms are in the general code
    }
    if constexpr (!REG)
        if (chain_warps(p.s.L, p.s.wp) != 8) return backward_t<T, MT, 16, false, 0>(p, st, ready);
    return backward_t<T, MT, 8, REG, 0>(p, st, ready);
}
template <typename T>
bool backward_t(const ResidentMlp& p, cudaStream_t st, bool ready) {
    if (p.g.mt_b == 1) return p.partial != nullptr ? backward_t<T, 1, true>(p, st, ready) : backward_t<T, 1, false>(p, st, ready);
    return p.partial != nullptr ? backward_t<T, 2, true>(p, st, ready) : backward_t<T, 2, false>(p, st, ready);
}

}  // namespace

// The line is the shared memory of a block: weights once, and backward every layer input of a step's stages (about 95 K weights at 8 rows a
// block, fewer at 16); beyond it the weights stream (small_mlp.cu).  8 rows a block while that gives every SM one block at most: half the epilogue
// and half the rows' reads per SM.  Training pass of 8 RK4 steps unless it says otherwise, ms streamed / resident: 64-64-64 at 1500 samples 0.72 / 0.48;
// 64-128-64 at 2300 0.95 / 0.55; 40-136-136-40 at 2300 1.23 / 0.63; 72-160-72 at 1300 0.81 / 0.48; 32-96-96-32, float16 dynamic, 16 steps, at 200
// 2.52 / 1.58; linear 100 wide, 40 steps, at 300 1.56 / 0.75; linear 128 wide forward, 40 steps, at 4000 0.50 / 0.16; 64-240-240-64 forward at 1000
// 0.23 / 0.11.  Chains of 16 warps hold two row tiles at most (four spill).
ResidentPlan plan_resident(mpode_dtype dt, int B, int L, const int* wp, bool bias, bool time) {
    ResidentPlan g;
    if (dt == MPODE_F32 || L < 1 || L > SMALL_MAX_L || wp[0] > 256) return g;
    int floats = 0;
    for (int l = 0; l <= L; ++l) {
        if (wp[l] > 1000) return g;
        g.sw[l] = image_width(L, wp[l]) + 8;
    }
    for (int l = 0; l < L; ++l) {
        g.w_at[l] = g.w_elems;
        g.w_elems += image_width(L, wp[l + 1]) * g.sw[l];
        g.b_at[l] = floats;
        floats += up16(wp[l + 1]);
    }
    g.t_at = floats;
    floats += up16(wp[1]);
    g.image_bytes = (g.w_elems * 2 + floats * 4 + 15) / 16 * 16;
    const int sms = sm_count();
    auto tiles = [&](int most) { int mt = 1; while (mt < most && (B + 8 * mt - 1) / (8 * mt) > sms) mt *= 2; return mt; };
    g.mt_f = tiles(chain_warps(L, wp) == 8 ? 4 : 2); g.blocks_f = (B + 8 * g.mt_f - 1) / (8 * g.mt_f);
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
    if (blocks > sm_count() * 4) blocks = sm_count() * 4;
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
