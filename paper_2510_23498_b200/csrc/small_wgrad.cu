// Weight, bias and time-column gradients of the row-local paths: dW_l = sum over the rows of dZ_{l+1}^T X_l from the slabs of layer inputs and
// cotangents, all layers and steps of a chunk in one launch.  The rows of all stages of a step are one matrix of stages * B rows, in pieces
// of 64 (float32: 32) that the blocks of a cluster share out among themselves; a block keeps a 64 x 64 piece of a layer's gradient in
// registers, its eight warps split over the piece and over the rows of a stage of the ring, and the cluster's sums meet in distributed shared
// memory, added in a fixed order.  The bias gradient and the time column are two more columns (ones, stage times) of the pieces in the
// first column of pieces.  CHECK (a policy that looks for overflow): the sums meet once per step, before the factor h / S, and an entry of
// the step's gradient that does not fit the format raises the flag.
// Measured, us a launch (pieces of 32 x 32 or 16 x 16 a block, float32 a launch per layer and step): 72-200-200-72, 4000 rows 13.9 (35), four such steps
// checked 53 (142); 64-64, two steps of 4096 rows 18.0 (57); 64-256-256-64, 4096 rows, float32 43 (111; 403 M multiply-adds, 11 us at full rate);
// 56-56, 11 steps of 46 rows, float32 30 (131).  Few rows: 120-392-120, 360 rows 6.9 (7.7); 128-256-128, 16 steps of 64 rows, checked 34 (31);
// 32-40-32, 5 steps of 180 rows, checked 20 (15.6); 152-312-64-200-152, 2 steps of 237 rows, checked 14.3 (13.0).
// What bounds it is the rows' way from the L2 (16 KB a stage at about 64 bytes a cycle and SM), the fill of the ring, and with few rows the
// meeting of the sums.  16-bit formats multiply with mma.sync.  float32 holds 8 x 8 sums a thread and reads four 16-byte words for 64
// multiply-adds.
#include "small_mlp.h"

#include "profiler.h"
#include "tc_ptx.cuh"
#include "tensormap.h"

#include <type_traits>

namespace mpode {
using namespace tc;
namespace {

constexpr int kThreads = 256, kTile = 64, kMaxCluster = 8;
template <typename T> struct Geo {
    static constexpr int E = 16 / sizeof(T), Pieces = kTile / E, Rows = 512 / Pieces;      // elements of 16 bytes; rows of a stage
    static constexpr int LD = sizeof(T) == 4 ? kTile : kTile + 8;                          // (eight 16-bit rows hit eight 16-byte slots)
    static constexpr int Groups = sizeof(T) == 4 ? 4 : 2;                                  // threads' groups that share out a stage's rows
    static constexpr int Stages = sizeof(T) == 4 ? 6 : 4, Blocks = sizeof(T) == 4 ? 1 : 2;  // of the ring; blocks that share an SM
    static constexpr int StageBytes = 2 * Rows * LD * (int)sizeof(T);
    static constexpr int GroupThreads = kThreads / Groups, Quads = sizeof(T) == 4 ? 20 : 10;      // of a group; sums of a thread, in fours
    static constexpr int Smem = Stages * StageBytes + Groups * Quads * GroupThreads * 16;
};

struct Items { int first[SMALL_MAX_L + 1]; int S; };

__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
}
__device__ __forceinline__ float4 lds_of(uint32_t addr, int rank) {      // 16 bytes of another block's shared memory
    uint32_t a;
    float4 v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(addr), "r"(rank));
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a) : "memory");
    return v;
}

// A thread's share of the 64 x 64 piece and of the two columns of sums.
// 16-bit: warp = 32 x 32 of the piece (two of two), half of the stage's rows.
template <typename T> struct Sums {
    float w[2][4][4], s[2][4];
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                s[m][i] = 0.f;
#pragma unroll
                for (int n = 0; n < 4; ++n) w[m][n][i] = 0.f;
            }
    }
    __device__ __forceinline__ void add(float c, const Sums& o) {
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                s[m][i] = fmaf(c, o.s[m][i], s[m][i]);
#pragma unroll
                for (int n = 0; n < 4; ++n) w[m][n][i] = fmaf(c, o.w[m][n][i], w[m][n][i]);
            }
    }
    // rows 64 of a stage; tau: of each of this thread's rows; `sums`: whether the two columns are wanted
    template <typename F>
    __device__ __forceinline__ void stage(uint32_t A, uint32_t B, bool sums, F&& tau) {
        constexpr int LD = Geo<T>::LD;
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, m0 = (warp & 1) * 32, n0 = ((warp >> 1) & 1) * 32;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int k0 = ((warp >> 2) * 2 + q) * 16;
            uint32_t a[2][4], b[2][4];
#pragma unroll
            for (int m = 0; m < 2; ++m) ldm4_t(A + (uint32_t)(((k0 + (lane & 7) + (lane >> 4) * 8) * LD + m0 + m * 16 + ((lane >> 3) & 1) * 8) * 2), a[m]);
#pragma unroll
            for (int n = 0; n < 2; ++n) ldm4_t(B + (uint32_t)(((k0 + (lane & 7) + ((lane >> 3) & 1) * 8) * LD + n0 + n * 16 + (lane >> 4) * 8) * 2), b[n]);
#pragma unroll
            for (int m = 0; m < 2; ++m)
#pragma unroll
                for (int n = 0; n < 4; ++n) mma_k16<T>(w[m][n], a[m], b[n >> 1][2 * (n & 1)], b[n >> 1][2 * (n & 1) + 1]);
            if (sums && n0 == 0) {      // column 0: ones, column 1: the rounded stage time of the row
                uint32_t o0 = 0u, o1 = 0u;
                const int c = lane >> 2, k = k0 + 2 * (lane & 3);
                if (c == 0) o0 = o1 = cvt_pack<T>(1.f, 1.f);
                else if (c == 1) { o0 = cvt_pack<T>(tau(k), tau(k + 1)); o1 = cvt_pack<T>(tau(k + 8), tau(k + 9)); }
#pragma unroll
                for (int m = 0; m < 2; ++m) mma_k16<T>(s[m], a[m], o0, o1);
            }
        }
    }
    // The sums in fours, as they lie in the registers: four f of thread t of a group at [f][t].  (Rows of the piece instead took three times as
    // long to meet: scattered words, and an index worked out for each.)
    __device__ __forceinline__ void put(float4* red, int, int, float = 1.f, bool = false) const {
        red += (threadIdx.x >> 7) * 10 * 128 + (threadIdx.x & 127);
#pragma unroll
        for (int m = 0; m < 2; ++m) {
#pragma unroll
            for (int n = 0; n < 4; ++n) red[(m * 4 + n) * 128] = make_float4(w[m][n][0], w[m][n][1], w[m][n][2], w[m][n][3]);
            red[(8 + m) * 128] = make_float4(s[m][0], s[m][1], s[m][2], s[m][3]);
        }
    }
    // where word i of four f of thread t goes: row r + 8 (i / 2), column c + i % 2; or, f >= 8, the bias (i even) and time column of that row
    static __device__ __forceinline__ bool place(int f, int t, int& r, int& c) {      // whether it is one of the sums
        const int warp = t >> 5, lane = t & 31, n0 = (warp >> 1) * 32;
        r = (warp & 1) * 32 + (lane >> 2) + (f < 8 ? f >> 2 : f - 8) * 16;
        c = f < 8 ? n0 + (f & 3) * 8 + 2 * (lane & 3) : n0 + (lane & 3);      // (of the sums: those of column 0)
        return f >= 8;
    }
    static constexpr __device__ int row(int i, bool) { return 8 * (i >> 1); }
    static constexpr __device__ int col(int i) { return i & 1; }
    static constexpr __device__ bool time(int, int i) { return i & 1; }
};
// float32: a group of 64 threads has the whole piece, 8 x 8 a thread (two by two squares of 4), and every fourth of the stage's rows
template <> struct Sums<float> {
    float w[8][8], b[8], t[8];
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            b[i] = t[i] = 0.f;
#pragma unroll
            for (int j = 0; j < 8; ++j) w[i][j] = 0.f;
        }
    }
    __device__ __forceinline__ void add(float c, const Sums& o) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            b[i] = fmaf(c, o.b[i], b[i]);
            t[i] = fmaf(c, o.t[i], t[i]);
#pragma unroll
            for (int j = 0; j < 8; ++j) w[i][j] = fmaf(c, o.w[i][j], w[i][j]);
        }
    }
    template <typename F>
    __device__ __forceinline__ void stage(uint32_t A, uint32_t B, bool sums, F&& tau) {
        const int g = threadIdx.x >> 6, tx = threadIdx.x & 7, ty = (threadIdx.x >> 3) & 7;
#pragma unroll 4
        for (int q = 0; q < Geo<float>::Rows / 4; ++q) {
            const int k = g * (Geo<float>::Rows / 4) + q;
            const uint32_t ra = A + (uint32_t)((k * kTile + ty * 4) * 4), rb = B + (uint32_t)((k * kTile + tx * 4) * 4);
            const uint4 a0 = lds128(ra), a1 = lds128(ra + 128), b0 = lds128(rb), b1 = lds128(rb + 128);
            const float av[8] = {__uint_as_float(a0.x), __uint_as_float(a0.y), __uint_as_float(a0.z), __uint_as_float(a0.w),
                                 __uint_as_float(a1.x), __uint_as_float(a1.y), __uint_as_float(a1.z), __uint_as_float(a1.w)};
            const float bv[8] = {__uint_as_float(b0.x), __uint_as_float(b0.y), __uint_as_float(b0.z), __uint_as_float(b0.w),
                                 __uint_as_float(b1.x), __uint_as_float(b1.y), __uint_as_float(b1.z), __uint_as_float(b1.w)};
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < 8; ++j) w[i][j] = fmaf(av[i], bv[j], w[i][j]);
            if (sums && tx == 0) {
                const float tk = tau(k);
#pragma unroll
                for (int i = 0; i < 8; ++i) { b[i] += av[i]; t[i] = fmaf(av[i], tk, t[i]); }
            }
        }
    }
    // red = (or, with `add`, +=) k times the sums that lie in the piece; a thread's own words
    __device__ __forceinline__ void put(float4* red, int rows, int cols, float k = 1.f, bool add = false) const {
        const int tx = threadIdx.x & 7, ty = (threadIdx.x >> 3) & 7;
        red += (threadIdx.x >> 6) * 20 * 64 + (threadIdx.x & 63);
        auto one = [&](int f, const float* v) {
            const float4 o = add ? red[f * 64] : make_float4(0.f, 0.f, 0.f, 0.f);
            red[f * 64] = make_float4(fmaf(k, v[0], o.x), fmaf(k, v[1], o.y), fmaf(k, v[2], o.z), fmaf(k, v[3], o.w));
        };
#pragma unroll
        for (int f = 0; f < 16; ++f)
            if (ty * 4 + (f >> 3) * 32 < rows && tx * 4 + (f & 1) * 32 < cols) one(f, &w[f >> 1][4 * (f & 1)]);
        if (tx != 0) return;
#pragma unroll
        for (int h = 0; h < 2; ++h) { one(16 + h, b + 4 * h); one(18 + h, t + 4 * h); }
    }
    static __device__ __forceinline__ bool place(int f, int t, int& r, int& c) {
        const int tx = t & 7, ty = t >> 3;
        r = ty * 4 + (f < 16 ? ((f >> 1) & 3) + (f >> 3) * 32 : (f & 1) * 32);
        c = f < 16 ? tx * 4 + (f & 1) * 32 : tx;
        return f >= 16;
    }
    static constexpr __device__ int row(int i, bool sum) { return sum ? i : 0; }
    static constexpr __device__ int col(int i) { return i; }
    static __device__ __forceinline__ bool time(int f, int) { return f >= 18; }
};

// look: 0 at no step's gradient, 1 at each of several, 2 at each as it is added (launches of one step; float32)
enum { kNo, kEach, kAsAdded };
template <typename T, int CHECK>
__global__ void __launch_bounds__(kThreads, Geo<T>::Blocks) small_wgrad_kernel(const __grid_constant__ SmallMlp p, const __grid_constant__ Items items) {
    chain_begin();
    using G = Geo<T>;
    constexpr int kStages = G::Stages;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ float taus[SMALL_MAX_CHUNK][RK_MAX_STAGES];
    const int S = items.S, rank = (int)blockIdx.x % S, item = (int)blockIdx.x / S;
    int l = 0;
    while (item >= items.first[l + 1]) ++l;
    const int M = p.wp[l + 1], N = p.wp[l], tn = (N + kTile - 1) / kTile;
    const int m0 = (item - items.first[l]) / tn * kTile, n0 = (item - items.first[l]) % tn * kTile;
    const bool time = p.time && l == 0, sums = n0 == 0 && (p.bias || time);
    const int KR = p.stages * p.B, pieces = (KR + G::Rows - 1) / G::Rows;
    const int mine = rank < pieces ? (pieces - rank + S - 1) / S : 0;      // pieces rank, rank + S, ... of every step
    if ((int)threadIdx.x < p.count * RK_MAX_STAGES) taus[threadIdx.x >> 2][threadIdx.x & 3] = p.scal[p.step_hi - (int)(threadIdx.x >> 2)].tau16[threadIdx.x & 3];
    const T* Z = (const T*)p.zs[l + 1];
    const T* X = (const T*)p.xs[l];
    const uint32_t ring = smem_u32(smem);
    float4* red = (float4*)(smem + kStages * G::StageBytes);
    // this thread's four pieces of 16 bytes of a stage: row, column, operand are the same for every stage
    int fs = 0, fi = 0, fslot = 0;
    auto fetch = [&]() {
        if (fs < p.count && mine > 0) {
            const int row0 = (rank + S * fi) * G::Rows;
            const uint32_t dst = ring + (uint32_t)(fslot * G::StageBytes);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int id = (int)threadIdx.x + kThreads * (q & 1), r = id / G::Pieces, c = id % G::Pieces * G::E;
                const bool isA = q < 2;
                const int row = row0 + r, W = isA ? M : N, col = (isA ? m0 : n0) + c;
                const bool on = row < KR && col < W;
                const T* src = (isA ? Z : X) + ((long long)fs * KR + row) * W + col;
                copy16(dst + (uint32_t)(((isA ? 0 : G::Rows) + r) * G::LD + c) * (uint32_t)sizeof(T), on ? src : Z, on);
            }
            if (++fi == mine) { fi = 0; ++fs; }
            if (++fslot == kStages) fslot = 0;
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // What earlier steps gave: a second set of sums; in float32, which has no registers for it, the words that the sums meet in.  Checked float32
    // passes need those for each step's sums: their steps meet one by one, in memory.
    // (Checked 16-bit launches of one step too: the sums meet once instead of twice.)
    constexpr bool kTotal = sizeof(T) == 2, kBySteps = CHECK == kAsAdded;
    static_assert(kTotal || CHECK != kEach, "no second set of sums");
    Sums<T> acc, tot;
    acc.zero();
    if (kTotal) tot.zero();
    // the piece's rows and columns (worked out where they are used: no registers for them in the loop over the rows)
    auto rows_in = [&]() { return min(kTile, p.wr[l + 1] - m0); };
    auto cols_in = [&]() { return min(kTile, p.wr[l] - n0); };
    const uint32_t red_u = smem_u32(red);
    const int t = (int)threadIdx.x % G::GroupThreads;
    auto all_sync = [&]() { if (S == 1) __syncthreads(); else cluster_sync(); };
    // The groups' and the blocks' sums meet in fours; each thread of the cluster takes up to kMine.  What a thread does here is a chain of single
    // instructions, some five cycles each with two warps a scheduler: the parameters' places are worked out once a launch.
    constexpr int kMine = G::Quads / G::Groups;
    const int f0 = (int)threadIdx.x / G::GroupThreads + G::Groups * rank, step = G::Groups * S;
    auto places = [&](int f, int (&at)[4]) {      // the parameters of four f, or -1
        const int in_full = p.wr[l] + (time ? 1 : 0), mr = rows_in(), nc = cols_in();
        const int w_at = (int)p.woff[l] + m0 * in_full + n0, b_at = p.bias && sums ? (int)p.boff[l] + m0 : -1, t_at = time && sums ? (int)p.woff[l] + m0 * in_full + p.wr[l] : -1;
        int r, c;
        const bool sum = Sums<T>::place(f, t, r, c), on = f < G::Quads;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int ri = r + Sums<T>::row(i, sum);
            const bool tm = Sums<T>::time(f, i);
            at[i] = !on || ri >= mr ? -1
                  : !sum ? (c + Sums<T>::col(i) < nc ? w_at + ri * in_full + c + Sums<T>::col(i) : -1)
                  : c != 0 ? -1 : tm ? (t_at >= 0 ? t_at + ri * in_full : -1) : (b_at >= 0 ? b_at + ri : -1);
        }
    };
    uint32_t mine_on = 0u;      // bit 4 u + i: word i of this thread's u-th four is a parameter's
    if (CHECK == kEach) {
#pragma unroll 1
        for (int u = 0; u < kMine; ++u) {
            int at[4];
            places(f0 + u * step, at);
#pragma unroll
            for (int i = 0; i < 4; ++i) mine_on |= (at[i] >= 0 ? 1u : 0u) << (4 * u + i);
        }
    }
    // before the blocks': the groups' sums, so that a four is one read of each block
    auto own_sums = [&]() {
        if (S == 1) return;
        __syncthreads();
        const int mr = rows_in(), nc = cols_in();
        float4 v[kMine];
#pragma unroll
        for (int u = 0; u < kMine; ++u) {
            v[u] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (!kTotal) {
                int r, c;
                if (Sums<T>::place(u * G::Groups + (int)threadIdx.x / G::GroupThreads, t, r, c) ? c != 0 || !sums : r >= mr || c >= nc) continue;
            }
            const float4* q = red + u * kThreads + threadIdx.x;
            v[u] = *q;
#pragma unroll
            for (int g = 1; g < G::Groups; ++g) { const float4 o = q[g * G::Quads * G::GroupThreads]; v[u].x += o.x; v[u].y += o.y; v[u].z += o.z; v[u].w += o.w; }
        }
#pragma unroll
        for (int u = 0; u < kMine; ++u) red[u * kThreads + threadIdx.x] = v[u];
    };
    auto sum_of = [&](int f, float (&v)[4], auto at_once) {      // groups first, then blocks, in ascending order; words of how many blocks in flight
        v[0] = v[1] = v[2] = v[3] = 0.f;
        auto take = [&](auto sets, auto&& word) {
            float4 q[decltype(sets)::value];
#pragma unroll
            for (int g = 0; g < decltype(sets)::value; ++g) q[g] = word((g * G::Quads + f) * G::GroupThreads + t);
#pragma unroll
            for (int g = 1; g < decltype(sets)::value; ++g) { q[0].x += q[g].x; q[0].y += q[g].y; q[0].z += q[g].z; q[0].w += q[g].w; }
            v[0] += q[0].x; v[1] += q[0].y; v[2] += q[0].z; v[3] += q[0].w;
        };
        if (S == 1) { take(std::integral_constant<int, G::Groups>(), [&](int w) { return red[w]; }); return; }
#pragma unroll(decltype(at_once)::value)
        for (int z = 0; z < S; ++z) take(std::integral_constant<int, 1>(), [&](int w) { return lds_of(red_u + (uint32_t)w * 16u, z); });
    };
    bool bad = false;
    auto check = [&](const Sums<T>& w) {      // a step's gradient, before the factor h / S
        w.put(red, rows_in(), cols_in());
        own_sums();
        all_sync();
        auto look = [&](int u) {
            const uint32_t on = mine_on >> (4 * u) & 15u;
            if (on == 0u) return;
            float v[4];
            sum_of(f0 + u * step, v, std::integral_constant<int, 4>());
#pragma unroll
            for (int i = 0; i < 4; ++i) bad |= !(fabsf(v[i]) < low_limit<T>()) && (on >> i & 1u);
        };
        if (S == 1) {
#pragma unroll
            for (int u = 0; u < kMine; ++u) look(u);
        } else {
#pragma unroll 1
            for (int u = 0; u * step < G::Quads; ++u) look(u);
        }
        all_sync();      // (no block goes on, or ends, while another reads its sums)
    };
    int at[kMine][4];
    auto find_places = [&]() {
#pragma unroll
        for (int u = 0; u < kMine; ++u) {
            at[u][0] = at[u][1] = at[u][2] = at[u][3] = -1;
            if (u * step < G::Quads) places(f0 + u * step, at[u]);
        }
    };
    // out = beta out + cf times the sum of the words put; what is added to is requested before the barrier
    auto add_to = [&](float beta, float cf) {
        float before[kMine][4];
#pragma unroll
        for (int u = 0; u < kMine; ++u) {
            if (u * step >= G::Quads) break;
#pragma unroll
            for (int i = 0; i < 4; ++i) before[u][i] = at[u][i] >= 0 && beta != 0.f ? beta * p.out[at[u][i]] : 0.f;
        }
        own_sums();
        all_sync();
#pragma unroll
        for (int u = 0; u < kMine; ++u) {
            if (u * step >= G::Quads) break;
            bool any = false;
#pragma unroll
            for (int i = 0; i < 4; ++i) any |= at[u][i] >= 0;
            if (!any) continue;
            float v[4];
            sum_of(f0 + u * step, v, std::integral_constant<int, kMaxCluster>());
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (at[u][i] >= 0) {
                    if (kBySteps) bad |= !(fabsf(v[i]) < low_limit<T>());
                    p.out[at[u][i]] = kBySteps ? fmaf(cf, v[i], before[u][i]) : before[u][i] + v[i];
                }
        }
        all_sync();
    };
    if (kBySteps || !kTotal) find_places();      // (while the first rows are on their way; 16-bit loops have no registers for them)
    for (int k = 0; k < kStages - 1; ++k) fetch();
    __syncthreads();
    int slot = 0;
    for (int s = 0; s < p.count; ++s) {
        for (int i = 0; i < mine; ++i) {
            asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
            __syncthreads();
            fetch();      // into the stage that every thread has left behind at this barrier
            const int row0 = (rank + S * i) * G::Rows;
            const uint32_t A = ring + (uint32_t)(slot * G::StageBytes);
            acc.stage(A, A + (uint32_t)(G::Rows * G::LD * sizeof(T)), sums, [&](int k) {
                const int row = row0 + k;
                return taus[s][(row >= p.B) + (row >= 2 * p.B) + (row >= 3 * p.B)];      // (rows behind the last are zero)
            });
            if (++slot == kStages) slot = 0;
        }
        if (kBySteps) {
            acc.put(red, rows_in(), cols_in());
            add_to(s == 0 ? p.beta : 1.f, p.coef[s]);
        } else {
            if (CHECK == kEach) check(acc);
            if (kTotal) tot.add(p.coef[s], acc);
            else acc.put(red, rows_in(), cols_in(), p.coef[s], s > 0);
        }
        acc.zero();
    }
    copies_done();
    if (!kBySteps) {
        if (kTotal) { tot.put(red, 0, 0); find_places(); }
        add_to(p.beta, 1.f);
    }
    if (CHECK) warp_flag_or(p.flag, bad);
}

template <typename T, int CHECK>
bool wgrad_t(const SmallMlp& p, const Items& items, cudaStream_t st, bool ready) {
    static bool done[kMaxDevices] = {false};
    static int at_once[kMaxDevices][kMaxCluster + 1] = {{0}};      // clusters of each size that the GPU holds at once
    const int dev = current_device();
    cudaLaunchConfig_t cfg{};
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = Geo<T>::Smem;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    if (!done[dev]) {
        if (cudaFuncSetAttribute(small_wgrad_kernel<T, CHECK>, cudaFuncAttributeMaxDynamicSharedMemorySize, Geo<T>::Smem) != cudaSuccess) { cudaGetLastError(); return false; }
        cfg.numAttrs = 1;
        for (int S = 1; S <= kMaxCluster; ++S) {
            at[0].val.clusterDim.x = (unsigned)S;
            cfg.gridDim = dim3((unsigned)S);
            if (cudaOccupancyMaxActiveClusters(&at_once[dev][S], small_wgrad_kernel<T, CHECK>, &cfg) != cudaSuccess) { cudaGetLastError(); at_once[dev][S] = 0; }
        }
        done[dev] = true;
    }
    if (ready) return true;
    // the largest cluster of which all pieces' run at once, with a stage of rows for each of its blocks
    const int n = items.first[p.L], stages = (p.stages * p.B + Geo<T>::Rows - 1) / Geo<T>::Rows;
    Items it = items;
    it.S = 1;
    for (int S = 2; S <= kMaxCluster && S <= stages; ++S)
        if (at_once[dev][S] >= n) it.S = S;
    at[0].val.clusterDim.x = (unsigned)it.S;
    cfg.gridDim = dim3((unsigned)(n * it.S));
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, small_wgrad_kernel<T, CHECK>, p, it) == cudaSuccess;
}
template <typename T>
bool wgrad_t(const SmallMlp& p, const Items& items, cudaStream_t st) {
    if (p.flag == nullptr) return wgrad_t<T, kNo>(p, items, st, false);
    if constexpr (sizeof(T) == 2)
        if (p.count > 1) return wgrad_t<T, kEach>(p, items, st, false);
    return wgrad_t<T, kAsAdded>(p, items, st, false);
}
template <typename T>
bool wgrad_ready(const SmallMlp& p) {
    if constexpr (sizeof(T) == 2)
        if (!wgrad_t<T, kEach>(p, Items{}, nullptr, true)) return false;
    return wgrad_t<T, kNo>(p, Items{}, nullptr, true) && wgrad_t<T, kAsAdded>(p, Items{}, nullptr, true);
}

}  // namespace

bool small_wgrad_ready(mpode_dtype dt, const SmallMlp& p) {
    return dt == MPODE_BF16 ? wgrad_ready<__nv_bfloat16>(p) : dt == MPODE_F16 ? wgrad_ready<__half>(p) : wgrad_ready<float>(p);
}

void launch_small_wgrad(mpode_dtype dt, const SmallMlp& p, cudaStream_t st, long long* launches) {
    Items it{};
    for (int l = 0; l < p.L; ++l) it.first[l + 1] = it.first[l] + ((p.wp[l + 1] + kTile - 1) / kTile) * ((p.wp[l] + kTile - 1) / kTile);
    if (dt == MPODE_BF16) wgrad_t<__nv_bfloat16>(p, it, st);
    else if (dt == MPODE_F16) wgrad_t<__half>(p, it, st);
    else wgrad_t<float>(p, it, st);
    if (launches) ++*launches;
    if (tl_counters) {
        if (dt == MPODE_F32) tl_counters->simt += (long long)p.L * p.count;
        else ++tl_counters->fused;
    }
}

}  // namespace mpode
