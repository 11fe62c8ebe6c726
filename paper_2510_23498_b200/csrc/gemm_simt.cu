// Contractions on the CUDA cores: C(m, n) = sum_k A(m, k) B(n, k), fp32 accumulation in a fixed order (deterministic), and the
// fused epilogues of the velocity layers.  They serve every shape and all three low formats: the float32 path (TF32 cannot meet
// the 1e-5 accuracy target) and the fallback for shapes the tensor-core kernels do not take.  Two kernels: one for plain operands
// (gemm_dense_kernel) and a general one that also has an implicit 3x3-convolution view of one operand (gemm_simt_kernel).
#include <cooperative_groups.h>

#include "common.cuh"
#include "tensormap.h"

namespace mpode {
namespace {

constexpr int BM = 64, BN = 64, BK = 16, TM = 4, TN = 4;
constexpr int kGemmThreads = (BM / TM) * (BN / TN);  // 256

// Element (i, k) of an operand.  In the convolution view the pixel index is the row index of operand A
// (pix_is_k = false) or the reduction index of operand B (pix_is_k = true); the other index is (tap, channel).
template <typename T>
__device__ __forceinline__ float load_operand(const T* __restrict__ p, long long rs, long long ks, int i, int k,
                                              int rows, int K, bool conv, bool pix_is_k, int H, int W, int Cd, int Ct,
                                              float tau) {
    if (i >= rows || k >= K) return 0.f;
    if (!conv) return Low<T>::to_f(p[i * rs + k * ks]);
    int pixel = pix_is_k ? k : i;
    int tc = pix_is_k ? i : k;
    int tap = tc / Ct, c = tc - tap * Ct;
    int x = pixel % W;
    int y = (pixel / W) % H;
    int dy = tap / 3 - 1, dx = tap % 3 - 1;
    if (y + dy < 0 || y + dy >= H || x + dx < 0 || x + dx >= W) return 0.f;
    if (c >= Cd) return tau;
    return Low<T>::to_f(p[((long long)pixel + (long long)dy * W + dx) * Cd + c]);
}

// The layer epilogue of one output element; returns whether the rounded value of an input gradient
// is not finite.
template <typename T>
__device__ __forceinline__ bool finish_element(const GemmArgs& g, int m, int n, float v) {
    if (g.epi == EPI_FWD) {
        if (g.out2 != nullptr && m >= g.m_split) {
            ((T*)g.out2)[(long long)(m - g.m_split) * g.ldo + n] = Low<T>::from_f(v);
        } else {
            if (g.bias != nullptr) v += Low<T>::to_f(((const T*)g.bias)[n]);
            if (g.wt != nullptr) v = fmaf(g.tau, Low<T>::to_f(((const T*)g.wt)[n]), v);
            ((T*)g.out)[(long long)m * g.ldo + n] = Low<T>::from_f(act_fwd(g.act, v));
        }
    } else if (g.epi == EPI_DGRAD) {
        if (g.hprev != nullptr) v *= act_deriv_from_output(g.act, Low<T>::to_f(((const T*)g.hprev)[(long long)m * g.ldh + n]));
        const T q = Low<T>::from_f(v);
        ((T*)g.out)[(long long)m * g.ldo + n] = q;
        return Low<T>::nonfinite(q);
    } else if (g.epi == EPI_WGRAD) {
        float* o = (float*)g.out + (long long)m * g.ldo + n;
        *o = v + (g.beta != 0.f ? *o : 0.f);
    } else {
        ((float*)g.out)[(long long)m * g.ldo + n] = v;
    }
    return false;
}

template <typename T>
__global__ void __launch_bounds__(kGemmThreads) gemm_simt_kernel(GemmArgs g) {
    chain_begin();
    __shared__ float As[BK][BM + 4];
    __shared__ float Bs[BK][BN + 4];
    const T* A = (const T*)g.A;
    const T* B = (const T*)g.B;
    int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
    int tx = threadIdx.x % (BN / TN), ty = threadIdx.x / (BN / TN);
    float acc[TM][TN];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = 0.f;

    int k_begin = 0, k_end = g.K;
    if (g.split_k > 1) {
        int chunk = ((g.K + g.split_k - 1) / g.split_k + BK - 1) / BK * BK;
        k_begin = blockIdx.z * chunk;
        k_end = min(g.K, k_begin + chunk);
    }
    // When the reduction index is the contiguous one, consecutive threads walk k; otherwise they walk rows.
    bool a_kfast = (g.conv_on == 1) || (g.a_ks == 1);
    bool b_kfast = (g.conv_on != 2) && (g.b_ks == 1);
    for (int k0 = k_begin; k0 < k_end; k0 += BK) {
#pragma unroll
        for (int it = 0; it < (BM * BK) / kGemmThreads; ++it) {
            int idx = threadIdx.x + it * kGemmThreads;
            int mm = a_kfast ? idx / BK : idx % BM;
            int kk = a_kfast ? idx % BK : idx / BM;
            int kg = k0 + kk;
            As[kk][mm] = load_operand<T>(A, g.a_rs, g.a_ks, m0 + mm, kg < k_end ? kg : g.K, g.M, g.K, g.conv_on == 1, false,
                                         g.conv_h, g.conv_w, g.conv_cd, g.conv_ct, g.conv_tau);
        }
#pragma unroll
        for (int it = 0; it < (BN * BK) / kGemmThreads; ++it) {
            int idx = threadIdx.x + it * kGemmThreads;
            int nn = b_kfast ? idx / BK : idx % BN;
            int kk = b_kfast ? idx % BK : idx / BN;
            int kg = k0 + kk;
            Bs[kk][nn] = load_operand<T>(B, g.b_rs, g.b_ks, n0 + nn, kg < k_end ? kg : g.K, g.N, g.K, g.conv_on == 2, true,
                                         g.conv_h, g.conv_w, g.conv_cd, g.conv_ct, g.conv_tau);
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            float a[TM], b[TN];
#pragma unroll
            for (int i = 0; i < TM; ++i) a[i] = As[kk][ty * TM + i];
#pragma unroll
            for (int j = 0; j < TN; ++j) b[j] = Bs[kk][tx * TN + j];
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
    }

    bool bad = false;
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        int m = m0 + ty * TM + i;
#pragma unroll
        for (int j = 0; j < TN; ++j) {
            int n = n0 + tx * TN + j;
            if (m >= g.M || n >= g.N) continue;
            if (g.epi == EPI_WGRAD && g.split_k > 1) g.partial[((long long)blockIdx.z * g.M + m) * g.N + n] = acc[i][j];
            else bad |= finish_element<T>(g, m, n, acc[i][j]);
        }
    }
    if (g.epi == EPI_DGRAD) warp_flag_or(g.flag, bad);
}

// ---------------------------------------------------------------- plain operands
// 64 x 64 output tile, 256 threads with 4 x 4 outputs each, reduction chunks of 32 through two shared-memory buffers (the next
// chunk's global loads are in registers while this one is multiplied).  Both operands have the reduction index contiguous
// (KFAST: layers and input gradients) or the row index (weight gradients).  The layer shapes of a small network give a handful of
// tiles, so a cluster of up to 8 blocks cuts the reduction range and the blocks' sums meet in distributed shared memory, added in
// ascending rank: no scratch, no second launch, and each block finishes its share of the tile's rows.  FMA issue bounds a chunk
// (32 x 32 cycles against 24 x 32 of shared-memory reads).  Measured, float32 MLP 64 -> 256 -> 256 -> 64, 1024 samples, 16 RK4 steps,
// forward and backward: 33.4 ms with the general kernel (no slices, column sums in launches of their own), 10.8 ms with this one.
constexpr int DM = 64, DN = 64, DK = 32, kDenseThreads = 256, kDenseLd = DM + 4;

template <typename T> struct alignas(4 * sizeof(T)) Quad { T v[4]; };

// four consecutive elements along the contiguous index `c` of line `l` (limits lc, ll; zero outside)
template <typename T>
__device__ __forceinline__ float4 load_quad(const T* __restrict__ p, long long ld, int l, int c, int ll, int lc, bool vec) {
    float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
    if (l >= ll || c >= lc) return r;
    const T* q = p + (long long)l * ld + c;
    if (vec && c + 3 < lc) {
        const Quad<T> w = *reinterpret_cast<const Quad<T>*>(q);
        r = make_float4(Low<T>::to_f(w.v[0]), Low<T>::to_f(w.v[1]), Low<T>::to_f(w.v[2]), Low<T>::to_f(w.v[3]));
    } else {
        r.x = Low<T>::to_f(q[0]);
        if (c + 1 < lc) r.y = Low<T>::to_f(q[1]);
        if (c + 2 < lc) r.z = Low<T>::to_f(q[2]);
        if (c + 3 < lc) r.w = Low<T>::to_f(q[3]);
    }
    return r;
}

template <typename T, bool KFAST>
__global__ void __launch_bounds__(kDenseThreads) gemm_dense_kernel(GemmArgs g, int per_slice, int vec_a, int vec_b) {
    chain_begin();
    namespace cg = cooperative_groups;
    __shared__ __align__(16) float As[2][DK][kDenseLd];
    __shared__ __align__(16) float Bs[2][DK][kDenseLd];
    __shared__ float rows[DM];
    const T* A = (const T*)g.A;
    const T* B = (const T*)g.B;
    const int m0 = blockIdx.y * DM, n0 = blockIdx.x * DN, t = threadIdx.x;
    const int tx = t & 15, ty = t >> 4;
    const int k_begin = blockIdx.z * per_slice, k_end = min(g.K, k_begin + per_slice);
    // the bias gradient is the row sum of A over the reduction range: taken along by the first column of tiles
    const bool sum_rows = !KFAST && (g.row_sum != nullptr || g.row_sum_time != nullptr) && blockIdx.x == 0;
    float acc[4][4], rs[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;

    float4 ra[2], rb[2];
    auto fetch = [&](int k0) {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            if (KFAST) {      // line = row, lanes walk the rows: the transposed stores below hit 32 banks
                const int r = t & 63, k = k0 + 4 * ((t >> 6) + 4 * u);
                ra[u] = load_quad<T>(A, g.a_rs, m0 + r, k, g.M, k_end, vec_a);
                rb[u] = load_quad<T>(B, g.b_rs, n0 + r, k, g.N, k_end, vec_b);
            } else {
                const int r = 4 * (t & 15), k = k0 + (t >> 4) + 16 * u;
                ra[u] = load_quad<T>(A, g.a_ks, k, m0 + r, k_end, g.M, vec_a);
                rb[u] = load_quad<T>(B, g.b_ks, k, n0 + r, k_end, g.N, vec_b);
            }
        }
    };
    auto stash = [&](int buf) {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            if (KFAST) {
                const int r = t & 63, k = 4 * ((t >> 6) + 4 * u);
                As[buf][k][r] = ra[u].x; As[buf][k + 1][r] = ra[u].y; As[buf][k + 2][r] = ra[u].z; As[buf][k + 3][r] = ra[u].w;
                Bs[buf][k][r] = rb[u].x; Bs[buf][k + 1][r] = rb[u].y; Bs[buf][k + 2][r] = rb[u].z; Bs[buf][k + 3][r] = rb[u].w;
            } else {
                const int r = 4 * (t & 15), k = (t >> 4) + 16 * u;
                *reinterpret_cast<float4*>(&As[buf][k][r]) = ra[u];
                *reinterpret_cast<float4*>(&Bs[buf][k][r]) = rb[u];
            }
        }
    };
    if (k_begin < k_end) {
        fetch(k_begin);
        stash(0);
    }
    __syncthreads();
    int buf = 0;
    for (int k0 = k_begin; k0 < k_end; k0 += DK, buf ^= 1) {
        const bool more = k0 + DK < k_end;
        if (more) fetch(k0 + DK);
#pragma unroll 8
        for (int kk = 0; kk < DK; ++kk) {
            const float4 a4 = *reinterpret_cast<const float4*>(&As[buf][kk][ty * 4]);
            const float4 b4 = *reinterpret_cast<const float4*>(&Bs[buf][kk][tx * 4]);
            const float a[4] = {a4.x, a4.y, a4.z, a4.w}, b[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
            if (sum_rows) {
#pragma unroll
                for (int i = 0; i < 4; ++i) rs[i] += a[i];
            }
        }
        if (more) stash(buf ^ 1);
        __syncthreads();
    }

    bool bad = false;
    auto put_row_sum = [&](int m, float s) {
        if (g.row_sum != nullptr) g.row_sum[m] = s + (g.beta != 0.f ? g.row_sum[m] : 0.f);
        if (g.row_sum_time != nullptr) {
            float* o = g.row_sum_time + (long long)m * g.ldo;
            *o = fmaf(g.tau, s, g.beta != 0.f ? *o : 0.f);
        }
        if (g.row_sum_raw != nullptr) g.row_sum_raw[m] = s;
    };
    const int S = (int)gridDim.z;
    if (S == 1) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int m = m0 + ty * 4 + i;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int n = n0 + tx * 4 + j;
                if (m < g.M && n < g.N) bad |= finish_element<T>(g, m, n, acc[i][j]);
            }
            if (sum_rows && tx == 0 && m < g.M) put_row_sum(m, rs[i]);
        }
    } else {      // the slices of one tile are one cluster: rank r adds up the tile's rows [r, r + 1) * DM / S
        cg::cluster_group cl = cg::this_cluster();
        float(*tile)[kDenseLd] = (float(*)[kDenseLd]) & As[0][0][0];      // 64 rows: the two operand buffers together
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            *reinterpret_cast<float4*>(&tile[ty * 4 + i][tx * 4]) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
            if (sum_rows && tx == 0) rows[ty * 4 + i] = rs[i];
        }
        cl.sync();
        const int rank = (int)blockIdx.z, per = DM / S;
        for (int e = t; e < per * DN; e += kDenseThreads) {
            const int r = rank * per + e / DN, c = e % DN, m = m0 + r, n = n0 + c;
            if (m >= g.M || n >= g.N) continue;
            float v = 0.f;
            for (int z = 0; z < S; ++z) v += *cl.map_shared_rank(&tile[r][c], z);
            bad |= finish_element<T>(g, m, n, v);
        }
        if (sum_rows && t < per && m0 + rank * per + t < g.M) {
            float v = 0.f;
            for (int z = 0; z < S; ++z) v += *cl.map_shared_rank(&rows[rank * per + t], z);
            put_row_sum(m0 + rank * per + t, v);
        }
        cl.sync();      // no block leaves while another reads its shared memory
    }
    if (g.epi == EPI_DGRAD) warp_flag_or(g.flag, bad);
}

// Blocks of a cluster share a reduction of at least 64: as many (up to 8) as it takes to give every SM a block.
int dense_slices(int tiles, int K) {
    int s = 1;
    while (s < 8 && tiles * s < sm_count() && K >= 64 * 2 * s) s *= 2;
    return s;
}

template <typename T>
bool launch_dense(const GemmArgs& g, cudaStream_t st) {
    const bool rfast = g.a_rs == 1 && g.b_rs == 1, kfast = g.a_ks == 1 && g.b_ks == 1 && !(g.epi == EPI_WGRAD && rfast);
    if (g.conv_on != 0 || g.split_k > 1 || (!kfast && !rfast)) return false;
    const long long lda = kfast ? g.a_rs : g.a_ks, ldb = kfast ? g.b_rs : g.b_ks;
    const int vec_a = lda % 4 == 0 && ((uintptr_t)g.A % (4 * sizeof(T))) == 0, vec_b = ldb % 4 == 0 && ((uintptr_t)g.B % (4 * sizeof(T))) == 0;
    const int tn = (g.N + DN - 1) / DN, tm = (g.M + DM - 1) / DM;
    if (tm > 65535) return false;
    int S = dense_slices(tn * tm, g.K);
    const int per = ((g.K + S - 1) / S + DK - 1) / DK * DK;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)tn, (unsigned)tm, (unsigned)S);
    cfg.blockDim = dim3(kDenseThreads);
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = 1; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = (unsigned)S;
    cfg.attrs = at;
    cfg.numAttrs = S > 1 ? 2 : 1;
    const bool clean = cudaPeekAtLastError() == cudaSuccess;
    const cudaError_t e = kfast ? cudaLaunchKernelEx(&cfg, gemm_dense_kernel<T, true>, g, per, vec_a, vec_b) : cudaLaunchKernelEx(&cfg, gemm_dense_kernel<T, false>, g, per, vec_a, vec_b);
    if (e != cudaSuccess && clean) cudaGetLastError();      // the general kernel runs instead: this error is dealt with (an earlier one is not)
    return e == cudaSuccess;
}

__global__ void splitk_reduce_kernel(const float* __restrict__ partial, int S, int M, int N, float* __restrict__ out,
                                     long long ldo, float beta, int keep_m, int keep_n) {
    chain_begin();
    long long n_el = (long long)M * N;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n_el; i += (long long)gridDim.x * blockDim.x) {
        if (i / N >= keep_m || i % N >= keep_n) continue;
        float s = 0.f;
        for (int z = 0; z < S; ++z) s += partial[(long long)z * n_el + i];
        float* o = out + (i / N) * ldo + (i % N);
        *o = (beta != 0.f ? *o : 0.f) + s;
    }
}

// The same four columns at a time (N a multiple of 4, fewer than 2^31 elements): the slices are still added in ascending order per
// element.  VEC: the destination rows are 16-byte aligned too; otherwise (a row with an appended column, cropped padding) its four
// elements are written one by one.
template <bool VEC>
__global__ void splitk_reduce4_kernel(const float4* __restrict__ partial, int S, unsigned slice4, unsigned n4, unsigned N4, float* __restrict__ out,
                                      long long ldo, float beta, unsigned keep_n) {
    chain_begin();
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += gridDim.x * blockDim.x) {
        float4 s = partial[i];
        for (int z = 1; z < S; ++z) {
            const float4 v = partial[(size_t)z * slice4 + i];
            s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
        }
        const unsigned row = i / N4, col = 4 * (i - row * N4);
        float* o = out + (long long)row * ldo + col;
        if (VEC) {
            if (beta != 0.f) {
                const float4 old = *reinterpret_cast<const float4*>(o);
                s.x += old.x; s.y += old.y; s.z += old.z; s.w += old.w;
            }
            *reinterpret_cast<float4*>(o) = s;
        } else {
            const float v[4] = {s.x, s.y, s.z, s.w};
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (col + e < keep_n) o[e] = (beta != 0.f ? o[e] : 0.f) + v[e];
        }
    }
}

void reduce_slices(const float* partial, int S, int M, int N, float* out, long long ldo, float beta, cudaStream_t st, int crop_m = 0, int crop_n = 0) {
    const int keep_m = crop_m > 0 ? crop_m : M, keep_n = crop_n > 0 ? crop_n : N;
    const long long n_el = (long long)M * N;
    if (N % 4 == 0 && n_el < 0x7fffffffLL && ((uintptr_t)partial & 15) == 0 && S >= 1) {
        const unsigned N4 = (unsigned)(N / 4), n4 = (unsigned)keep_m * N4, slice4 = (unsigned)(n_el / 4);
        int blocks = (int)((n4 + 255) / 256);
        if (blocks > 148 * 8) blocks = 148 * 8;
        const float4* p4 = reinterpret_cast<const float4*>(partial);
        if (keep_n == N && ldo % 4 == 0 && ((uintptr_t)out & 15) == 0) launch_chain(splitk_reduce4_kernel<true>, dim3(blocks), dim3(256), 0, st, p4, S, slice4, n4, N4, out, ldo, beta, N);
        else launch_chain(splitk_reduce4_kernel<false>, dim3(blocks), dim3(256), 0, st, p4, S, slice4, n4, N4, out, ldo, beta, keep_n);
        return;
    }
    int blocks = (int)((n_el + 255) / 256);
    if (blocks > 148 * 8) blocks = 148 * 8;
    launch_chain(splitk_reduce_kernel, dim3(blocks), dim3(256), 0, st, partial, S, M, N, out, ldo, beta, keep_m, keep_n);
}

}  // namespace

void launch_splitk_reduce(const float* partial, int S, int M, int N, float* out, long long ldo, float beta, cudaStream_t st,
                          long long* launches, int crop_m, int crop_n) {
    reduce_slices(partial, S, M, N, out, ldo, beta, st, crop_m, crop_n);
    if (launches) ++*launches;
}

bool launch_gemm_simt(mpode_dtype dt, const GemmArgs& g, cudaStream_t st, long long* launches) {
    if (g.M <= 0 || g.N <= 0) return true;
    const bool dense = dt == MPODE_BF16 ? launch_dense<__nv_bfloat16>(g, st) : (dt == MPODE_F16 ? launch_dense<__half>(g, st) : launch_dense<float>(g, st));
    if (dense) {
        if (launches) ++*launches;
        return true;
    }
    dim3 grid((g.N + BN - 1) / BN, (g.M + BM - 1) / BM, g.split_k > 1 ? g.split_k : 1);
    if (dt == MPODE_BF16) launch_chain(gemm_simt_kernel<__nv_bfloat16>, dim3(grid), dim3(kGemmThreads), 0, st, g);
    else if (dt == MPODE_F16) launch_chain(gemm_simt_kernel<__half>, dim3(grid), dim3(kGemmThreads), 0, st, g);
    else launch_chain(gemm_simt_kernel<float>, dim3(grid), dim3(kGemmThreads), 0, st, g);
    if (launches) ++*launches;
    if (g.split_k > 1) {
        reduce_slices(g.partial, g.split_k, g.M, g.N, (float*)g.out, g.ldo, g.beta, st);
        if (launches) ++*launches;
    }
    return false;
}

}  // namespace mpode
