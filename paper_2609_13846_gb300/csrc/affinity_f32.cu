// affinity_f32.cu -- fp32 mode of the first-order affinity (Sec. 3 "Affinity
// scores") on the CUDA cores, plus the finalize and ||w^d||^2 helpers.
//
// The fp32 mode exists for tight checks (fp32 operands, fp32 FMA); TF32
// tensor cores would not meet a 1e-5 relative error.  A block computes a tile
// of 128 x 128 (or 64 x 64) tokens and neurons, gate and up together: the X pass gives
// (alpha, beta) per (token, neuron), kept in shared memory, then each head pass
// gives (pg, pu) and Delta^2 is summed over the block's tokens.  Per-tile
// partials go to the workspace and are added into A in a fixed order, so the
// result is deterministic.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "dtp_common.cuh"

namespace dtp {
namespace f32 {

constexpr int TK = 16;        // k block
constexpr int kThreads = 256;
constexpr int kTokMin = 64;   // tokens per tile of the smaller form (the workspace is sized for it)

// Bound by the FMA pipe.  A thread owns TPT tokens x NPT neurons of gate and of up and multiplies with
// packed fma.rn.f32x2 (each half rounds as a scalar fma: the sums over k are those of a scalar loop), a
// weight pair from shared memory times an activation repeated in both halves.  8 x 8 per thread (128 x 128
// tiles, one block per SM): per k six float4 shared loads for 64 packed FMAs, which keeps the pipe and not
// the loads the limit; 4 x 4 (64 x 64 tiles, two blocks per SM) for layers with few tiles.  alpha and beta
// live in shared memory, the next k block is loaded from global memory during the current one.
// T = 1024, d = 1024, 8 heads, N = 3072 on a GB300: 4.34 ms with 4 x 4 scalar tiles, 2.80 ms with 8 x 4
// packed ones, 2.40 with 8 x 8.  There the FMA pipe is 70% busy and the shared-memory path 57%: with two
// warps a scheduler the rest is waiting at barriers, for shared loads and in the epilogues.
template <int TPT, int NPT>
struct Tile {
    static constexpr int TM = 16 * TPT;          // tokens
    static constexpr int TN = 16 * NPT;          // neurons
    static constexpr int kBlocks = NPT == 8 ? 1 : 2;   // per SM
    // floats per k of the activations and of the weights (gate, up): 16-byte rows whose start moves by
    // half the banks every 4 k, so that the transposing stores do not collide
    static constexpr int SA = TM + 4;
    static constexpr int SB = 2 * TN + 4;
    static constexpr int kStage = TK * (SA + SB);
    static constexpr int kAb = kThreads * TPT * NPT * 2;   // alpha, beta
    static constexpr size_t kSmem = sizeof(float) * (2 * kStage + kAb + 8 * TN);
};
static_assert(Tile<8, 8>::kSmem <= 227 * 1024 && 2 * (Tile<4, 4>::kSmem + 1024) <= 227 * 1024, "shared memory");

__device__ __forceinline__ void fma2(uint64_t& d, uint64_t a, uint64_t b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
__device__ __forceinline__ uint64_t twice(float v) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(v));
    return r;
}
__device__ __forceinline__ float2 unpack2(uint64_t v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}

// Neuron of the thread's j-th column: float4 groups 64 apart.
__device__ __forceinline__ int col_of(int tx, int j) { return 64 * (j >> 2) + 4 * tx + (j & 3); }

// acc_g[i][p], acc_u[i][p] = sum over k of act[t_i, k] (Wg, Wu)[n_2p, n_2p+1; k] for the thread's tokens
// t_i = t0 + TPT ty + i and neurons n_j = n0 + col_of(tx, j).  Rows and k beyond the edges read as zero.
template <int TPT, int NPT>
__device__ __forceinline__ void tile_gemm(const float* __restrict__ act, int64_t T, int d,
                                          const float* __restrict__ Wg, const float* __restrict__ Wu, int N,
                                          int64_t t0, int n0, uint64_t (&acc_g)[TPT][NPT / 2],
                                          uint64_t (&acc_u)[TPT][NPT / 2], float* stages) {
    using S = Tile<TPT, NPT>;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    constexpr int kRowsA = TPT / 4, kRowsW = NPT / 4;    // rows per thread
    const int row = tid >> 2, kq = (tid & 3) * 4;        // 64 rows x 4 float4 per round
#pragma unroll
    for (int i = 0; i < TPT; ++i)
#pragma unroll
        for (int q = 0; q < NPT / 2; ++q) acc_g[i][q] = acc_u[i][q] = 0;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    float4 ra[kRowsA], rg[kRowsW], ru[kRowsW];
    const float* pa = act + (t0 + row) * d + kq;
    const int64_t wo = static_cast<int64_t>(n0 + row) * d + kq;
    auto fetch = [&](int k0) {
        const bool k_in = k0 + kq < d;                   // d is a multiple of 8
#pragma unroll
        for (int e = 0; e < kRowsA; ++e) {
            const bool in = k_in && t0 + row + 64 * e < T;
            ra[e] = in ? *reinterpret_cast<const float4*>(pa + 64 * e * static_cast<int64_t>(d) + k0) : zero;
        }
#pragma unroll
        for (int e = 0; e < kRowsW; ++e) {
            const bool in = k_in && n0 + row + 64 * e < N;
            const int64_t o = wo + 64 * e * static_cast<int64_t>(d) + k0;
            rg[e] = in ? *reinterpret_cast<const float4*>(Wg + o) : zero;
            ru[e] = in ? *reinterpret_cast<const float4*>(Wu + o) : zero;
        }
    };
    auto stash = [&](float* st) {
        auto put = [](float* to, int stride, const float4& v) {
            to[0] = v.x, to[stride] = v.y, to[2 * stride] = v.z, to[3 * stride] = v.w;
        };
#pragma unroll
        for (int e = 0; e < kRowsA; ++e) put(st + kq * S::SA + row + 64 * e, S::SA, ra[e]);
        float* bs = st + TK * S::SA + kq * S::SB + row;
#pragma unroll
        for (int e = 0; e < kRowsW; ++e) {
            put(bs + 64 * e, S::SB, rg[e]);
            put(bs + S::TN + 64 * e, S::SB, ru[e]);
        }
    };
    fetch(0);
    stash(stages);
    __syncthreads();
    const int blocks = (d + TK - 1) / TK;
    for (int b = 0; b < blocks; ++b) {
        const bool more = b + 1 < blocks;
        if (more) fetch((b + 1) * TK);
        const float* as = stages + (b & 1) * S::kStage + TPT * ty;
        const float* bs = stages + (b & 1) * S::kStage + TK * S::SA + 4 * tx;
#pragma unroll
        for (int kk = 0; kk < TK; ++kk) {
            uint64_t a[TPT], g[NPT / 2], u[NPT / 2];
#pragma unroll
            for (int i = 0; i < TPT; i += 4) {
                const float4 v = *reinterpret_cast<const float4*>(as + kk * S::SA + i);
                a[i] = twice(v.x), a[i + 1] = twice(v.y), a[i + 2] = twice(v.z), a[i + 3] = twice(v.w);
            }
#pragma unroll
            for (int q = 0; q < NPT / 4; ++q) {
                const ulonglong2 vg = *reinterpret_cast<const ulonglong2*>(bs + kk * S::SB + 64 * q);
                const ulonglong2 vu = *reinterpret_cast<const ulonglong2*>(bs + kk * S::SB + S::TN + 64 * q);
                g[2 * q] = vg.x, g[2 * q + 1] = vg.y, u[2 * q] = vu.x, u[2 * q + 1] = vu.y;
            }
#pragma unroll
            for (int i = 0; i < TPT; ++i)
#pragma unroll
                for (int q = 0; q < NPT / 2; ++q) {
                    fma2(acc_g[i][q], a[i], g[q]);
                    fma2(acc_u[i][q], a[i], u[q]);
                }
        }
        if (more) stash(stages + ((b + 1) & 1) * S::kStage);   // its last readers passed the previous barrier
        __syncthreads();
    }
}

// Blocks: `whole` tiles (neuron tile fastest), then the remaining tiles, each split by heads over `split`
// blocks (each repeats the X pass; the first adds the activation term).
template <int TPT, int NPT>
__global__ void __launch_bounds__(kThreads, Tile<TPT, NPT>::kBlocks)
affinity_fo_f32_kernel(const float* __restrict__ X, const float* __restrict__ C, const float* __restrict__ Wg,
                       const float* __restrict__ Wu, int64_t T, int d, int G, int N, float* __restrict__ partial,
                       const float* __restrict__ rms, float* __restrict__ partial_act, int64_t whole, int split) {
    using S = Tile<TPT, NPT>;
    extern __shared__ __align__(16) float f32_smem[];
    float* stages = f32_smem;
    float2* ab = reinterpret_cast<float2*>(f32_smem + 2 * S::kStage);      // [TPT * NPT][threads]
    float* red = f32_smem + 2 * S::kStage + S::kAb;                        // [8 warps][TN]
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4, warp = tid >> 5;
    int64_t unit = blockIdx.x;
    int part = 0, parts = 1;
    if (unit >= whole) {
        part = static_cast<int>((unit - whole) % split);
        parts = split;
        unit = whole + (unit - whole) / split;
    }
    const int nt = (N + S::TN - 1) / S::TN;
    const int n0 = static_cast<int>(unit % nt) * S::TN;
    const int64_t tile = unit / nt;
    const int64_t t0 = tile * S::TM;
    const int h0 = G * part / parts, h1 = G * (part + 1) / parts;

    // sum over the block's tokens of the threads' per-neuron sums, in a fixed order, to dst[n]
    auto reduce = [&](const float (&s)[NPT], float* dst) {
#pragma unroll
        for (int j = 0; j < NPT; ++j) {
            const float v = s[j] + __shfl_xor_sync(0xFFFFFFFFu, s[j], 16);   // the warp's two token rows
            if ((tid & 16) == 0) red[warp * S::TN + col_of(tx, j)] = v;
        }
        __syncthreads();
        if (tid < S::TN && n0 + tid < N) {
            float v = 0.0f;
#pragma unroll
            for (int w = 0; w < 8; ++w) v += red[w * S::TN + tid];
            dst[n0 + tid] = v;
        }
        // red is rewritten after the next tile_gemm's barriers
    };

    uint64_t acc_g[TPT][NPT / 2], acc_u[TPT][NPT / 2];
    tile_gemm<TPT, NPT>(X, T, d, Wg, Wu, N, t0, n0, acc_g, acc_u, stages);
    {
        float act[NPT];
#pragma unroll
        for (int j = 0; j < NPT; ++j) act[j] = 0.0f;
        const bool want = rms && part == 0;
#pragma unroll
        for (int i = 0; i < TPT; ++i) {
            const int64_t t = t0 + TPT * ty + i;
            const float r = want && t < T ? rms[t] : 0.0f;
            const float ir2 = want && t < T ? 1.0f / (r * r) : 0.0f;
#pragma unroll
            for (int j = 0; j < NPT; ++j) {
                const float2 g2 = unpack2(acc_g[i][j >> 1]), u2 = unpack2(acc_u[i][j >> 1]);
                const float g = (j & 1) ? g2.y : g2.x, u = (j & 1) ? u2.y : u2.x;
                const float s = 1.0f / (1.0f + expf(-g));
                const float beta = g * s;
                ab[(NPT * i + j) * kThreads + tid] = make_float2(s * (1.0f + g * (1.0f - s)) * u, beta);
                // down-edge activation term: (silu(g) u)^2 / r'^2
                if (want && t < T) act[j] = fmaf((beta * u) * (beta * u), ir2, act[j]);
            }
        }
        if (want) reduce(act, partial_act + tile * N);
    }
    for (int h = h0; h < h1; ++h) {
        tile_gemm<TPT, NPT>(C + static_cast<int64_t>(h) * T * d, T, d, Wg, Wu, N, t0, n0, acc_g, acc_u, stages);
        float sum[NPT];
#pragma unroll
        for (int j = 0; j < NPT; ++j) sum[j] = 0.0f;
#pragma unroll
        for (int i = 0; i < TPT; ++i)
#pragma unroll
            for (int j = 0; j < NPT; ++j) {
                const float2 pg2 = unpack2(acc_g[i][j >> 1]), pu2 = unpack2(acc_u[i][j >> 1]);
                const float pg = (j & 1) ? pg2.y : pg2.x, pu = (j & 1) ? pu2.y : pu2.x;
                const float2 w = ab[(NPT * i + j) * kThreads + tid];
                const float dlt = w.x * pg + w.y * pu;
                sum[j] = fmaf(dlt, dlt, sum[j]);
            }
        reduce(sum, partial + (tile * G + h) * N);
    }
}

// A[g,k] += sum over heads h of row g (qpg consecutive heads) and token tiles, head by head.
__global__ void f32_reduce_kernel(const float* __restrict__ partial, float* __restrict__ A, int G, int N,
                                  int64_t tiles, const float* __restrict__ partial_act, float* __restrict__ act2,
                                  int qpg) {
    const int64_t heads_n = static_cast<int64_t>(G) * N;
    const int64_t total_a = static_cast<int64_t>(G / qpg) * N;
    const int64_t total = total_a + (act2 ? N : 0);
    for (int64_t idx = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; idx < total;
         idx += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        float s = 0.0f;
        if (idx < total_a) {
            const int64_t g = idx / N, k = idx % N;
            for (int64_t h = g * qpg; h < (g + 1) * qpg; ++h)
                for (int64_t t = 0; t < tiles; ++t) s += partial[t * heads_n + h * N + k];
            A[idx] += s;
        } else {
            const int64_t k = idx - total_a;
            for (int64_t t = 0; t < tiles; ++t) s += partial_act[t * N + k];
            act2[k] += s;
        }
    }
}

size_t workspace_bytes(int64_t T, int d, int G, int N) {
    (void)d;
    const int64_t tiles = (T + kTokMin - 1) / kTokMin;
    return kWorkspaceHeader + static_cast<size_t>(tiles) * (G + 1) * N * sizeof(float);
}

int launch_grouped(const float* X, const float* C, const float* Wg, const float* Wu, int64_t T, int d, int G, int N,
                   float* A, void* workspace, cudaStream_t stream, const float* rms, float* act2, int qpg) {
    if (qpg < 1 || G % qpg) return DTP_ERR_ARG;
    const int64_t tiles64 = (T + kTokMin - 1) / kTokMin;
    if (tiles64 > 65535) return DTP_ERR_UNSUPPORTED;
    float* partial = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(workspace) + kWorkspaceHeader);
    float* partial_act = partial + tiles64 * static_cast<int64_t>(G) * N;
    const bool want_act = rms && act2;
    int dev = 0, sms = 0;
    DTP_CUDA_TRY(cudaGetDevice(&dev));
    DTP_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    // 128 x 128 tiles when there are enough for two thirds of the SMs, else 64 x 64 ones; the tiles left
    // over after the last full round are split by heads so that they spread over the chip
    const int64_t large_tiles = static_cast<int64_t>((N + 127) / 128) * ((T + 127) / 128);
    const bool large = 3 * large_tiles >= 2 * sms;
    const int64_t tiles = large ? (T + 127) / 128 : tiles64;
    const int64_t units = large ? large_tiles : static_cast<int64_t>((N + 63) / 64) * tiles64;
    const int64_t slots = large ? sms : 2 * sms;
    const int64_t whole = units / slots * slots, left = units - whole;
    int split = 1;
    if (left > 0) split = static_cast<int>(slots / left < G ? slots / left : G);
    const int64_t blocks = whole + left * split;
    if (blocks > 0x7FFFFFFF) return DTP_ERR_UNSUPPORTED;
    auto kernel = large ? affinity_fo_f32_kernel<8, 8> : affinity_fo_f32_kernel<4, 4>;
    const size_t smem = large ? Tile<8, 8>::kSmem : Tile<4, 4>::kSmem;
    DTP_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem)));
    kernel<<<static_cast<unsigned>(blocks), kThreads, smem, stream>>>(X, C, Wg, Wu, T, d, G, N, partial,
                                                                     want_act ? rms : nullptr, partial_act, whole, split);
    DTP_CUDA_TRY(cudaGetLastError());
    const int64_t total = static_cast<int64_t>(G / qpg) * N + (want_act ? N : 0);
    const int rblocks = static_cast<int>((total + 255) / 256 < 1024 ? (total + 255) / 256 : 1024);
    f32_reduce_kernel<<<rblocks, 256, 0, stream>>>(partial, A, G, N, tiles, partial_act, want_act ? act2 : nullptr,
                                                  qpg);
    DTP_CUDA_TRY(cudaGetLastError());
    return DTP_OK;
}

int launch(const float* X, const float* C, const float* Wg, const float* Wu, int64_t T, int d, int G, int N,
           float* A, void* workspace, cudaStream_t stream, const float* rms, float* act2) {
    return launch_grouped(X, C, Wg, Wu, T, d, G, N, A, workspace, stream, rms, act2, 1);
}

// S_down[g,k] = act2[k] / T_total * bn[g,k]
__global__ void down_finalize_kernel(const float* __restrict__ act2, const float* __restrict__ bn, int G, int N,
                                     float inv_t, float* __restrict__ S) {
    const int64_t total = static_cast<int64_t>(G) * N;
    for (int64_t idx = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; idx < total;
         idx += static_cast<int64_t>(gridDim.x) * blockDim.x)
        S[idx] = act2[idx % N] * inv_t * bn[idx];
}

}  // namespace f32

// --------------------------------------------------------------------------
// finalize: A[h,k] *= wd_sqnorm[k] / T_total
// --------------------------------------------------------------------------
__global__ void finalize_kernel(float* __restrict__ A, int G, int N, float inv_t, const float* __restrict__ wd) {
    const int64_t total = static_cast<int64_t>(G) * N;
    for (int64_t idx = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; idx < total;
         idx += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int k = static_cast<int>(idx % N);
        const float f = wd ? wd[k] : 1.0f;
        A[idx] = A[idx] * f * inv_t;
    }
}

// out[k] = sum_i W_down[i,k]^2 over the d rows of W_down [d, N].  Bound by reading W_down once.  LPR
// lanes read VEC neighbouring columns each (16 bytes where the rows allow it), the block's other threads
// take other rows, and a tree in shared memory adds the row sums in a fixed order.  One thread per column
// left 12 blocks walking 1024 rows in turn on a 1024 x 3072 matrix: 72 us cold, 7.8 us now.
constexpr int kSqThreads = 256;
template <typename T, int VEC, int LPR>
__global__ void __launch_bounds__(kSqThreads) down_sqnorm_kernel(const T* __restrict__ W, int d, int N,
                                                                 float* __restrict__ out) {
    constexpr int kRows = kSqThreads / LPR;          // rows in flight
    constexpr int kCols = LPR * VEC;
    __shared__ float sums[kRows][kCols + 1];
    const int lane = threadIdx.x % LPR, slot = threadIdx.x / LPR;
    const int k0 = blockIdx.x * kCols + lane * VEC;
    float acc[VEC];
#pragma unroll
    for (int v = 0; v < VEC; ++v) acc[v] = 0.0f;
    if (k0 < N) {                                    // VEC > 1: N is a multiple of VEC
#pragma unroll 8
        for (int i = slot; i < d; i += kRows) {
            union { uint4 q; T e[VEC]; } w;
            const T* src = W + static_cast<int64_t>(i) * N + k0;
            if constexpr (VEC > 1) w.q = *reinterpret_cast<const uint4*>(src);
            else w.e[0] = *src;
#pragma unroll
            for (int v = 0; v < VEC; ++v) {
                const float x = static_cast<float>(w.e[v]);
                acc[v] = fmaf(x, x, acc[v]);
            }
        }
    }
#pragma unroll
    for (int v = 0; v < VEC; ++v) sums[slot][lane * VEC + v] = acc[v];
    __syncthreads();
    for (int half = kRows / 2; half > 0; half >>= 1) {
        for (int x = threadIdx.x; x < half * kCols; x += kSqThreads)
            sums[x / kCols][x % kCols] += sums[x / kCols + half][x % kCols];
        __syncthreads();
    }
    static_assert(kCols <= kSqThreads, "a thread per column");
    const int k = blockIdx.x * kCols + threadIdx.x;
    if (threadIdx.x < kCols && k < N) out[k] = sums[0][threadIdx.x];
}

int launch_down_finalize(const float* act2, const float* bn, int G, int N, int64_t T_total, float* S,
                         cudaStream_t stream) {
    const int64_t total = static_cast<int64_t>(G) * N;
    const int blocks = static_cast<int>((total + 255) / 256 < 1024 ? (total + 255) / 256 : 1024);
    f32::down_finalize_kernel<<<blocks, 256, 0, stream>>>(act2, bn, G, N,
                                                         static_cast<float>(1.0 / static_cast<double>(T_total)), S);
    DTP_CUDA_TRY(cudaGetLastError());
    return DTP_OK;
}

// Top-group share of each layer (Sec. 5 diagnostic): the mean over neurons with a non-zero column of
// max_g A[g,k] / sum_g A[g,k], in fp64.  One block per layer; the per-thread sums are combined in a
// fixed order (warp butterflies, then the warps in index order), so the result is reproducible.
__global__ void __launch_bounds__(1024) top_share_kernel(const float* __restrict__ A, int G, int N,
                                                         double* __restrict__ share) {
    __shared__ double ssum[32];
    __shared__ int scnt[32];
    const float* a = A + static_cast<int64_t>(blockIdx.x) * G * N;
    double acc = 0.0;
    int cnt = 0;
    for (int k = threadIdx.x; k < N; k += blockDim.x) {
        double tot = 0.0, mx = 0.0;
        for (int g = 0; g < G; ++g) {
            const double v = a[static_cast<int64_t>(g) * N + k];
            tot += v;
            mx = v > mx ? v : mx;
        }
        if (tot > 0.0) {
            acc += mx / tot;
            ++cnt;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        acc += __shfl_xor_sync(0xFFFFFFFFu, acc, o);
        cnt += __shfl_xor_sync(0xFFFFFFFFu, cnt, o);
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) ssum[warp] = acc, scnt[warp] = cnt;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        int c = 0;
        for (int w = 0; w < static_cast<int>(blockDim.x >> 5); ++w) t += ssum[w], c += scnt[w];
        share[blockIdx.x] = c ? t / c : 0.0;
    }
}

int launch_top_share(const float* A, int layers, int G, int N, double* share, cudaStream_t stream) {
    top_share_kernel<<<layers, 1024, 0, stream>>>(A, G, N, share);
    DTP_CUDA_TRY(cudaGetLastError());
    return DTP_OK;
}

int launch_finalize(float* A, int G, int N, int64_t T_total, const float* wd, cudaStream_t stream) {
    const int64_t total = static_cast<int64_t>(G) * N;
    const int blocks = static_cast<int>((total + 255) / 256 < 1024 ? (total + 255) / 256 : 1024);
    finalize_kernel<<<blocks, 256, 0, stream>>>(A, G, N, static_cast<float>(1.0 / static_cast<double>(T_total)), wd);
    DTP_CUDA_TRY(cudaGetLastError());
    return DTP_OK;
}

// 16-byte loads where every row starts on a 16-byte boundary, else one column per lane, 32 a row.  4 lanes a
// row keep 64 rows in flight in a block; where that is half of them or more, and N still gives two blocks
// an SM with it, 32 lanes (96 x 100000 fp32, cold: 10.6 us against 18.0; 256 x 100000 bf16: 21.5 against 19.0).
template <typename T>
static int down_sqnorm(const T* W, int d, int N, float* out, cudaStream_t stream) {
    constexpr int kVec = static_cast<int>(16 / sizeof(T));
    int dev = 0, sms = 0;
    DTP_CUDA_TRY(cudaGetDevice(&dev));
    DTP_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const bool words = N % kVec == 0 && aligned16(W);
    if (words && d <= 128 && N / (32 * kVec) >= 2 * sms)
        down_sqnorm_kernel<T, kVec, 32><<<(N + 32 * kVec - 1) / (32 * kVec), kSqThreads, 0, stream>>>(W, d, N, out);
    else if (words)
        down_sqnorm_kernel<T, kVec, 4><<<(N + 4 * kVec - 1) / (4 * kVec), kSqThreads, 0, stream>>>(W, d, N, out);
    else
        down_sqnorm_kernel<T, 1, 32><<<(N + 31) / 32, kSqThreads, 0, stream>>>(W, d, N, out);
    DTP_CUDA_TRY(cudaGetLastError());
    return DTP_OK;
}

int launch_down_sqnorm(const void* W, int d, int N, int dtype, float* out, cudaStream_t stream) {
    return dtype == DTP_BF16 ? down_sqnorm(static_cast<const __nv_bfloat16*>(W), d, N, out, stream)
                             : down_sqnorm(static_cast<const float*>(W), d, N, out, stream);
}

}  // namespace dtp
