// search.cu -- the layout optimiser (search.cuh) on layers that fit in shared memory, the whole-model
// search's normalisation and scoring kernels, and the host side: how a layer is split, workspaces, launches.
#include <atomic>

#include "search.cuh"

namespace dtp {
namespace search {

Kernels kernels_in_shared(int D) { return kernels_for<true>(D); }

int64_t unlabelled_count(int G, int D) {
    const int cap = G / D;
    uint64_t n = fact_u64(G);
    for (int l = 0; l < D; ++l) n /= fact_u64(cap);
    return static_cast<int64_t>(n / fact_u64(D));
}

// floor(q 2^43 / total) for q <= total, 2^39 <= total < 2^62 (the largest q is at least 2^39).
// m is the reciprocal word floor((2^128 - 1) / tn) - 2^64 of tn = total << s, s its leading zeros
// (2 .. 24): the estimate from it is at most one too small, and the remainder, below 2^63, says so.
__device__ __forceinline__ int64_t unit_mass(uint64_t q, uint64_t total, uint64_t m, int s) {
    const uint64_t y = q << (s - 1);
    uint64_t n = (y + __umul64hi(y, m)) >> 20;
    const uint64_t rem = (q << kNormBits) - n * total;
    n += rem >= total;
    return static_cast<int64_t>(n);
}

// One team per matrix: m < L is the up edge of layer m, m >= L the down edge of layer m - L; each block
// takes a part of the matrix.  head / nu (may be null) receive the contiguous start layout.  The state
// was cleared before.  Three passes over 98 KB and a division per entry: one block per matrix took 18 us
// for 28 Qwen-shaped layers, four take 8.
__global__ void __launch_bounds__(kThreads, 1)
chain_normalize_kernel(const float* __restrict__ S_up, const float* __restrict__ S_down, int L, int G, int N, int D,
                       int64_t* __restrict__ nbuf, int32_t* __restrict__ head, int32_t* __restrict__ nu,
                       ChainState* st, int* ws_status, int64_t* J_q, double* J, int32_t* iters_done,
                       int64_t* __restrict__ tops) {
    Shared& sh = shared();
    Team tm = make_team();
    const int m = blockIdx.x / tm.cl;
    const int64_t GN = static_cast<int64_t>(G) * N;
    const int64_t per = (GN / tm.cl + 3) / 4 * 4 + 4;            // whole 16-byte words of the matrix
    const int64_t at = per * tm.rank < GN ? per * tm.rank : GN;
    const int64_t n = GN - at < per ? GN - at : per;
    const float* src = (m < L ? S_up + m * GN : S_down + (m - L) * GN) + at;
    int64_t* dst = nbuf + m * GN + at;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *J_q = 0;
        *J = 0.0;
        if (iters_done) *iters_done = 0;
        st->prev = INT64_MIN;
    }
    if (m < L && head && tm.rank == 0 && threadIdx.x < G) head[m * G + threadIdx.x] = (threadIdx.x * D) / G;
    if (m < L && nu)
        for (int k = tm.rank * kThreads + threadIdx.x; k < N; k += static_cast<int>(tm.cl) * kThreads)
            nu[static_cast<int64_t>(m) * N + k] = static_cast<int>((static_cast<int64_t>(k) * D) / N);
    uint32_t top = 0, unused = 0;
    for_each_a(src, n, [&](int64_t, float a) { top = max(top, valid_bits(a)); });
    team_min_max(unused, top, tm);
    if (top == 0xFFFFFFFFu) {
        if (threadIdx.x == 0 && tm.rank == 0) {
            atomicMin(ws_status, static_cast<int>(DTP_ERR_ARG));
            st->done = 1;
        }
        team_sync(tm);
        return;
    }
    const float amax = __uint_as_float(top);
    int e = 0;
    if (amax > 0.0f) frexpf(amax, &e);
    int64_t part = 0;
    for_each_a(src, n, [&](int64_t, float a) { part += quantize_bits(a, e, kNormPreBits); });
    part = block_sum_i64(part);
    if (threadIdx.x == 0) sh.xl[tm.lph][0] = part;
    team_sum_i64(1, tm);
    const uint64_t total = static_cast<uint64_t>(sh.B[0]);
    team_sync(tm);                     // no block leaves while a peer may still read its shared memory
    if (total == 0) {
        if (threadIdx.x == 0 && tm.rank == 0) tops[m] = 0;
        for (int64_t i = threadIdx.x; i < n; i += kThreads) dst[i] = 0;
        return;
    }
    const int s = __clzll(static_cast<long long>(total));
    const uint64_t mr = static_cast<uint64_t>(~static_cast<unsigned __int128>(0) / (total << s));   // less 2^64
    if (threadIdx.x == 0 && tm.rank == 0)
        tops[m] = unit_mass(static_cast<uint64_t>(quantize_bits(amax, e, kNormPreBits)), total, mr, s);
    for_each_a(src, n, [&](int64_t i, float a) {
        dst[i] = unit_mass(static_cast<uint64_t>(quantize_bits(a, e, kNormPreBits)), total, mr, s);
    });
}

// J of a given layout, per edge (Eq. objective): one block per edge, edge 2i =
// up_i (h_i(g) == nu_i(k)), edge 2i+1 = down_i (nu_i(k) == h_{i+1}(g)).
// Entries of h or nu outside [0, D) are reported as DTP_ERR_ARG.
__global__ void __launch_bounds__(kThreads, 1)
chain_edge_kernel(int Lyr, int G, int N, int D, const int64_t* __restrict__ nbuf, const int32_t* __restrict__ head,
                  const int32_t* __restrict__ nu, int64_t* __restrict__ edge, ChainState* st, int* ws_status) {
    Shared& sh = shared();
    if (*reinterpret_cast<volatile int*>(&st->done)) return;
    const int e = blockIdx.x;
    const int i = e >> 1;
    const bool up = (e & 1) == 0;
    const int64_t GN = static_cast<int64_t>(G) * N;
    const int64_t* n = nbuf + (up ? i : Lyr + i) * GN;
    const int32_t* hg = head + static_cast<int64_t>(up ? i : i + 1) * G;
    const int32_t* nk = nu + static_cast<int64_t>(i) * N;
    if (threadIdx.x < G) sh.h[threadIdx.x] = hg[threadIdx.x];
    __syncthreads();
    int bad = 0;
    if (threadIdx.x < G && (sh.h[threadIdx.x] < 0 || sh.h[threadIdx.x] >= D)) bad = 1;
    int64_t part = 0;
    for (int k = threadIdx.x; k < N; k += kThreads) {
        const int l = nk[k];
        if (l < 0 || l >= D) {
            bad = 1;
            continue;
        }
        for (int g = 0; g < G; ++g)
            if (sh.h[g] == l) part += n[static_cast<int64_t>(g) * N + k];
    }
    bad = __syncthreads_or(bad);
    const int64_t tot = block_sum_i64(part);
    if (threadIdx.x == 0) {
        edge[e] = tot;
        if (bad) atomicMin(ws_status, static_cast<int>(DTP_ERR_ARG));
    }
}

__global__ void chain_total_kernel(int n_edges, const int64_t* __restrict__ edge, const ChainState* st,
                                   int64_t* J_q, double* J) {
    if (threadIdx.x != 0 || st->done) return;
    int64_t t = 0;
    for (int e = 0; e < n_edges; ++e) t += edge[e];
    *J_q = t;
    *J = ldexp(static_cast<double>(t), -kNormBits);
}

// --------------------------------------------------------------------- host --

int64_t partition_count(int G, int D) {
    // G! / ((G/D)!)^D
    double f[GMAX + 1];
    f[0] = 1.0;
    for (int i = 1; i <= GMAX; ++i) f[i] = f[i - 1] * i;
    double c = f[G];
    for (int l = 0; l < D; ++l) c /= f[G / D];
    return static_cast<int64_t>(c + 0.5);
}

// Workspace of a layer that may have to live in global memory (where no cluster can hold it): int64
// gains, int32 labels and N more words, which cover the slices of any team (slice_bytes: 2 D + 11 bytes a
// neuron fewer, against 16 neurons and 256 bytes a block of rounding, on more than 3000 neurons).
static size_t global_layer_bytes(int N, int D) {
    return align_up(static_cast<size_t>(N) * D * sizeof(int64_t) + static_cast<size_t>(N) * sizeof(int32_t), 256) +
           align_up(static_cast<size_t>(N) * sizeof(uint64_t), 256);
}

// Layers that one block always holds in shared memory: no global buffer is ever needed.
static bool fits_block(int N, int D) {
    return align_up(static_cast<size_t>(N) * D * sizeof(int64_t) + static_cast<size_t>(N) * sizeof(int32_t), 256) <=
           kWorkspaceFree;
}

struct Plan {
    int cl;        // blocks per team
    int global;    // 1: the layer lives in the workspace
    size_t dyn;
    View vw;
};

static int slice_np(int N, int cl) { return static_cast<int>(align_up((N + cl - 1) / cl, 16)); }

// Teams of `cl` blocks (a power of two) of these kernels that the device can hold at once, 0 if none;
// found once per device (every kernel here runs 512 threads and asks for at most the same shared memory,
// which leaves one block per SM).
static int resident_teams(int dev, int cl) {
    static std::atomic<int> cache[64][5];          // teams + 1, 0: not yet known
    int slot = 0;
    while ((1 << slot) < cl) ++slot;
    const int known = dev < 64 ? cache[dev][slot].load(std::memory_order_relaxed) : 0;
    if (known) return known - 1;
    int n = 0;
    auto kern = kernels_in_shared(8).search;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kData + kSmemBudget)) ==
            cudaSuccess &&
        cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = cl;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3(cl);
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = kData + kSmemBudget;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) n = 0;
    }
    (void)cudaGetLastError();
    if (dev < 64) cache[dev][slot].store(n + 1, std::memory_order_relaxed);
    return n;
}

// Blocks per team for `teams` layers of `rows` score rows at once.  A layer that fits in one block is
// gathered there and the other blocks build gains and sum columns: one layer alone takes two blocks,
// which a pass capped at one SM less than the chip leaves free (it rounds down; 28 Qwen-shaped layers,
// D = 4, whole model: 493 us with one block each, 415 with two, 354 with four; one layer, D = 2: 76, 60
// and 52, but beside the affinity pass four blocks cost 1% of a step and two nothing).  A larger layer
// takes as few blocks as hold it, then up to 8 (the portable cluster size) while a block has more than
// kSliceTarget neurons and every team has its SMs to itself (N = 14336, D = 8: 4.5 ms in one block with
// the layer in global memory, 0.25 ms in 8).  A layer too large for that lives in the workspace and takes
// the largest team, or 8 blocks where such teams run one after another: its passes wait for L2, and fewer
// layers at a time stay there (N = 262144, D = 2: one layer 5.6 ms in one block, 0.26 in 16; 160 layers
// 10.8 ms in a block each, 6.3 in teams of 8).
constexpr int kSliceTarget = 1024, kGatheredTarget = 768;
static int make_plan(int64_t teams, int rows, int N, int D, Plan* p) {
    int dev = 0, sms = 0;
    DTP_CUDA_TRY(cudaGetDevice(&dev));
    DTP_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    int most = 1;
    while (most < kMaxCluster && resident_teams(dev, 2 * most) > 0) most *= 2;
    int cl = 1;
    while (cl < kMaxCluster && slice_bytes(slice_np(N, cl), D) > kSmemBudget) cl *= 2;
    if (cl > most || slice_bytes(slice_np(N, cl), D) > kSmemBudget) {
        if (fits_block(N, D)) return DTP_ERR_WORKSPACE;   // no room was asked for: never with the budgets above
        cl = most > 8 && teams > resident_teams(dev, most) ? 8 : most;
        if (cl * align_up(slice_bytes(slice_np(N, cl), D), 256) > global_layer_bytes(N, D)) return DTP_ERR_WORKSPACE;
        p->cl = cl;
        p->global = 1;
        p->dyn = 0;
        p->vw.np = slice_np(N, cl);
        p->vw.gathered = cl == 1;
        p->vw.rows = 0;
        return DTP_OK;
    }
    const bool gathered = slice_bytes(slice_np(N, 1), D) <= kSmemBudget;
    const int target = gathered ? kGatheredTarget : kSliceTarget;
    const int limit = gathered && teams == 1 ? 2 : 8;
    while (cl < limit && 2 * cl <= most && (N + cl - 1) / cl > target && teams * 2 * cl <= sms) cl *= 2;
    p->cl = cl;
    p->global = 0;
    p->vw.np = slice_np(N, cl);
    p->vw.gathered = gathered;
    const size_t m = align_up(slice_bytes(gains_np(p->vw, N), D), 16), q = static_cast<size_t>(rows) * p->vw.np * 6;
    p->vw.rows = m + q <= kSmemBudget ? rows : 0;
    p->dyn = m + (p->vw.rows ? q : 0);
    return DTP_OK;
}

// Launches `teams` teams of kern.  cooperative: all of them at once, or none (DTP_ERR_UNSUPPORTED when the
// device cannot hold them).
template <class... Params, class... Args>
static int launch_teams(void (*kern)(Params...), bool cooperative, int64_t teams, const Plan& p, cudaStream_t stream,
                        Args... args) {
    DTP_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kData + kSmemBudget)));
    if (p.cl > 8) DTP_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = static_cast<unsigned>(p.cl);
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeCooperative;
    attr[1].val.cooperative = 1;
    cfg.gridDim = dim3(static_cast<unsigned>(teams * p.cl));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kData + p.dyn;
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = cooperative ? 2 : (p.cl > 1 ? 1 : 0);
    const cudaError_t err = cudaLaunchKernelEx(&cfg, kern, static_cast<Params>(args)...);
    if (cooperative && err == cudaErrorCooperativeLaunchTooLarge) {
        (void)cudaGetLastError();
        return DTP_ERR_UNSUPPORTED;
    }
    DTP_CUDA_TRY(err);
    DTP_CUDA_TRY(cudaGetLastError());
    return DTP_OK;
}

size_t workspace_bytes(int layers, int G, int N, int D) {
    (void)G;
    size_t b = kWorkspaceHeader + align_up(static_cast<size_t>(layers) * sizeof(int), 256);
    if (!fits_block(N, D)) b += static_cast<size_t>(layers) * global_layer_bytes(N, D);
    return b;
}

int launch(const float* A, int layers, int G, int N, int D, int iters, int32_t* head, int32_t* nu, int64_t* score_q,
           double* score, int32_t* iters_done, void* workspace, cudaStream_t stream) {
    uint8_t* ws = reinterpret_cast<uint8_t*>(workspace);
    int* ws_status = reinterpret_cast<int*>(ws);
    int* status = reinterpret_cast<int*>(ws + kWorkspaceHeader);
    uint8_t* gbuf = ws + kWorkspaceHeader + align_up(static_cast<size_t>(layers) * sizeof(int), 256);
    Plan p;
    const int st = make_plan(layers, G, N, D, &p);
    if (st != DTP_OK) return st;
    // the header status word starts at DTP_OK; every team writes its layer's word
    DTP_CUDA_TRY(cudaMemsetAsync(ws_status, 0, kWorkspaceHeader, stream));
    return launch_teams(p.global ? kernels_in_global(D).search : kernels_in_shared(D).search, false, layers, p, stream, A, G, N, iters, head, nu, score_q, score, iters_done, status,
                        ws_status, p.global ? gbuf : static_cast<uint8_t*>(nullptr), global_layer_bytes(N, D), p.vw);
}

// ---- whole model

static int launch_normalize(const float* S_up, const float* S_down, int Lyr, int G, int N, int D, int64_t* nbuf,
                            int32_t* head, int32_t* nu, ChainState* st, int* ws_status, int64_t* J_q, double* J,
                            int32_t* iters_done, int64_t* tops, cudaStream_t stream) {
    int dev = 0;
    DTP_CUDA_TRY(cudaGetDevice(&dev));
    Plan p = {};
    p.cl = resident_teams(dev, 4) > 0 ? 4 : 1;
    return launch_teams(chain_normalize_kernel, false, 2 * Lyr - 1, p, stream, S_up, S_down, Lyr, G, N, D, nbuf, head, nu,
                        st, ws_status, J_q, J, iters_done, tops);
}

struct ChainLayout {
    size_t state, score, prices, arrived, sums, tops, nbuf, gbuf, total;
};

static ChainLayout chain_layout(int Lyr, int G, int N, int D) {
    const size_t GN = static_cast<size_t>(G) * N;
    ChainLayout o;
    size_t x = kWorkspaceHeader;
    o.state = x;
    x += 256;
    o.prices = x;
    x += align_up(static_cast<size_t>(Lyr) * DMAX * sizeof(int64_t), 256);
    o.arrived = x;                                                          // cleared from the header up to here
    x += align_up(static_cast<size_t>(Lyr) * sizeof(int), 256);
    o.score = x;
    x += align_up(static_cast<size_t>(2 * Lyr) * sizeof(int64_t), 256);     // layer scores / edge scores
    o.sums = x;
    x += align_up(static_cast<size_t>(2 * Lyr) * GMAX * DMAX * sizeof(int64_t), 256);
    o.tops = x;
    x += align_up(static_cast<size_t>(2 * Lyr) * sizeof(int64_t), 256);
    o.nbuf = x;
    x += align_up(static_cast<size_t>(2 * Lyr - 1) * GN * sizeof(int64_t), 256);
    o.gbuf = x;
    if (!fits_block(N, D)) x += static_cast<size_t>(Lyr) * global_layer_bytes(N, D);
    o.total = x;
    return o;
}

size_t chain_workspace_bytes(int Lyr, int G, int N, int D) { return chain_layout(Lyr, G, N, D).total; }

int launch_chain(const float* S_up, const float* S_down, int Lyr, int G, int N, int D, int iters,
                 const uint8_t* move_heads, const uint8_t* move_neurons, int minimize, int32_t* head, int32_t* nu,
                 int64_t* J_q, double* J, int32_t* iters_done, void* workspace, cudaStream_t stream) {
    uint8_t* ws = reinterpret_cast<uint8_t*>(workspace);
    const ChainLayout o = chain_layout(Lyr, G, N, D);
    Plan p;
    int rc = make_plan(Lyr, 2 * G, N, D, &p);
    if (rc != DTP_OK) return rc;
    const Kernels k = p.global ? kernels_in_global(D) : kernels_in_shared(D);
    ChainArgs c;
    c.Lyr = Lyr;
    c.G = G;
    c.N = N;
    c.nbuf = reinterpret_cast<int64_t*>(ws + o.nbuf);
    c.top = reinterpret_cast<int64_t*>(ws + o.tops);
    c.head = head;
    c.nu = nu;
    c.prices = reinterpret_cast<int64_t*>(ws + o.prices);
    c.up_sums = reinterpret_cast<int64_t*>(ws + o.sums);
    c.down_sums = c.up_sums + static_cast<size_t>(Lyr) * GMAX * DMAX;
    c.arrived = reinterpret_cast<int*>(ws + o.arrived);
    c.layer_score = reinterpret_cast<int64_t*>(ws + o.score);
    c.st = reinterpret_cast<ChainState*>(ws + o.state);
    c.ws_status = reinterpret_cast<int*>(ws);
    c.gbuf = p.global ? ws + o.gbuf : nullptr;
    c.per_layer = global_layer_bytes(N, D);
    c.vw = p.vw;
    c.move_neurons = move_neurons;
    c.move_heads = move_heads;
    c.minimize = minimize;
    c.J_q = J_q;
    c.J = J;
    c.iters_done = iters_done;
    // header, state, prices and arrival counters
    DTP_CUDA_TRY(cudaMemsetAsync(ws, 0, o.score, stream));
    rc = launch_normalize(S_up, S_down, Lyr, G, N, D, reinterpret_cast<int64_t*>(ws + o.nbuf), head, nu, c.st,
                          c.ws_status, J_q, J, iters_done, reinterpret_cast<int64_t*>(ws + o.tops), stream);
    if (rc != DTP_OK) return rc;
    // all iterations in one launch while every layer's team has its SMs, else one launch each
    int dev = 0;
    DTP_CUDA_TRY(cudaGetDevice(&dev));
    if (iters > 1 && resident_teams(dev, p.cl) >= Lyr) {
        c.rounds = iters;
        rc = launch_teams(k.chain, true, Lyr, p, stream, c);
        if (rc != DTP_ERR_UNSUPPORTED) return rc;
    }
    c.rounds = 1;
    for (int it = 0; it < iters; ++it) {
        rc = launch_teams(k.chain, false, Lyr, p, stream, c);
        if (rc != DTP_OK) return rc;
    }
    return DTP_OK;
}

int launch_chain_score(const float* S_up, const float* S_down, int Lyr, int G, int N, int D, const int32_t* head,
                       const int32_t* nu, int64_t* edge_q, int64_t* J_q, double* J, void* workspace,
                       cudaStream_t stream) {
    uint8_t* ws = reinterpret_cast<uint8_t*>(workspace);
    const ChainLayout o = chain_layout(Lyr, G, N, D);
    int* ws_status = reinterpret_cast<int*>(ws);
    ChainState* st = reinterpret_cast<ChainState*>(ws + o.state);
    int64_t* edge = edge_q ? edge_q : reinterpret_cast<int64_t*>(ws + o.score);
    int64_t* nbuf = reinterpret_cast<int64_t*>(ws + o.nbuf);
    DTP_CUDA_TRY(cudaMemsetAsync(ws, 0, o.prices, stream));
    const int rc = launch_normalize(S_up, S_down, Lyr, G, N, D, nbuf, nullptr, nullptr, st, ws_status, J_q, J, nullptr,
                                    reinterpret_cast<int64_t*>(ws + o.tops), stream);
    if (rc != DTP_OK) return rc;
    chain_edge_kernel<<<2 * Lyr - 1, kThreads, kData, stream>>>(Lyr, G, N, D, nbuf, head, nu, edge, st, ws_status);
    chain_total_kernel<<<1, 32, 0, stream>>>(2 * Lyr - 1, edge, st, J_q, J);
    DTP_CUDA_TRY(cudaGetLastError());
    return DTP_OK;
}

// ---- exact optimum of one layer

// Teams of the item kernel: one per item up to this many blocks (the workspace holds a buffer per
// block when the layer may have to live in global memory).
constexpr int kGlobalMaxGrid = 160;

static size_t global_layout_bytes(int layers, int G, int N, int D, size_t* off_vals, size_t* off_gbuf) {
    size_t o = kWorkspaceHeader;
    *off_vals = o;
    o += align_up(static_cast<size_t>(layers) * unlabelled_count(G, D) * sizeof(int64_t), 256);
    *off_gbuf = o;
    if (!fits_block(N, D))
        o += static_cast<size_t>(kGlobalMaxGrid > layers ? kGlobalMaxGrid : layers) * global_layer_bytes(N, D);
    return o;
}

size_t global_workspace_bytes(int layers, int G, int N, int D) {
    size_t a, b;
    return global_layout_bytes(layers, G, N, D, &a, &b);
}

int launch_global(const float* A, int layers, int G, int N, int D, int32_t* head, int32_t* nu, int64_t* score_q,
                  double* score, void* workspace, cudaStream_t stream) {
    uint8_t* ws = reinterpret_cast<uint8_t*>(workspace);
    int dev = 0, sms = 0;
    DTP_CUDA_TRY(cudaGetDevice(&dev));
    DTP_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    if (sms > kGlobalMaxGrid) sms = kGlobalMaxGrid;
    size_t o_vals, o_gbuf;
    global_layout_bytes(layers, G, N, D, &o_vals, &o_gbuf);
    int* ws_status = reinterpret_cast<int*>(ws);
    int64_t* vals = reinterpret_cast<int64_t*>(ws + o_vals);
    const int64_t n_unl = unlabelled_count(G, D);
    const int64_t items = static_cast<int64_t>(layers) * n_unl;
    Plan pi, pp;
    int rc = make_plan(items, G, N, D, &pi);
    if (rc == DTP_OK) rc = make_plan(layers, G, N, D, &pp);
    if (rc != DTP_OK) return rc;
    int64_t teams = sms / pi.cl > 0 ? sms / pi.cl : 1;
    if (items < teams) teams = items;
    DTP_CUDA_TRY(cudaMemsetAsync(ws_status, 0, kWorkspaceHeader, stream));
    rc = launch_teams(pi.global ? kernels_in_global(D).items : kernels_in_shared(D).items, false, teams, pi, stream, A, layers, G, N, n_unl, vals, ws_status,
                      pi.global ? ws + o_gbuf : static_cast<uint8_t*>(nullptr), global_layer_bytes(N, D), pi.vw);
    if (rc != DTP_OK) return rc;
    return launch_teams(pp.global ? kernels_in_global(D).pick : kernels_in_shared(D).pick, false, layers, pp, stream, A, G, N, n_unl, vals, head, nu, score_q, score,
                        ws_status, pp.global ? ws + o_gbuf : static_cast<uint8_t*>(nullptr),
                        global_layer_bytes(N, D), pp.vw);
}

}  // namespace search
}  // namespace dtp
