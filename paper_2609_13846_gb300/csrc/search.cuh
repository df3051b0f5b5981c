// search.cuh -- the layout optimiser of Sec. 3 ("Objective", "Optimiser") on
// the GPU: coordinate ascent over balanced head partitions h and balanced
// neuron assignments nu of one layer, maximising the co-located up-edge mass.
//
// One team per layer: a thread block cluster of 1 to 16 blocks of 512 threads,
// each holding a slice of the layer's neurons in shared memory (in global
// memory when even 16 slices do not fit).  Each block
// reduces its slice, one cluster barrier later every block reads its peers'
// partial results over distributed shared memory and continues with the same
// totals, so the serial parts are repeated by every block instead of broadcast.
// The layers of a batch are independent because the up-edge objective decouples
// across layers.
//
// Exactness.  A is mapped to q[g,k] = floor(A[g,k] * 2^(40-e)) (max A < 2^e),
// computed from the fp32 bit pattern with integer shifts, and every score is
// an int64 sum, so no summation order can change a decision.
//
// Neuron step (exact balanced linear assignment, lexicographically smallest
// optimum), gain M[k,l] = sum over heads g with h(g) == l of q[g,k]:
//   D == 2  device 0 takes the N/2 largest M[k,0]-M[k,1], lower index first on
//           ties: a histogram selection of the threshold.
//   D >  2  (a) device prices from Gauss-Seidel sweeps on the gains' upper 29
//           bits, each price set by a histogram selection so that about N/D
//           neurons prefer its device (approximate: only speed depends on it);
//           (b) every neuron to its best device at those prices -- optimal for
//           the resulting device counts by complementary slackness;
//           (c) the excess is moved along maximum-gain paths of the exchange
//           graph restricted to the candidates, the neurons whose gap to another
//           device is below a bound; outside them the bound itself limits every
//           exchange, so a closed all-pairs computation certifies that the result
//           is optimal and that no other optimum precedes it lexicographically;
//           (d) without that certificate (ties, mostly), the same steps over all
//           neurons: one unit of excess per maximum-gain path, then for k = 0, 1,
//           ... move k to the smallest device l < nu(k) that a zero-gain exchange
//           cycle through neurons > k allows.
// Head step: B[g,l] = sum over neurons on l of q[g,k]; the best labelled balanced
// partition, lexicographically smallest on ties, by dynamic programming over the
// devices' remaining capacities.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "dtp_common.cuh"

namespace dtp {
namespace search {

constexpr int kThreads = 512;   // 128 registers a thread: at 1024 the steps spilled, and beside 180 KB of shared
                                 // memory the L1 cache is too small to hold spills
constexpr int kWarps = kThreads / 32;
constexpr int DMAX = 8;
constexpr int GMAX = 16;
constexpr int kFixedBits = 40;
constexpr int kIdxBits = 18;                       // N <= 2^18
constexpr int64_t kValBias = int64_t(1) << 45;     // |gain| < 2^44 (H_kv <= 16): fits the 46-bit field
constexpr int64_t kNegInf = INT64_MIN / 4;
constexpr int kMaxPasses = 24;                      // price passes before the exact repair
constexpr int kLoBits = 15;                         // a score row is stored as a value's upper bits and lower 15
constexpr int kHiBits = 29;                         // a gain as its upper 29 bits (of the layer's largest) and the rest
constexpr int32_t kPriceMax = 1 << 30;              // |price| in units of 2^sh (Layer::sh)
constexpr int kBins = 1024;                         // histogram bins (32 groups of 32)
constexpr int kCounters = 64;                       // counters merged together with a histogram
constexpr int kPairs = DMAX;                        // first counter of device pairs (28 of them)
constexpr int kCand = 256;                          // candidates of the restricted exchange graph
constexpr int kCandTarget = 240;                    // candidates asked for (the rest is rounding slack)
constexpr int64_t kBoundMax = int64_t(1) << 50;     // above any difference of reduced gains
constexpr int kStates = 1024;                       // head-step states (G/D + 1)^D of every accepted size
constexpr int kMaxCluster = 16;
constexpr int kSums = 2 * GMAX * DMAX + 8;           // int64 sums of one exchange
// A block's slice of the gains, nu and (if they fit) the scores; struct Shared before it takes up to
// 43 KB of the 227 KB.
constexpr size_t kSmemBudget = 184 * 1024;
// Layers of up to this many bytes of int64 gains and int32 labels need no global buffer even
// without clusters (the workspace's size rule; the kernels' own layout is smaller).
constexpr size_t kWorkspaceFree = 220 * 1024;
// One block holds every such layer: its np <= N + 15 neurons of 6 D + 1 bytes (slice_bytes) take less than
// 3/4 of N's 8 D + 4 and 15 neurons more.  So a layer that lives in the workspace has room there.
static_assert(kWorkspaceFree / 4 * 3 + 15 * (6 * DMAX + 1) <= kSmemBudget, "layers without a workspace fit one block");

struct Shared {
    uint32_t hist[2][kBins + kCounters];   // this block's counts, two phases
    uint32_t wsum[2][32];                  // this block's sums of 32 bins each, two phases
    uint32_t pick[4];                      // a merged histogram's bin, elements above it, in it; found
    uint32_t counters[kCounters];          // the team's counters
    uint32_t wmm[2][2][kWarps];            // per-warp minima and maxima, two phases
    uint32_t mm[2][2];                     // this block's, two phases
    uint32_t mmt[2];                       // the team's
    int64_t xl[2][kSums];                  // this block's int64 sums, two phases
    int64_t B[kSums];                      // the team's sums: head-step columns, then a total
    int64_t part[kWarps][DMAX];
    union {
        int64_t cv[DMAX][kCand];           // candidates: gains less prices
        int64_t f[kStates];                // head step: best completion of a state
    };
    int32_t ck[kCand];                     // candidate neuron
    uint8_t cnu[kCand];                    // its device
    uint8_t clist[DMAX][kCand];            // the slots on each device
    int clen[DMAX];
    int ncand;
    uint64_t E[DMAX][DMAX];                // candidate exchange graph: packed (gain, slot), 0 = none
    uint64_t wl[2][DMAX * DMAX];           // exchange graph over all neurons of the slice, two phases
    uint64_t w[DMAX][DMAX];                // the team's (0 = no neuron on the source device)
    uint64_t wk[DMAX][DMAX];               // and over the neurons above an index
    int64_t P[DMAX][DMAX];                 // all-pairs max-gain paths
    int64_t bound[DMAX][DMAX];             // a neuron on a with gap <= bound[a][b] for some b is a candidate
    int64_t pi[DMAX];                      // device prices
    float scale[DMAX];                     // a device's mean gain in units of 2^sh (relative size only)
    int32_t price[DMAX];                   // prices in units of 2^sh, handed from one warp or block to the others
    int32_t best_price[DMAX];              // the prices of the smallest excess so far
    int32_t price_step[DMAX];              // the size of a price's last change by a sweep (negative: none yet)
    int count[DMAX];
    int64_t J, Jprev;
    int h[GMAX];
    int hn[GMAX];                          // next layer's head partition (whole-model search)
    int glist[GMAX], gnlist[GMAX];         // heads listed device by device, for h and for hn
    int status;
    int flag;
    unsigned dirty;                        // devices whose edges of E or w are to be found again
    int best_idx;
    int64_t red_i64[kWarps];
    int red_int[kWarps];
    int* beat;                             // where long repairs show that they go on, or null
};

// The block's dynamic shared memory starts with Shared; the layer's data follow at kData.  Named this
// way (and not through pointers) the compiler emits shared-memory instructions everywhere.
extern __shared__ __align__(16) uint8_t dsm[];
constexpr int kData = (static_cast<int>(sizeof(Shared)) + 127) / 128 * 128;
static_assert(kData + kSmemBudget <= 227 * 1024, "shared memory");
__device__ __forceinline__ Shared& shared() { return *reinterpret_cast<Shared*>(dsm); }

// ------------------------------------------------------------------- teams --

// The blocks that share one layer.  The phases select double-buffered exchange areas: a block
// rewrites an area only after a barrier that follows the barrier after which its peers read it.
struct Team {
    uint32_t cl, rank;
    uint32_t ph, mph, lph, wph;
};

__device__ __forceinline__ uint32_t cluster_nctarank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ Team make_team() {
    Team t;
    t.cl = cluster_nctarank();
    t.rank = cluster_ctarank();
    t.ph = t.mph = t.lph = t.wph = 0;
    return t;
}

__device__ __forceinline__ void team_sync(const Team& t) {
    if (t.cl == 1) __syncthreads();
    else cluster_sync();
}

// The same shared variable in block r of the team, as a generic pointer.
template <class T>
__device__ __forceinline__ T* at_rank(T* p, uint32_t r) {
    uint64_t a;
    asm volatile("mapa.u64 %0, %1, %2;" : "=l"(a) : "l"(reinterpret_cast<uint64_t>(p)), "r"(r));
    return reinterpret_cast<T*>(a);
}

__device__ __forceinline__ uint32_t load_peer(const uint32_t* p, uint32_t r) {
    uint32_t v;
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(mapa_shared(smem_u32(p), r)));
    return v;
}
__device__ __forceinline__ int64_t load_peer(const int64_t* p, uint32_t r) {
    int64_t v;
    asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(v) : "r"(mapa_shared(smem_u32(p), r)));
    return v;
}
__device__ __forceinline__ uint64_t load_peer(const uint64_t* p, uint32_t r) {
    return static_cast<uint64_t>(load_peer(reinterpret_cast<const int64_t*>(p), r));
}

// op over *p of every block of the team (p: this block's variable).  The peers' loads are issued
// together: one after another, the seven of an 8-block team cost 5,000 cycles per exchange.
template <class T, class Op>
__device__ __forceinline__ T team_combine(const T* p, const Team& t, Op op) {
    T own = *p;
    for (uint32_t base = 1; base < t.cl; base += 8) {
        T v[8];
#pragma unroll
        for (uint32_t i = 0; i < 8; ++i)
            if (base + i < t.cl) v[i] = load_peer(p, (t.rank + base + i) & (t.cl - 1));
#pragma unroll
        for (uint32_t i = 0; i < 8; ++i)
            if (base + i < t.cl) own = op(own, v[i]);
    }
    return own;
}

// ---------------------------------------------------------------- helpers --

__device__ __forceinline__ size_t align_up_dev(size_t x, size_t a) { return (x + a - 1) / a * a; }

// f(i, a[i]) for every i < n, the block's threads taking consecutive elements: 16-byte loads of
// four elements when a is 16-byte aligned (the tail, and unaligned arrays, element by element).
// Every caller's result is independent of the visiting order (a max, an exact integer sum, or an
// element-wise copy).
template <class F>
__device__ __forceinline__ void for_each_a(const float* __restrict__ a, int64_t n, F&& f) {
    int64_t head = 0;
    if ((reinterpret_cast<uintptr_t>(a) & 15u) == 0) {
        const int64_t n4 = n >> 2;
        const float4* a4 = reinterpret_cast<const float4*>(a);
        for (int64_t i = threadIdx.x; i < n4; i += kThreads) {
            const float4 v = a4[i];
            f(4 * i, v.x);
            f(4 * i + 1, v.y);
            f(4 * i + 2, v.z);
            f(4 * i + 3, v.w);
        }
        head = n4 << 2;
    }
    for (int64_t i = head + threadIdx.x; i < n; i += kThreads) f(i, a[i]);
}

// floor(a * 2^(bits-e)) for a finite a >= 0, by shifting the fp32 significand.
__device__ __forceinline__ int64_t quantize_bits(float a, int e, int bits) {
    const uint32_t b = __float_as_uint(a);
    const uint32_t ex = (b >> 23) & 0xFFu;
    uint64_t m = b & 0x7FFFFFu;
    int E;
    if (ex == 0) {
        E = -149;
    } else {
        m |= 0x800000u;
        E = static_cast<int>(ex) - 150;
    }
    const int s = E + bits - e;
    if (s >= 0) return static_cast<int64_t>(m << s);
    if (s <= -40) return 0;
    return static_cast<int64_t>(m >> (-s));
}

// floor(a * 2^(40-e)) < 2^40 as its upper 25 bits and its lower kLoBits bits, in 32-bit arithmetic
// (PTX shifts by 32 or more give zero).
__device__ __forceinline__ uint32_t shl32(uint32_t x, uint32_t n) {
    uint32_t r;
    asm("shl.b32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(n));
    return r;
}
__device__ __forceinline__ uint32_t shr32(uint32_t x, uint32_t n) {
    uint32_t r;
    asm("shr.u32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(n));
    return r;
}
__device__ __forceinline__ void quantize_split(float a, int e, uint32_t& hi, uint32_t& lo) {
    const uint32_t b = __float_as_uint(a);
    const int ex = static_cast<int>((b >> 23) & 0xFFu);
    const uint32_t m = (b & 0x7FFFFFu) | (ex ? 0x800000u : 0u);
    const int s = (ex ? ex : 1) - 150 + kFixedBits - e;            // q = m * 2^s, s <= 16
    hi = shr32(shl32(m, static_cast<uint32_t>(max(s - kLoBits, 0))), static_cast<uint32_t>(max(kLoBits - s, 0)));
    lo = shr32(shl32(m, static_cast<uint32_t>(max(s, 0))), static_cast<uint32_t>(max(-s, 0))) & ((1u << kLoBits) - 1u);
}

// The bit pattern of |a| for a finite a >= 0 (ordered as the values), all ones for any other a.
__device__ __forceinline__ uint32_t valid_bits(float a) {
    const uint32_t b = __float_as_uint(a);
    const uint32_t m = b & 0x7FFFFFFFu;
    return (m >= 0x7F800000u || b > 0x80000000u) ? 0xFFFFFFFFu : m;
}

__device__ __forceinline__ uint64_t pack_gain(int64_t v, int k) {
    return (static_cast<uint64_t>(v + kValBias) << kIdxBits) |
           static_cast<uint64_t>((1 << kIdxBits) - 1 - k);
}
__device__ __forceinline__ int64_t gain_of(uint64_t key) {
    return static_cast<int64_t>(key >> kIdxBits) - kValBias;
}
__device__ __forceinline__ int index_of(uint64_t key) {
    return (1 << kIdxBits) - 1 - static_cast<int>(key & ((1u << kIdxBits) - 1));
}

// Candidate edges: reduced gains (|gain| < 2^47) and slots of the candidate list.
constexpr int64_t kCandBias = int64_t(1) << 47;
__device__ __forceinline__ uint64_t pack_cand(int64_t v, int slot) {
    return (static_cast<uint64_t>(v + kCandBias) << 8) | static_cast<uint64_t>(kCand - 1 - slot);
}
__device__ __forceinline__ int64_t cand_gain(uint64_t key) { return static_cast<int64_t>(key >> 8) - kCandBias; }
__device__ __forceinline__ int cand_slot(uint64_t key) { return kCand - 1 - static_cast<int>(key & 255u); }

__device__ __forceinline__ uint64_t warp_max_u64(uint64_t x) {
    const uint32_t hi = static_cast<uint32_t>(x >> 32);
    const uint32_t mhi = __reduce_max_sync(0xFFFFFFFFu, hi);
    const uint32_t lo = (hi == mhi) ? static_cast<uint32_t>(x) : 0u;
    const uint32_t mlo = __reduce_max_sync(0xFFFFFFFFu, lo);
    return (static_cast<uint64_t>(mhi) << 32) | mlo;
}

__device__ __forceinline__ int64_t warp_sum_i64(int64_t x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xFFFFFFFFu, x, o);
    return x;
}

static __device__ __noinline__ int64_t block_sum_i64(int64_t x) {
    Shared& sh = shared();
    x = warp_sum_i64(x);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __syncthreads();
    if (lane == 0) sh.red_i64[warp] = x;
    __syncthreads();
    int64_t t = 0;
    for (int i = 0; i < kWarps; ++i) t += sh.red_i64[i];
    return t;
}

// The smallest and the largest of the team's per-thread values (lo and hi), in every thread.
__device__ __forceinline__ void team_min_max(uint32_t& lo, uint32_t& hi, Team& tm) {
    Shared& sh = shared();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    lo = __reduce_min_sync(0xFFFFFFFFu, lo);
    hi = __reduce_max_sync(0xFFFFFFFFu, hi);
    if (lane == 0) sh.wmm[tm.mph][0][warp] = lo, sh.wmm[tm.mph][1][warp] = hi;
    __syncthreads();
    if (tm.cl == 1 || warp == 0) {
        lo = __reduce_min_sync(0xFFFFFFFFu, sh.wmm[tm.mph][0][lane % kWarps]);
        hi = __reduce_max_sync(0xFFFFFFFFu, sh.wmm[tm.mph][1][lane % kWarps]);
    }
    if (tm.cl > 1) {
        if (threadIdx.x == 0) sh.mm[tm.mph][0] = lo, sh.mm[tm.mph][1] = hi;
        team_sync(tm);
        if (warp == 0) {                       // lane r reads block r's
            const uint32_t r = lane < tm.cl ? lane : tm.rank;
            lo = __reduce_min_sync(0xFFFFFFFFu, load_peer(&sh.mm[tm.mph][0], r));
            hi = __reduce_max_sync(0xFFFFFFFFu, load_peer(&sh.mm[tm.mph][1], r));
            if (lane == 0) sh.mmt[0] = lo, sh.mmt[1] = hi;
        }
        __syncthreads();
        lo = sh.mmt[0];
        hi = sh.mmt[1];
    }
    tm.mph ^= 1;
}

// sh.B[i] = the team's sum of sh.xl[phase][i], i < cnt <= kSums.
static __device__ __noinline__ void team_sum_i64(int cnt, Team& tm) {
    Shared& sh = shared();
    team_sync(tm);
    if (threadIdx.x < cnt)
        sh.B[threadIdx.x] = team_combine(&sh.xl[tm.lph][threadIdx.x], tm, [](int64_t a, int64_t b) { return a + b; });
    __syncthreads();
    tm.lph ^= 1;
}

__device__ __forceinline__ uint32_t warp_scan(uint32_t x) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
        if (lane >= o) x += y;
    }
    return x;
}

struct Pick {
    uint32_t bin, above, inside;
    bool found;
};

// A warp finds the bin that holds the rank-th element counted from the top bin down: `group` gives
// the sum of the 32 bins of group g, `single` a bin's count.
template <class GroupFn, class BinFn>
__device__ __forceinline__ Pick warp_pick(uint32_t rank, GroupFn group, BinFn single) {
    const int lane = threadIdx.x & 31;
    Pick p;
    const uint32_t w = group(31 - lane);
    const uint32_t wi = warp_scan(w);
    const unsigned who = __ballot_sync(0xFFFFFFFFu, wi >= rank);
    p.found = who != 0;
    p.bin = p.above = p.inside = 0;
    if (!p.found) return p;
    const int src = __ffs(who) - 1;
    const uint32_t above = __shfl_sync(0xFFFFFFFFu, wi - w, src);
    const uint32_t b = single((31 - src) * 32 + 31 - lane);
    const uint32_t bi = warp_scan(b);
    const int l2 = __ffs(__ballot_sync(0xFFFFFFFFu, bi >= rank - above)) - 1;
    p.bin = static_cast<uint32_t>((31 - src) * 32 + 31 - l2);
    p.above = above + __shfl_sync(0xFFFFFFFFu, bi - b, l2);
    p.inside = __shfl_sync(0xFFFFFFFFu, b, l2);
    return p;
}

// After every thread's increments of sh.hist[phase]: the bin of the team's summed histogram that
// holds the rank-th element counted from the top bin down, the number of elements above that bin
// and in it (found == false: fewer than rank elements); the team's counters into sh.counters.  One
// warp reads the peers' 32 group sums and then the 32 bins it needs: reading all 1024 bins of seven
// peers by every block took 8,000 cycles.  The other phase, which every block has read before this
// barrier, is cleared.
__device__ __forceinline__ Pick team_pick(uint32_t rank, Team& tm) {
    Shared& sh = shared();
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    auto add = [](uint32_t a, uint32_t b) { return a + b; };
    const uint32_t* h = sh.hist[tm.ph];
    const uint32_t* ws = sh.wsum[tm.ph];
    __syncthreads();
#pragma unroll
    for (int g = 0; g < 32; g += kWarps) {
        const uint32_t s = __reduce_add_sync(0xFFFFFFFFu, h[g * 32 + t]);
        if (lane == 0) sh.wsum[tm.ph][g + warp] = s;
    }
    team_sync(tm);
    if (warp == 0) {
        const Pick p = warp_pick(rank, [&](int g) { return team_combine(ws + g, tm, add); },
                                 [&](int b) { return team_combine(h + b, tm, add); });
        if (lane == 0) sh.pick[0] = p.bin, sh.pick[1] = p.above, sh.pick[2] = p.inside, sh.pick[3] = p.found;
    } else if (t >= 32 && t < 32 + kCounters) {
        sh.counters[t - 32] = team_combine(h + kBins + t - 32, tm, add);
    }
    for (int i = t; i < kBins + kCounters; i += kThreads) sh.hist[tm.ph ^ 1][i] = 0;
    __syncthreads();
    Pick p;
    p.bin = sh.pick[0];
    p.above = sh.pick[1];
    p.inside = sh.pick[2];
    p.found = sh.pick[3] != 0;
    tm.ph ^= 1;
    return p;
}

// The counters alone (the histogram bins of this phase are all zero).
__device__ __forceinline__ void team_counters(Team& tm) {
    Shared& sh = shared();
    const int t = threadIdx.x;
    team_sync(tm);
    const uint32_t* h = sh.hist[tm.ph];
    if (t < kCounters) sh.counters[t] = team_combine(h + kBins + t, tm, [](uint32_t a, uint32_t b) { return a + b; });
    for (int i = t; i < kBins + kCounters; i += kThreads) sh.hist[tm.ph ^ 1][i] = 0;
    __syncthreads();
    tm.ph ^= 1;
}

__device__ __forceinline__ int bin_shift(uint32_t range) {
    const int s = 22 - __clz(range);          // range >> s < 1024
    return s > 0 ? s : 0;
}

// f(k) for the block's threads' neurons k < n, two at a time so that their loads overlap.
template <class F>
__device__ __forceinline__ void for_neurons(int n, F&& f) {
    int k = threadIdx.x;
    for (; k + kThreads < n; k += 2 * kThreads) {
#pragma unroll
        for (int u = 0; u < 2; ++u) f(k + u * kThreads);
    }
    if (k < n) f(k);
}

// A threshold on the keys key(k), k < n, of the team's neurons in [lo, lo + range] (others, and
// those for which key returns false, do not count): the smallest t found with at most rank + tol
// keys >= t and at least rank, by histograms of 1024 equal bins, each refining the bin that holds
// the rank-th largest.  ge: the number of keys >= t.  False: fewer than rank keys.
template <class KeyFn>
__device__ bool select_threshold(int n, uint32_t lo, uint32_t range, uint32_t rank, uint32_t tol, KeyFn key,
                                 uint32_t& t, uint32_t& ge, Team& tm) {
    Shared& sh = shared();
    ge = 0;
    for (;;) {
        const int s = bin_shift(range);
        uint32_t* hist = sh.hist[tm.ph];
        for_neurons(n, [&](int k) {
            uint32_t x;
            if (key(k, x) && x - lo <= range) atomicAdd(&hist[(x - lo) >> s], 1u);
        });
        const Pick p = team_pick(rank, tm);
        if (!p.found) return false;
        lo += p.bin << s;
        ge += p.above;
        rank -= p.above;
        if (s == 0 || p.inside <= rank + tol) {
            ge += p.inside;
            t = lo;
            return true;
        }
        range = (1u << s) - 1u;
    }
}

// A block's part of a layer.  Scores come as exact integers in two parts, value = hi << 15 | lo: per
// head in qh, ql (rows [rows][rnp] of the block's slice of neurons, staged once in shared memory when
// they fit, else null and recomputed from global memory), per device (the gains M) in hi, lo with gain = hi << sh | lo.
// Two ways of keeping the gains: `gathered`, block 0 holds those of all neurons and takes the neuron
// step alone (the others build gains for it and sum columns), or each block holds its slice's and all
// take the step together.
struct Layer {
    const float* A;     // [G][N] from the slice's first neuron (single-layer search)
    const int64_t* nU;  // [G][N] from the slice's first neuron (whole-model search)
    const int64_t* nD;  // the same for the down edge, or null
    int G, N, D, cap, e;
    int sh;             // a gain's low bits (0 .. 15): the upper part has kHiBits at the layer's largest gain
    int n, k0;          // neurons of this block's slice (in a step: of the gains) and the first one's index
    int np;             // column stride of hi and lo
    int rnp;            // row stride of qh and ql
    int32_t* hi;        // [D][np] gains >> sh
    uint16_t* lo;       // [D][np] gains' low sh bits
    uint8_t* nu;        // [np]
    uint16_t* lists;    // neurons of the slice by device [D][rnp]: over the block's own gains
    uint32_t* qh;
    uint16_t* ql;
    int q_off, q_rows;  // with qh: its offset in the dynamic shared memory and its rows
};

// With SM (every layer that fits) the gains start at kData and the staged rows lie at L.q_off; without
// SM the pointers of Layer are used.
template <bool SM>
__device__ __forceinline__ int32_t* hi_of(const Layer& L) {
    if constexpr (SM) return reinterpret_cast<int32_t*>(dsm + kData);
    else return L.hi;
}
template <bool SM>
__device__ __forceinline__ uint16_t* lo_of(const Layer& L) {
    if constexpr (SM) return reinterpret_cast<uint16_t*>(dsm + kData + L.np * L.D * 4);
    else return L.lo;
}
template <bool SM>
__device__ __forceinline__ uint8_t* nu_of(const Layer& L) {
    if constexpr (SM) return dsm + kData + L.np * L.D * 6;
    else return L.nu;
}

// Row r (a head; G + head: the down edge) of local neuron k.
template <bool SM>
__device__ __forceinline__ void score_parts(const Layer& L, int r, int k, uint32_t& hi, uint32_t& lo) {
    if (L.qh) {
        if constexpr (SM) {
            hi = reinterpret_cast<const uint32_t*>(dsm + L.q_off)[r * L.rnp + k];
            lo = reinterpret_cast<const uint16_t*>(dsm + L.q_off + L.q_rows * L.rnp * 4)[r * L.rnp + k];
        } else {
            hi = L.qh[r * L.rnp + k];
            lo = L.ql[r * L.rnp + k];
        }
    } else if (L.A) {
        quantize_split(L.A[static_cast<int64_t>(r) * L.N + k], L.e, hi, lo);
    } else {
        const int64_t v = r < L.G ? L.nU[static_cast<int64_t>(r) * L.N + k]
                                  : L.nD[static_cast<int64_t>(r - L.G) * L.N + k];
        hi = static_cast<uint32_t>(v >> kLoBits);
        lo = static_cast<uint32_t>(v) & ((1u << kLoBits) - 1u);
    }
}

template <bool SM>
__device__ __forceinline__ int64_t gain_at(const Layer& L, int l, int k) {
    const int i = l * L.np + k;
    return (static_cast<int64_t>(hi_of<SM>(L)[i]) << L.sh) | lo_of<SM>(L)[i];
}

__device__ __forceinline__ void set_gain(const Layer& L, int l, int k, int64_t m) {
    const int i = l * L.np + k;
    L.hi[i] = static_cast<int32_t>(m >> L.sh);
    L.lo[i] = static_cast<uint16_t>(m & ((1 << L.sh) - 1));
}

// Bytes of a slice of np neurons (np a multiple of 16): hi, lo, nu.
__host__ __device__ inline size_t slice_bytes(int np, int D) {
    return static_cast<size_t>(np) * (static_cast<size_t>(D) * 6 + 1);
}

// sh.glist / sh.gnlist: heads in device order, each device's in increasing index.  Warp 0.
__device__ __forceinline__ void list_heads(const int* h, int* list, int G, int cap) {
    const int lane = threadIdx.x & 31;
    const int l = lane < G ? h[lane] : -1;
    const unsigned same = __match_any_sync(0xFFFFFFFFu, l);
    if (lane < G) list[l * cap + __popc(same & ((1u << lane) - 1u))] = lane;
}

// M of the slice from the scores: M[k,l] = sum over the heads that sh.glist puts on device l, plus,
// with a down edge, those that sh.gnlist does; minimising: sum_l' M[k,l'] - M[k,l].
template <int DT, bool SM>
__device__ __noinline__ void build_gain(const Layer& layer, bool down, bool minimize) {
    Shared& sh = shared();
    const Layer L = layer;
    const int per = L.G / DT;
    for (int k = threadIdx.x; k < L.n; k += kThreads) {
        int gi = 0;
        if (!minimize) {
#pragma unroll
            for (int l = 0; l < DT; ++l) {
                uint32_t hs = 0, ls = 0, h, lo;
                for (int j = 0; j < per; ++j, ++gi) {
                    score_parts<SM>(L, sh.glist[gi], k, h, lo);
                    hs += h, ls += lo;
                    if (down) {
                        score_parts<SM>(L, L.G + sh.gnlist[gi], k, h, lo);
                        hs += h, ls += lo;
                    }
                }
                set_gain(L, l, k, (static_cast<int64_t>(hs) << kLoBits) + ls);
            }
        } else {
            int64_t m[DT], r = 0;
#pragma unroll
            for (int l = 0; l < DT; ++l) {
                m[l] = 0;
                uint32_t h, lo;
                for (int j = 0; j < per; ++j, ++gi) {
                    score_parts<SM>(L, sh.glist[gi], k, h, lo);
                    m[l] += (static_cast<int64_t>(h) << kLoBits) + lo;
                    if (down) {
                        score_parts<SM>(L, L.G + sh.gnlist[gi], k, h, lo);
                        m[l] += (static_cast<int64_t>(h) << kLoBits) + lo;
                    }
                }
                r += m[l];
            }
#pragma unroll
            for (int l = 0; l < DT; ++l) set_gain(L, l, k, r - m[l]);
        }
    }
    __syncthreads();
}

// ------------------------------------------------------------ neuron steps --

template <bool SM>
__device__ __noinline__ void neuron_step_d2(const Layer& layer, Team& tm) {
    Shared& sh = shared();
    const Layer L = layer;
    // order: larger M0 - M1 first, then the lower index, as a 32-bit key of the difference's upper
    // bits and a 32-bit key of its low bits and the index (unique); the second is only looked at
    // when the threshold falls between neurons that share the first
    auto diff = [&](int k) -> int64_t { return gain_at<SM>(L, 0, k) - gain_at<SM>(L, 1, k); };
    const int cut = L.sh > 1 ? L.sh - 1 : 0;       // |d| < 2^(29 + sh): the upper key has 30 bits and a sign
    auto upper = [cut](int64_t d) -> uint32_t { return static_cast<uint32_t>(static_cast<int32_t>(d >> cut)) ^ 0x80000000u; };
    auto lower = [&](int64_t d, int k) -> uint32_t {
        return (static_cast<uint32_t>(d & ((1 << cut) - 1)) << kIdxBits) |
               static_cast<uint32_t>((1 << kIdxBits) - 1 - (L.k0 + k));
    };
    const uint32_t rank = static_cast<uint32_t>(L.cap);
    uint32_t lo = 0xFFFFFFFFu, hi = 0u;
    for_neurons(L.n, [&](int k) {
        const uint32_t u = upper(diff(k));
        lo = min(lo, u);
        hi = max(hi, u);
    });
    team_min_max(lo, hi, tm);
    uint32_t t, ge, t2 = 0, ge2;
    bool ok = select_threshold(L.n, lo, hi - lo, rank, 0, [&](int k, uint32_t& x) { x = upper(diff(k)); return true; }, t,
                               ge, tm);
    if (ok && ge > rank) {
        // more neurons share the upper key t than the device takes: (ge - inside) lie above it
        uint32_t eq = 0;
        for (int k = threadIdx.x; k < L.n; k += kThreads) eq += upper(diff(k)) == t;
        eq = __reduce_add_sync(0xFFFFFFFFu, eq);
        if ((threadIdx.x & 31) == 0) atomicAdd(&sh.hist[tm.ph][kBins], eq);
        team_counters(tm);
        const uint32_t inside = sh.counters[0];
        ok = select_threshold(L.n, 0u, 0xFFFFFFFFu, rank - (ge - inside), 0,
                              [&](int k, uint32_t& x) {
                                  const int64_t d = diff(k);
                                  x = lower(d, k);
                                  return upper(d) == t;
                              },
                              t2, ge2, tm);
    }
    if (!ok && threadIdx.x == 0) sh.status = DTP_ERR_NOT_CONVERGED;   // rank out of range
    for (int k = threadIdx.x; k < L.n; k += kThreads) {
        const int64_t d = diff(k);
        const uint32_t u = upper(d);
        nu_of<SM>(L)[k] = (u > t || (u == t && lower(d, k) >= t2)) ? 0 : 1;
    }
    __syncthreads();
}

// Warp 0: max-gain paths over the devices by Bellman-Ford, lane b holding device b and the gains
// w[a] of its incoming edges (kNegInf: none).  src: mask of start devices (distance 0).
template <int DT>
__device__ __forceinline__ void bellman_ford_warp(unsigned src, const int64_t (&w)[DT], int64_t& dist, int& pred) {
    const int b = threadIdx.x & 31;
    dist = (src >> b) & 1u ? 0 : kNegInf;
    pred = -1;
    for (int round = 0; round < DT - 1; ++round) {
        const int64_t before = dist;
        bool moved = false;
#pragma unroll
        for (int a = 0; a < DT; ++a) {
            const int64_t x = __shfl_sync(0xFFFFFFFFu, before, a) + w[a];   // no edge or no path: far below any gain
            if (x > dist && x > kNegInf / 2) dist = x, pred = a, moved = true;
        }
        if (!__any_sync(0xFFFFFFFFu, moved)) break;
    }
}

// Max-plus closure of sh.P over the D devices, by warp 0.
__device__ __forceinline__ void close_paths(int D) {
    Shared& sh = shared();
    const int lane = threadIdx.x & 31;
    for (int c = 0; c < D; ++c) {
        for (int i = lane; i < D * D; i += 32) {
            const int a = i / D, b = i % D;
            const int64_t x = sh.P[a][c], y = sh.P[c][b];
            if (x != kNegInf && y != kNegInf && x + y > sh.P[a][b]) sh.P[a][b] = x + y;
        }
        __syncwarp();
    }
}

// Steps (b) and (c): the assignment at the prices p (units of 2^sh) and its repair over the
// candidates.  True: L.nu holds the optimal assignment and sh.pi its prices; `unique` then says
// whether it is certified to be the lexicographically smallest optimum (because every exchange that
// would put a smaller device earlier loses).  False: L.nu holds the assignment at the prices.
//
// Candidates are the neurons whose gap to some device b (their gain less price on their own device
// a, less that on b) is at most bound[a][b] = tau * max(scale[a], scale[b]): tau (negative: every
// neuron) comes from a histogram of the gaps so that about 240 neurons qualify (on model-shaped layers
// the prices leave an excess of at most 3 D, and 240 candidates held every certificate).  A neuron
// outside the list has a gap of at least bound + 1 to every device, so max(best candidate edge,
// -bound - 1) is an upper bound of every edge of the exchange graph, whatever the scales are.  If the
// closure of those bounds has no positive cycle the assignment is optimal.
template <int DT, bool SM>
__device__ __noinline__ bool assign_candidates(const Layer& layer, Team& tm, const int32_t (&prices)[DT],
                                               float tau, bool& unique) {
    Shared& sh = shared();
    const Layer L = layer;               // in registers: the passes would reload what references name
    int32_t p[DT];
#pragma unroll
    for (int l = 0; l < DT; ++l) p[l] = prices[l];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    unique = false;
    auto values = [&](int k, int64_t (&v)[DT]) {
#pragma unroll
        for (int l = 0; l < DT; ++l) {
            const int i = l * L.np + k;
            v[l] = (static_cast<int64_t>(hi_of<SM>(L)[i] - p[l]) << L.sh) + lo_of<SM>(L)[i];
        }
    };
    if (tid < DT * DT) {
        const int a = tid / DT, b = tid % DT;
        const float x = tau * fmaxf(sh.scale[a], sh.scale[b]) * static_cast<float>(1 << L.sh);
        sh.bound[a][b] = tau < 0.0f || x >= 1.0e15f ? kBoundMax : static_cast<int64_t>(x);
    }
    __syncthreads();
    // the list is kept by block 0 of the team
    int* ncand = at_rank(&sh.ncand, 0);
    for (int k = tid; k < L.n; k += kThreads) {
        int64_t v[DT];
        values(k, v);
        int a = 0;
        int64_t va = v[0];
#pragma unroll
        for (int l = 1; l < DT; ++l)
            if (v[l] > va) va = v[l], a = l;
        nu_of<SM>(L)[k] = static_cast<uint8_t>(a);
        atomicAdd(&sh.hist[tm.ph][kBins + a], 1u);
        bool in = false;
#pragma unroll
        for (int l = 0; l < DT; ++l) in |= l != a && va - v[l] <= sh.bound[a][l];
        if (in) {
            const int slot = atomicAdd(ncand, 1);
            if (slot < kCand) {
                *at_rank(&sh.ck[slot], 0) = L.k0 + k;
                *at_rank(&sh.cnu[slot], 0) = static_cast<uint8_t>(a);
#pragma unroll
                for (int l = 0; l < DT; ++l) *at_rank(&sh.cv[l][slot], 0) = v[l];
            }
        }
    }
    team_counters(tm);
    if (tm.rank == 0) {
        const int C = sh.ncand;
        if (tid < DMAX) sh.count[tid] = tid < DT ? static_cast<int>(sh.counters[tid]) : 0;
        if (tid == 0) sh.flag = C <= kCand ? 0 : 2, sh.dirty = (1u << DT) - 1u;
        if (tid < DMAX) sh.clen[tid] = 0;
        __syncthreads();
        if (tid < C && C <= kCand) {
            const int a = sh.cnu[tid];
            sh.clist[a][atomicAdd(&sh.clen[a], 1)] = static_cast<uint8_t>(tid);
        }
        __syncthreads();
        // flag: 0 moving, 1 balanced, 2 given up; each round moves one unit of excess.  Only the
        // edges out of the devices that the last path touched change: a warp per edge.
        for (int round = 0; sh.flag == 0; ++round) {
            const unsigned dirty = sh.dirty;
            for (int e = warp; e < DT * DT; e += kWarps) {
                // entry e of the touched rows first, so that they spread over the warps
                int row = e / DT;
                unsigned rows = dirty;
                for (; row > 0 && rows; --row) rows &= rows - 1;
                if (!rows) break;
                const int a = __ffs(rows) - 1, b = e % DT;
                if (a == b) continue;
                uint64_t best = 0;
                const int len = sh.clen[a];
                for (int c = lane; c < len; c += 32) {
                    const int slot = sh.clist[a][c];
                    const uint64_t key = pack_cand(sh.cv[b][slot] - sh.cv[a][slot], slot);
                    best = key > best ? key : best;
                }
                best = warp_max_u64(best);
                if (lane == 0) sh.E[a][b] = best;
            }
            __syncthreads();
            if (warp == 0) {
                const int cnt = lane < DT ? sh.count[lane] : L.cap;
                const unsigned src = __ballot_sync(0xFFFFFFFFu, cnt > L.cap);
                const unsigned snk = __ballot_sync(0xFFFFFFFFu, cnt < L.cap);
                if (src == 0) {
                    if (lane == 0) sh.flag = 1;
                } else {
                    int64_t w[DT], dist;
                    int pred;
#pragma unroll
                    for (int a = 0; a < DT; ++a) {
                        const uint64_t e = lane < DT && lane != a ? sh.E[a][lane] : 0;
                        w[a] = e ? cand_gain(e) : kNegInf;
                    }
                    bellman_ford_warp<DT>(src, w, dist, pred);
                    int end = -1;
                    int64_t best = kNegInf;
                    for (int b = 0; b < DT; ++b) {
                        const int64_t x = __shfl_sync(0xFFFFFFFFu, dist, b);
                        if (((snk >> b) & 1u) && x > best) best = x, end = b;
                    }
                    unsigned touched = 0;
                    int v = end, steps = 0;
                    bool ok = end >= 0 && round < kCand;
                    while (ok) {
                        const int a = __shfl_sync(0xFFFFFFFFu, pred, v);
                        if (a < 0) break;
                        if (++steps > DT) { ok = false; break; }
                        const int slot = cand_slot(sh.E[a][v]), len = sh.clen[a];
                        const uint8_t tail = sh.clist[a][len - 1];
                        __syncwarp();
                        for (int c = lane; c < len; c += 32)
                            if (sh.clist[a][c] == slot) sh.clist[a][c] = tail;
                        if (lane == 0) {
                            sh.cnu[slot] = static_cast<uint8_t>(v);
                            sh.clen[a] = len - 1;
                            sh.clist[v][sh.clen[v]++] = static_cast<uint8_t>(slot);
                        }
                        __syncwarp();
                        touched |= (1u << a) | (1u << v);
                        v = a;
                    }
                    if (lane == 0) {
                        if (ok) sh.count[v] -= 1, sh.count[end] += 1, sh.dirty = touched;
                        else sh.flag = 2;
                    }
                }
            }
            __syncthreads();
        }
        if (warp == 0 && sh.flag == 1) {
            for (int i = lane; i < DT * DT; i += 32) {
                const int a = i / DT, b = i % DT;
                const uint64_t e = sh.E[a][b];
                const int64_t out = -sh.bound[a][b] - 1;
                const int64_t w = e ? cand_gain(e) : out;
                sh.P[a][b] = a == b ? 0 : (w > out ? w : out);
            }
            __syncwarp();
            close_paths(DT);
            const bool cycle = lane < DT && sh.P[lane][lane] > 0;
            if (__any_sync(0xFFFFFFFFu, cycle) && lane == 0) sh.flag = 2;
        }
    }
    team_sync(tm);
    if (*at_rank(&sh.flag, 0) != 1) return false;
    const int C = *at_rank(&sh.ncand, 0);
    if (tid < C) {
        const int k = *at_rank(&sh.ck[tid], 0) - L.k0;
        const uint8_t to = *at_rank(&sh.cnu[tid], 0);
        if (k >= 0 && k < L.n) nu_of<SM>(L)[k] = to;
    }
    if (tm.rank != 0 && tid >= kCand && tid < kCand + DT * DT) {
        const int a = (tid - kCand) / DT, b = (tid - kCand) % DT;
        sh.P[a][b] = *at_rank(&sh.P[a][b], 0);
    }
    __syncthreads();
    // another optimum would move some k from nu(k) = t to l < t and close the cycle at no loss
    bool open = false;
    for (int k = tid; k < L.n; k += kThreads) {
        int64_t v[DT];
        values(k, v);
        const int t = nu_of<SM>(L)[k];
        int64_t vt = v[0];
#pragma unroll
        for (int l = 1; l < DT; ++l)
            if (l == t) vt = v[l];
#pragma unroll
        for (int l = 0; l < DT; ++l) open |= l < t && v[l] - vt + sh.P[l][t] >= 0;
    }
    if (__any_sync(0xFFFFFFFFu, open) && lane == 0) atomicAdd(&sh.hist[tm.ph][kBins], 1u);
    if (tid < DT) {
        int64_t pot = 0;
        for (int a = 0; a < DT; ++a) pot = sh.P[a][tid] > pot ? sh.P[a][tid] : pot;
        int64_t own = 0;
#pragma unroll
        for (int l = 0; l < DT; ++l)
            if (l == tid) own = p[l];
        sh.pi[tid] = (own << L.sh) + pot;
    }
    team_counters(tm);
    unique = sh.counters[0] == 0;
    return true;
}

// Exchange graph over the team's neurons with index > lo: w[a][b] = packed (max gain of moving such a
// neuron from a to b, lowest index among ties).  lo < 0: all neurons, into sh.w, only the edges out of the
// devices in sh.dirty (the others stand from before); else into sh.wk.
template <int DT, bool SM>
__device__ __noinline__ void exchange_graph(const Layer& L, Team& tm, int lo) {
    Shared& sh = shared();
    uint64_t* wl = sh.wl[tm.wph];
    const unsigned rows = lo < 0 ? sh.dirty : (1u << DT) - 1u;
    const int first = lo < L.k0 ? 0 : lo + 1 - L.k0;
    if (threadIdx.x < DMAX * DMAX) wl[threadIdx.x] = 0;
    __syncthreads();
    for (unsigned left = rows; left; left &= left - 1) {
        const int a = __ffs(left) - 1;
        uint64_t best[DT];
#pragma unroll
        for (int b = 0; b < DT; ++b) best[b] = 0;
        for (int k = first + threadIdx.x; k < L.n; k += kThreads) {
            if (nu_of<SM>(L)[k] != a) continue;
            const int64_t ma = gain_at<SM>(L, a, k);
#pragma unroll
            for (int b = 0; b < DT; ++b)
                if (b != a) {
                    const uint64_t key = pack_gain(gain_at<SM>(L, b, k) - ma, L.k0 + k);
                    best[b] = key > best[b] ? key : best[b];
                }
        }
#pragma unroll
        for (int b = 0; b < DT; ++b)
            if (b != a) {
                const uint64_t r = warp_max_u64(best[b]);
                if ((threadIdx.x & 31) == 0 && r)
                    atomicMax(reinterpret_cast<unsigned long long*>(&wl[a * DMAX + b]), r);
            }
    }
    team_sync(tm);
    if (threadIdx.x < DMAX * DMAX) {
        const int a = threadIdx.x / DMAX, b = threadIdx.x % DMAX;
        if ((rows >> a) & 1u)
            (lo < 0 ? sh.w : sh.wk)[a][b] =
                team_combine(wl + threadIdx.x, tm, [](uint64_t a, uint64_t b) { return a > b ? a : b; });
    }
    __syncthreads();
    tm.wph ^= 1;
}

// bellman_ford_warp on an exchange graph in shared memory: the edges stay there, as registers that this
// takes are taken from the price steps.
template <int DT>
__device__ __forceinline__ void bellman_ford_graph(const uint64_t (&graph)[DMAX][DMAX], unsigned src, int64_t& dist,
                                                   int& pred) {
    const int b = threadIdx.x & 31;
    dist = (src >> b) & 1u ? 0 : kNegInf;
    pred = -1;
#pragma unroll 1
    for (int round = 0; round < DT - 1; ++round) {
        const int64_t before = dist;
        bool moved = false;
#pragma unroll 1
        for (int a = 0; a < DT; ++a) {
            const int64_t from = __shfl_sync(0xFFFFFFFFu, before, a);
            const uint64_t e = b < DT && b != a ? graph[a][b] : 0;
            if (e && from != kNegInf && from + gain_of(e) > dist) dist = from + gain_of(e), pred = a, moved = true;
        }
        if (!__any_sync(0xFFFFFFFFu, moved)) break;
    }
}

// Warp 0 of every block: the best neuron of each edge of the path ending at `end` moves (lane b holds
// device b's predecessor on the path, -1 at its start); each block applies the moves of its own slice.
// Returns the path's start, -1 if it has none; its devices go to sh.dirty.
template <int DT, bool SM>
__device__ __forceinline__ int apply_path(const Layer& L, const uint64_t (&graph)[DMAX][DMAX], int pred, int end) {
    Shared& sh = shared();
    const bool lane0 = (threadIdx.x & 31) == 0;
    unsigned touched = 0;
    int v = end;
    for (int steps = 0; steps < DT; ++steps) {        // a path visits a device once
        touched |= 1u << v;
        const int a = __shfl_sync(0xFFFFFFFFu, pred, v);
        if (a < 0) {
            if (lane0) sh.dirty = touched;
            return v;
        }
        const int k = index_of(graph[a][v]) - L.k0;
        if (lane0 && k >= 0 && k < L.n) nu_of<SM>(L)[k] = static_cast<uint8_t>(v);
        v = a;
    }
    return -1;
}

// Warp 0's parts of the repair, out of line: their registers would be taken from the price steps.
// One unit of excess along the maximum-gain path of sh.w.
template <int DT, bool SM>
__device__ __noinline__ void move_excess(const Layer& L) {
    Shared& sh = shared();
    const int lane = threadIdx.x & 31;
    const int cnt = lane < DT ? sh.count[lane] : L.cap;
    const unsigned src = __ballot_sync(0xFFFFFFFFu, cnt > L.cap);
    const unsigned snk = __ballot_sync(0xFFFFFFFFu, cnt < L.cap);
    int64_t dist;
    int pred;
    bellman_ford_graph<DT>(sh.w, src, dist, pred);
    int e = -1;
    int64_t best = kNegInf;
#pragma unroll 1
    for (int b = 0; b < DT; ++b) {
        const int64_t x = __shfl_sync(0xFFFFFFFFu, dist, b);
        if (((snk >> b) & 1u) && x > best) best = x, e = b;
    }
    const int s = e < 0 ? -1 : apply_path<DT, SM>(L, sh.w, pred, e);
    if (lane == 0) {
        if (s < 0) sh.status = DTP_ERR_NOT_CONVERGED;
        else sh.count[s] -= 1, sh.count[e] += 1;
    }
}

// All-pairs paths of sh.w, and prices for the next neuron step: longest paths from a zero root.
template <int DT>
__device__ __noinline__ void close_graph() {
    Shared& sh = shared();
    const int lane = threadIdx.x & 31;
    for (int i = lane; i < DT * DT; i += 32) {
        const int a = i / DT, b = i % DT;
        sh.P[a][b] = a == b ? 0 : (sh.w[a][b] ? gain_of(sh.w[a][b]) : kNegInf);
    }
    __syncwarp();
    close_paths(DT);
    if (lane < DT) {
        if (sh.P[lane][lane] > 0) sh.status = DTP_ERR_NOT_CONVERGED;   // a positive cycle: not optimal
        int64_t pot = 0;
        for (int a = 0; a < DT; ++a) pot = sh.P[a][lane] > pot ? sh.P[a][lane] : pot;
        sh.pi[lane] = pot;
    }
}

// Neuron kstar (its gains and its device t in sh.B) to the smallest device that a zero-gain path through
// sh.wk back to t allows.
template <int DT, bool SM>
__device__ __noinline__ void move_earlier(const Layer& L, int kstar) {
    Shared& sh = shared();
    const int lane = threadIdx.x & 31;
    const int t = static_cast<int>(sh.B[DT]);
    int64_t dist;
    int pred;
    if (lane == 0) sh.dirty = 0;
#pragma unroll 1
    for (int l = 0; l < t; ++l) {
        bellman_ford_graph<DT>(sh.wk, 1u << l, dist, pred);
        const int64_t to = __shfl_sync(0xFFFFFFFFu, dist, t);
        if (to == kNegInf || sh.B[l] - sh.B[t] + to != 0) continue;
        if (apply_path<DT, SM>(L, sh.wk, pred, t) < 0 && lane == 0) sh.status = DTP_ERR_NOT_CONVERGED;
        const int k = kstar - L.k0;
        if (lane == 0 && k >= 0 && k < L.n) nu_of<SM>(L)[k] = static_cast<uint8_t>(l);
        break;
    }
}

// Step (d) over all neurons.  assigned: L.nu is already optimal; else it is the assignment at some
// prices and is balanced first.  Warp 0 of every block of a team repeats the steps over the devices on
// equal data.
template <int DT, bool SM>
__device__ __noinline__ void repair_all(const Layer& L, Team& tm, bool assigned) {
    Shared& sh = shared();
    const int N = L.N, D = L.D, cap = L.cap;
    if (threadIdx.x == 0) sh.dirty = (1u << DT) - 1u;
    __syncthreads();
    if (!assigned) {
        for (int k = threadIdx.x; k < L.n; k += kThreads) atomicAdd(&sh.hist[tm.ph][kBins + nu_of<SM>(L)[k]], 1u);
        team_counters(tm);
        if (threadIdx.x < DMAX) sh.count[threadIdx.x] = static_cast<int>(sh.counters[threadIdx.x]);
        __syncthreads();
        // successive maximum-gain paths until balanced
        for (int aug = 0; aug < 4 * N + 16; ++aug) {
            int ex = 0;
            for (int l = 0; l < D; ++l) ex += sh.count[l] > cap ? 1 : 0;
            if (ex == 0) break;
            exchange_graph<DT, SM>(L, tm, -1);
            if (threadIdx.x < 32) move_excess<DT, SM>(L);
            if (threadIdx.x == 0 && sh.beat && (aug & 31) == 31) atomicAdd(sh.beat, 1);
            __syncthreads();
            if (sh.status != DTP_OK) return;
        }
        __syncthreads();
        if (threadIdx.x == 0)
            for (int l = 0; l < D; ++l)
                if (sh.count[l] != cap) sh.status = DTP_ERR_NOT_CONVERGED;
        __syncthreads();
        if (sh.status != DTP_OK) return;
    }
    // lexicographically smallest optimum
    int kstart = 0;
    for (int round = 0; round < N + 1; ++round) {
        exchange_graph<DT, SM>(L, tm, -1);
        if (threadIdx.x < 32) close_graph<DT>();
        if (threadIdx.x == 0 && sh.beat && (round & 31) == 31) atomicAdd(sh.beat, 1);
        __syncthreads();
        if (sh.status != DTP_OK) return;
        uint32_t cand = static_cast<uint32_t>(N);
        for (int k = threadIdx.x; k < L.n && cand == static_cast<uint32_t>(N); k += kThreads) {
            if (L.k0 + k < kstart) continue;
            const int t = nu_of<SM>(L)[k];
            const int64_t mt = gain_at<SM>(L, t, k);
            for (int l = 0; l < t; ++l)
                if (sh.P[l][t] != kNegInf && gain_at<SM>(L, l, k) - mt + sh.P[l][t] == 0) {
                    cand = static_cast<uint32_t>(L.k0 + k);
                    break;
                }
        }
        uint32_t unused = 0;
        team_min_max(cand, unused, tm);
        const int kstar = static_cast<int>(cand);
        if (kstar >= N) break;
        exchange_graph<DT, SM>(L, tm, kstar);
        // the gains and the device of kstar, from the block that holds it
        if (threadIdx.x <= DT) {
            const int k = kstar - L.k0;
            const bool own = k >= 0 && k < L.n;
            sh.xl[tm.lph][threadIdx.x] =
                !own ? 0 : (threadIdx.x < DT ? gain_at<SM>(L, threadIdx.x, k) : static_cast<int64_t>(nu_of<SM>(L)[k]));
        }
        team_sum_i64(DT + 1, tm);
        if (threadIdx.x < 32) move_earlier<DT, SM>(L, kstar);
        __syncthreads();
        if (sh.status != DTP_OK) return;
        kstart = kstar + 1;
    }
}

// One pass over n neurons of a slice at the prices p: the devices' neuron counts and, for every pair
// of devices, the neurons whose first two choices they are by less than tau (sh.counters; gaps over
// the larger of the two devices' scales); with the histogram of the gaps, `gap` = where about
// kCandTarget of them lie.  Returns the neurons in excess of cap.
template <int DT, bool SM>
__device__ __forceinline__ int gap_pass(const Layer& layer, int n, int cap, Team& tm,
                                     const int32_t (&prices)[DT], float tau, Pick& gap) {
    Shared& sh = shared();
    const Layer L = layer;
    int32_t p[DT];
#pragma unroll
    for (int l = 0; l < DT; ++l) p[l] = prices[l];
    constexpr uint32_t kExp0 = (127u - 45u) << 3;   // bins of an eighth of an octave from 2^-45
    float inv[DT];
#pragma unroll
    for (int l = 0; l < DT; ++l) inv[l] = 1.0f / sh.scale[l];
    uint32_t* hist = sh.hist[tm.ph];
    for_neurons(n, [&](int k) {
        int32_t v[DT];
#pragma unroll
        for (int l = 0; l < DT; ++l) v[l] = hi_of<SM>(L)[l * L.np + k] - p[l];
        int a = 0;
        int32_t va = v[0];
        float ia = inv[0];
#pragma unroll
        for (int l = 1; l < DT; ++l)
            if (v[l] > va) va = v[l], a = l, ia = inv[l];
        float m = __int_as_float(0x7F000000);
        int b = 0, vb = INT32_MIN;
#pragma unroll
        for (int l = 0; l < DT; ++l)
            if (l != a) {
                // the difference of two int32 needs 32 bits without a sign
                const uint32_t gap32 = static_cast<uint32_t>(va) - static_cast<uint32_t>(v[l]);
                m = fminf(m, __uint2float_rz(gap32) * fminf(ia, inv[l]));
                if (v[l] > vb) vb = v[l], b = l;
            }
        const uint32_t e = __float_as_uint(m) >> 20;
        const uint32_t bin = e <= kExp0 ? 0u : min(e - kExp0, static_cast<uint32_t>(kBins - 1));
        atomicAdd(&hist[kBins - 1 - bin], 1u);      // smallest gaps in the top bins
        atomicAdd(&hist[kBins + a], 1u);
        if (m <= tau) {
            const int lo = min(a, b), hi = max(a, b);
            atomicAdd(&hist[kBins + kPairs + lo * (2 * DT - lo - 1) / 2 + hi - lo - 1], 1u);
        }
    });
    gap = team_pick(kCandTarget + 1, tm);
    // gaps of the bins above the picked one are below this (the edge of a float's upper bits)
    gap.bin = (kBins - 1 - gap.bin + kExp0) << 20;
    int excess = 0;
#pragma unroll
    for (int l = 0; l < DT; ++l) {
        const int c = static_cast<int>(sh.counters[l]);
        excess += c > cap ? c - cap : 0;
    }
    return excess;
}

// A Newton step on the counts of the last gap_pass: with d[a][b] neurons per unit of price difference
// near the boundary of a and b (those within tau of it, both sides), raising the prices by x moves
// Laplacian(d) x neurons, so solve for the excess, device 0 fixed.  Warp 0 solves (lane j holds column
// j, lane DT the right side; diagonally dominant, so without pivoting) and hands the prices on.
template <int DT>
__device__ __forceinline__ void newton_step(int cap, float tau, int32_t (&p)[DT]) {
    Shared& sh = shared();
    const int lane = threadIdx.x & 31;
    if (threadIdx.x < 32) {
        float col[DT], piv[DT];
        float diag = 0.0f;
#pragma unroll
        for (int i = 0; i < DT; ++i) {
            col[i] = 0.0f;
            if (lane < DT && lane != i) {
                const int lo = min(i, lane), hi = max(i, lane);
                const float t = static_cast<float>(sh.counters[kPairs + lo * (2 * DT - lo - 1) / 2 + hi - lo - 1]);
                col[i] = -(t + 0.25f) / (2.0f * tau * fmaxf(sh.scale[i], sh.scale[lane]));
                diag -= col[i];
            } else if (lane == DT) {
                col[i] = static_cast<float>(static_cast<int>(sh.counters[i]) - cap);
            }
        }
#pragma unroll
        for (int i = 0; i < DT; ++i)
            if (lane == i) col[i] = diag;
#pragma unroll
        for (int c = 1; c < DT; ++c) {
            piv[c] = __shfl_sync(0xFFFFFFFFu, col[c], c);
            const float r = 1.0f / piv[c];
#pragma unroll
            for (int i = 1; i < DT; ++i) {
                const float f = __shfl_sync(0xFFFFFFFFu, col[i], c) * r;
                if (i != c) col[i] -= f * col[c];
            }
        }
        if (lane == DT) {
#pragma unroll
            for (int c = 0; c < DT; ++c) {
                const float x = c == 0 ? 0.0f : col[c] / piv[c == 0 ? 1 : c];
                const float q = static_cast<float>(p[c]) + x;
                sh.price[c] = static_cast<int32_t>(fminf(fmaxf(q, -0.99f * kPriceMax), 0.99f * kPriceMax));
                if (fabsf(x) < 8388608.0f) sh.price[c] = p[c] + static_cast<int32_t>(rintf(x));
            }
        }
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < DT; ++c) p[c] = max(-kPriceMax, min(kPriceMax, sh.price[c]));
    __syncthreads();
}

// A Gauss-Seidel sweep over n neurons of a slice: each price in turn is set so that about cap neurons
// (within tol) prefer its device at the others' prices.  A histogram of the keys around the old price on
// the scale of its last change (sh.price_step: every thread would keep the same) usually holds the new
// one, which saves the pass for their range and the refinement.
template <int DT, bool SM>
__device__ __forceinline__ void price_sweep(const Layer& layer, int n, int cap, uint32_t tol, Team& tm,
                                         int32_t (&prices)[DT]) {
    Shared& sh = shared();
    const Layer L = layer;
    int32_t p[DT];
#pragma unroll
    for (int l = 0; l < DT; ++l) p[l] = prices[l];
#pragma unroll 1
    for (int l = 0; l < DT; ++l) {
        auto key = [&](int k, uint32_t& x) -> bool {
            int32_t own = 0, alt = INT32_MIN;
#pragma unroll
            for (int m = 0; m < DT; ++m) {
                const int32_t h = hi_of<SM>(L)[m * L.np + k];
                if (m == l) own = h;
                else alt = max(alt, h - p[m]);
            }
            x = static_cast<uint32_t>(own - alt) ^ 0x80000000u;
            return true;
        };
        int32_t old = 0;
#pragma unroll
        for (int m = 0; m < DT; ++m)
            if (m == l) old = p[m];
        const int32_t width = sh.price_step[l];
        uint32_t t = 0, ge = 0;
        bool found = false;
        if (width >= 0) {
            // everything above the window counts in the top bin
            const int32_t w = max(width, kBins), from = old - w;
            const int s = bin_shift(static_cast<uint32_t>(2 * w));
            uint32_t* hist = sh.hist[tm.ph];
            for_neurons(n, [&](int k) {
                uint32_t x;
                key(k, x);
                const int64_t d = static_cast<int64_t>(static_cast<int32_t>(x ^ 0x80000000u)) - from;
                if (d >= 0) {
                    const int64_t b = d >> s;
                    atomicAdd(&hist[b < kBins - 1 ? static_cast<int>(b) : kBins - 1], 1u);
                }
            });
            const Pick near = team_pick(static_cast<uint32_t>(cap), tm);
            if (near.found && near.bin < kBins - 1 && near.inside <= cap - near.above + 2 * tol) {
                found = true;
                t = static_cast<uint32_t>(from + static_cast<int32_t>(near.bin << s)) ^ 0x80000000u;
            }
        }
        if (!found) {
            uint32_t lo = 0xFFFFFFFFu, hi = 0u;
            for_neurons(n, [&](int k) {
                uint32_t x;
                key(k, x);
                lo = min(lo, x);
                hi = max(hi, x);
            });
            team_min_max(lo, hi, tm);
            select_threshold(n, lo, hi - lo, static_cast<uint32_t>(cap), tol, key, t, ge, tm);
        }
        const int32_t now = max(-kPriceMax, min(kPriceMax, static_cast<int32_t>(t ^ 0x80000000u)));
#pragma unroll
        for (int m = 0; m < DT; ++m)
            if (m == l) {
                const int64_t d = static_cast<int64_t>(now) - p[m];
                const int64_t ad = d < 0 ? -d : d;
                if (threadIdx.x == 0) sh.price_step[m] = static_cast<int32_t>(ad < kPriceMax / 4 ? ad : kPriceMax / 4);
                p[m] = now;
            }
    }
#pragma unroll
    for (int l = 0; l < DT; ++l) prices[l] = p[l];
}

// Step (a): prices p at which at most `stop` of the n neurons are in excess of cap, or as near as the
// passes get.  A sweep costs DT exchanges and always makes headway; a Newton step costs one pass and
// shrinks a small excess 5 to 10 times, but not a large one: it is taken below n / 12 while it works.
// On model-shaped layers with 4 devices the excess goes 70%, 20% (sweep), 2% (sweep), 0.4%, 0.1%.
// Ends with a gap_pass at p, whose threshold for candidates is returned (-1: all neurons).  Gives up
// with -2 where an excess is above `most`.
template <int DT, bool SM>
__device__ __noinline__ float find_prices(const Layer& L, int n, int cap, int stop, int most, Team& tm,
                                          int32_t (&p)[DT]) {
    Shared& sh = shared();
    if (threadIdx.x < DT) sh.price_step[threadIdx.x] = -1;      // read after the first gap_pass's barriers
    int best = INT32_MAX, stalled = 0;
    bool newton = false;
    float tau = 0.015625f;
    Pick gap;
    for (int pass = 0;; ++pass) {
        const int excess = gap_pass<DT, SM>(L, n, cap, tm, p, tau, gap);
        if (excess <= stop || pass == kMaxPasses || stalled == 2) break;
        if (excess > most) return -2.0f;
        bool sweep = newton && excess > best - best / 3;
        if (excess < best) {
            if (!newton) stalled = 0;
            best = excess;
#pragma unroll
            for (int l = 0; l < DT; ++l)
                if (threadIdx.x == 0) sh.best_price[l] = p[l];   // read after the next gap_pass's barriers
        } else {
            if (!newton) ++stalled;                  // ties: no price separates them
#pragma unroll
            for (int l = 0; l < DT; ++l) p[l] = sh.best_price[l];
            sweep = true;
        }
        newton = !sweep && best <= cap * DT / 12;
        if (newton) newton_step<DT>(cap, tau, p);
        else price_sweep<DT, SM>(L, n, cap, static_cast<uint32_t>(best / (4 * DT)) + 1u, tm, p);
        // pairs are counted next time within twice the gap that holds the nearest candidates
        if (gap.found && gap.above > 0) tau = 2.0f * __uint_as_float(gap.bin);
    }
    if (!gap.found) return -1.0f;
    return gap.above == 0 ? 0.0f : __uint_as_float(gap.bin);
}

// Steps (a) to (c).  Returns what repair_all still has to do: 0 nothing, 1 the lexicographic order, 2 all.
template <int DT, bool SM>
__device__ __noinline__ int neuron_step_general(const Layer& L, Team& tm) {
    Shared& sh = shared();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    int32_t p[DT];                       // prices, the same in every thread of the team
    {
        int64_t base = sh.pi[0];
#pragma unroll
        for (int l = 1; l < DT; ++l) base = sh.pi[l] < base ? sh.pi[l] : base;
#pragma unroll
        for (int l = 0; l < DT; ++l) {
            const int64_t x = (sh.pi[l] - base) >> L.sh;
            p[l] = static_cast<int32_t>(x < kPriceMax ? x : kPriceMax);
        }
    }
    // the devices' relative gain sizes, from block 0's slice
    if (tm.rank == 0) {
        uint32_t hs[DT];
#pragma unroll
        for (int l = 0; l < DT; ++l) hs[l] = 0;
        for (int k = tid; k < L.n; k += kThreads)
#pragma unroll
            for (int l = 0; l < DT; ++l) hs[l] += static_cast<uint32_t>(hi_of<SM>(L)[l * L.np + k]) >> 10;
#pragma unroll
        for (int l = 0; l < DT; ++l) {
            // below 2^19 a neuron: slices in shared memory stay within 32 bits, larger ones need not
            const int64_t s = SM ? __reduce_add_sync(0xFFFFFFFFu, hs[l]) : warp_sum_i64(hs[l]);
            if (lane == 0) sh.part[warp][l] = s;
        }
        __syncthreads();
        if (warp < DT) {
            float s = lane < kWarps ? static_cast<float>(sh.part[lane][warp]) : 0.0f;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
            if (lane == 0) sh.scale[warp] = fmaxf(s * 1024.0f / static_cast<float>(L.n), 1.0f);
        }
        if (tid == 0) sh.ncand = 0;
    }
    team_sync(tm);
    if (tm.rank != 0 && tid < DT) sh.scale[tid] = *at_rank(&sh.scale[tid], 0);
    __syncthreads();
    // (a) prices.  A team first finds them for block 0's slice alone, which needs no exchange between
    // blocks (an exchange costs some 3,000 cycles): they leave a few percent of all neurons in excess.
    const int stop = 3 * DT, any = INT32_MAX;
    float tau = find_prices<DT, SM>(L, L.n, L.cap, stop, tm.cl > 1 ? L.N / 12 : any, tm, p);
    if (tau == -2.0f) {
        team_sync(tm);                               // the peers have read block 0's histogram
        if (tm.rank == 0) {
            Team own = tm;
            own.cl = 1;
            find_prices<DT, SM>(L, L.n, L.n / DT, max(2 * DT, L.n / 32), any, own, p);
            for (int i = tid; i < 2 * (kBins + kCounters); i += kThreads)
                sh.hist[i / (kBins + kCounters)][i % (kBins + kCounters)] = 0;
            if (tid < DT) {
#pragma unroll
                for (int l = 0; l < DT; ++l)
                    if (l == tid) sh.price[l] = p[l];
            }
        }
        team_sync(tm);
        if (tm.rank != 0) {
#pragma unroll
            for (int l = 0; l < DT; ++l) p[l] = *at_rank(&sh.price[l], 0);
        }
        tau = find_prices<DT, SM>(L, L.n, L.cap, stop, any, tm, p);
    }
    // (b) and (c)
    bool unique;
    if (!assign_candidates<DT, SM>(L, tm, p, tau, unique)) return 2;
    return unique ? 0 : 1;
}

template <int DT, bool SM>
__device__ __forceinline__ void neuron_step(const Layer& L, Team& tm) {
    Shared& sh = shared();
    if constexpr (DT == 2) neuron_step_d2<SM>(L, tm);
    else if (const int left = neuron_step_general<DT, SM>(L, tm)) repair_all<DT, SM>(L, tm, left == 1);   // (d)
}

// --------------------------------------------------------------- head step --

// sh.xl[phase][r * DT + l] = the slice's sum of score row r over its neurons on device l, for rows
// r < rows; nu: the slice's labels.  The neurons are first listed by device (over the gains, which the
// next step rebuilds),
// then a power of two of threads adds each (row, device) list: 2.5 times fewer instructions than
// walking every row with a select per device.  In global memory, where the loads' latency counts, several
// warps add a list where there are few, four neurons at a time; in shared memory that would only be more code
// to fetch (1 us of a small layer's 25).
template <int DT, bool SM>
__device__ __noinline__ void column_sums(const Layer& layer, const uint8_t* nu, Team& tm, int rows) {
    Shared& sh = shared();
    const Layer L = layer;
    const int tid = threadIdx.x, lane = tid & 31;
    uint16_t* lists = SM ? reinterpret_cast<uint16_t*>(dsm + kData) : L.lists;
    const bool wide = L.rnp > 65535;            // 32-bit indices: only where no cluster of four can be resident
    uint32_t* lists32 = reinterpret_cast<uint32_t*>(lists);
    if (tid < DMAX) sh.clen[tid] = 0;
    if (!SM && tid < rows * DT) sh.xl[tm.lph][tid] = 0;
    __syncthreads();
    for (int k0 = 0; k0 < L.n; k0 += kThreads) {
        const int k = k0 + tid;
        const int a = k < L.n ? nu[k] : DT;
        const unsigned same = __match_any_sync(0xFFFFFFFFu, a);
        int at = 0;
        if (a < DT && lane == __ffs(same) - 1) at = atomicAdd(&sh.clen[a], __popc(same));
        at = __shfl_sync(0xFFFFFFFFu, at, __ffs(same) - 1) + __popc(same & ((1u << lane) - 1u));
        if (a < DT) {
            if (wide) lists32[a * L.rnp + at] = static_cast<uint32_t>(k);
            else lists[a * L.rnp + at] = static_cast<uint16_t>(k);
        }
    }
    __syncthreads();
    const int pairs = rows * DT;                                // 4 to 256
    int tpp = SM ? 32 : kThreads / 4;
    while (tpp * pairs > kThreads) tpp >>= 1;                   // from 2
    if (tid < pairs * tpp) {                                    // whole groups of tpp lanes, or whole warps
        const int pair = tid / tpp, sub = tid % tpp;
        const int r = pair / DT, l = pair % DT;
        const int len = sh.clen[l];
        int64_t hs = 0;
        uint32_t ls = 0;
        auto entry = [&](int j) -> int {
            return wide ? static_cast<int>(lists32[l * L.rnp + j]) : lists[l * L.rnp + j];
        };
        int j = sub;
        if constexpr (!SM) {
            for (; j + 3 * tpp < len; j += 4 * tpp) {           // four neurons' loads in flight
                int k[4];
                uint32_t h[4], lo[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) k[u] = entry(j + u * tpp);
#pragma unroll
                for (int u = 0; u < 4; ++u) score_parts<SM>(L, r, k[u], h[u], lo[u]);
#pragma unroll
                for (int u = 0; u < 4; ++u) hs += h[u], ls += lo[u];
            }
        }
        for (; j < len; j += tpp) {
            uint32_t h, lo;
            score_parts<SM>(L, r, entry(j), h, lo);
            hs += h;
            ls += lo;
        }
        // the group's own lanes: their lists differ in length, so they need not leave the loop together
        const int width = tpp < 32 ? tpp : 32;
        const unsigned group = (0xFFFFFFFFu >> (32 - width)) << (lane & ~(width - 1));
        int64_t v = (hs << kLoBits) + ls;
        for (int o = width >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(group, v, o);
        if (SM || tpp <= 32) {
            if (sub == 0) sh.xl[tm.lph][pair] = v;
        } else if (lane == 0) {
            atomicAdd(reinterpret_cast<unsigned long long*>(&sh.xl[tm.lph][pair]), static_cast<unsigned long long>(v));
        }
    }
}

// The best labelled balanced partition for the column sums in sh.B, lexicographically smallest
// among ties, into sh.h (and sh.glist), its score into sh.J.  Dynamic programming over states, the
// devices' remaining capacities (digits of a number in base G/D + 1): f(state) = the largest sum
// that the last heads, as many as the state has places, can still add.  Every accepted (G, D) has at
// most 1024 states, against up to 2^26 partitions, and a state's value is an exact integer sum, so
// choosing the smallest device that attains f head by head gives the partition that scoring them
// all in lexicographic order would.  Block-wide; every block of a team repeats it.
template <int DT>
__device__ __noinline__ void choose_partition(int G) {
    Shared& sh = shared();
    const int per = G / DT, base = per + 1;
    const int tid = threadIdx.x, lane = tid & 31;
    int states = 1;
#pragma unroll
    for (int l = 0; l < DT; ++l) states *= base;
    constexpr int kPer = kStates / kThreads;                    // states per thread
    int sum[kPer];
    unsigned open[kPer];                                        // devices with places left in the state
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
        int rest = tid + u * kThreads;
        sum[u] = 0;
        open[u] = 0;
        if ((rest & ~31) < states) {
#pragma unroll
            for (int l = 0; l < DT; ++l) {
                const int q = rest / base, digit = rest - q * base;
                rest = q;
                sum[u] += digit;
                open[u] |= digit > 0 ? 1u << l : 0u;
            }
            if (tid + u * kThreads >= states) sum[u] = 0;
        }
    }
    if (tid == 0) sh.f[0] = 0;
    __syncthreads();
    for (int s = 1; s <= G; ++s) {
#pragma unroll
        for (int u = 0; u < kPer; ++u)
            if (sum[u] == s) {
                const int state = tid + u * kThreads;
                const int64_t* b = sh.B + (G - s) * DT;
                int64_t best = kNegInf;
                int place = 1;
#pragma unroll
                for (int l = 0; l < DT; ++l) {
                    if ((open[u] >> l) & 1u) {
                        const int64_t x = b[l] + sh.f[state - place];
                        best = x > best ? x : best;
                    }
                    place *= base;
                }
                sh.f[state] = best;
            }
        __syncthreads();
    }
    if (tid < 32) {
        // lane l holds device l's remaining places
        int place = 1;
        for (int l = 0; l < lane && l < DT; ++l) place *= base;
        int left = lane < DT ? per : 0;
        int state = states - 1;
        int64_t f = sh.f[state];
        if (lane == 0) sh.J = f;
        for (int g = 0; g < G; ++g) {
            int64_t x = 0;
            if (left > 0) x = sh.f[state - place];
            const bool hit = left > 0 && sh.B[g * DT + lane] + x == f;
            const int l = __ffs(__ballot_sync(0xFFFFFFFFu, hit)) - 1;
            state -= __shfl_sync(0xFFFFFFFFu, place, l);
            f = __shfl_sync(0xFFFFFFFFu, x, l);
            if (lane == l) --left;
            if (lane == 0) sh.h[g] = l;
        }
        __syncwarp();
        list_heads(sh.h, sh.glist, G, per);
    }
    __syncthreads();
}

// ------------------------------------------------------------- layer set-up --

// How a launch splits a layer: neurons per slice (a multiple of 16); whether block 0 gathers all gains;
// and the score rows that a block keeps in shared memory beside its gains (0: they do not fit and are
// read from global memory).
struct View {
    int np;
    int gathered;
    int rows;
};

__host__ __device__ inline int gains_np(const View& vw, int N) { return vw.gathered ? (N + 15) / 16 * 16 : vw.np; }

// Where a block's slice lies: in shared memory, or in the team's buffer of `per_team` bytes.
template <bool SM>
__device__ __forceinline__ uint8_t* slice_buf(uint8_t* gbuf, int64_t team, size_t per_team, const View& vw, int D,
                                              const Team& tm) {
    if constexpr (SM) return dsm + kData;
    else return gbuf + static_cast<size_t>(team) * per_team + tm.rank * align_up_dev(slice_bytes(vw.np, D), 256);
}

// This block's part, over buf.
static __device__ void layer_view(Layer& L, int G, int N, int D, uint8_t* buf, const View& vw, const Team& tm) {
    L.G = G;
    L.N = N;
    L.D = D;
    L.cap = N / D;
    L.e = 0;
    L.sh = kLoBits;
    L.np = gains_np(vw, N);
    L.rnp = vw.np;
    L.k0 = static_cast<int>(tm.rank) * vw.np;
    L.n = N - L.k0 < vw.np ? (N - L.k0 > 0 ? N - L.k0 : 0) : vw.np;
    L.hi = reinterpret_cast<int32_t*>(buf);
    L.lo = reinterpret_cast<uint16_t*>(buf + static_cast<size_t>(L.np) * D * 4);
    L.nu = buf + static_cast<size_t>(L.np) * D * 6;
    L.lists = reinterpret_cast<uint16_t*>(buf);
    L.A = nullptr;
    L.nU = L.nD = nullptr;
    L.qh = nullptr;
    L.ql = nullptr;
    L.q_off = kData + static_cast<int>(align_up_dev(slice_bytes(L.np, D), 16));
    L.q_rows = vw.rows;
}

// The gains that this block writes: its slice's places in block 0's arrays when gathered.
__device__ __forceinline__ Layer gains_of_slice(const Layer& L, const View& vw, const Team& tm) {
    Layer S = L;
    if (vw.gathered && tm.cl > 1) {
        S.hi = at_rank(L.hi, 0) + L.k0;
        S.lo = at_rank(L.lo, 0) + L.k0;
        S.nu = at_rank(L.nu, 0) + L.k0;
    }
    return S;
}

// Where the staged score rows lie: behind the gains and labels.
__device__ __forceinline__ uint32_t* staged_hi(const Layer& L, uint8_t* buf) {
    return reinterpret_cast<uint32_t*>(buf + align_up_dev(slice_bytes(L.np, L.D), 16));
}
__device__ __forceinline__ uint16_t* staged_lo(const Layer& L, uint8_t* buf, int rows) {
    return reinterpret_cast<uint16_t*>(staged_hi(L, buf) + static_cast<size_t>(rows) * L.rnp);
}

// Block 0's view of gathered gains.
__device__ __forceinline__ Layer whole_layer(const Layer& L) {
    Layer F = L;
    F.n = L.N;
    F.k0 = 0;
    return F;
}

// `own`: block 0 as a team of one, for steps on gathered gains.
__device__ __forceinline__ Team make_own(const Team& tm) {
    Team own = tm;
    own.cl = 1;
    return own;
}

// The neuron step of a layer whose gains have been built: by block 0 alone on gathered gains, else by
// the team.  Afterwards the labels can be read through gains_of_slice by every block.
template <int DT, bool SM>
__device__ __forceinline__ void team_neuron_step(const Layer& L, const View& vw, Team& tm, Team& own) {
    Shared& sh = shared();
    if (vw.gathered) {
        team_sync(tm);
        if (tm.rank == 0) {
            const Layer F = whole_layer(L);
            neuron_step<DT, SM>(F, own);
        }
        team_sync(tm);
        if (tm.rank != 0 && threadIdx.x == 0) sh.status = *at_rank(&sh.status, 0);
        __syncthreads();
    } else {
        neuron_step<DT, SM>(L, tm);
    }
}

// The low bits of gains of at most `most` (< 2^44).  A fixed 15 leaves a wide layer's normalised masses
// (2^40 over all entries) some 11 bits above the cut: so many ties at the selection's upper key that
// most of a step ran on the second key (one layer, N = 14336, D = 8: 10.1 ms fixed, 0.34 ms like this).
// The shift by a run-time count costs layers that would not need it: 28 layers, D = 4: 301 us fixed, 316.
__device__ __forceinline__ int low_bits(int64_t most) {
    const int bits = 64 - __clzll(most);
    return bits <= kHiBits ? 0 : (bits - kHiBits < kLoBits ? bits - kHiBits : kLoBits);
}

// Statuses, prices and both histograms cleared.
__device__ __forceinline__ void init_shared() {
    Shared& sh = shared();
    for (int i = threadIdx.x; i < 2 * (kBins + kCounters); i += kThreads)
        sh.hist[i / (kBins + kCounters)][i % (kBins + kCounters)] = 0;
    if (threadIdx.x < DMAX) sh.pi[threadIdx.x] = 0;
    if (threadIdx.x == 0) sh.status = DTP_OK, sh.beat = nullptr;
}

// Validity of A [G][N] (from the slice's first neuron), the fixed-point exponent, and the staged scores.
__device__ __forceinline__ bool layer_prologue(Layer& L, Team& tm, const float* A, uint8_t* buf, const View& vw) {
    Shared& sh = shared();
    uint32_t* qh = vw.rows ? staged_hi(L, buf) : nullptr;
    uint32_t top = 0;
    for (int k = threadIdx.x; k < L.n; k += kThreads)
#pragma unroll 8
        for (int g = 0; g < L.G; ++g) {
            const float a = A[static_cast<int64_t>(g) * L.N + k];
            if (qh) qh[g * L.rnp + k] = __float_as_uint(a);
            top = max(top, valid_bits(a));
        }
    uint32_t unused = 0xFFFFFFFFu;
    team_min_max(unused, top, tm);
    if (top == 0xFFFFFFFFu) return false;
    const float amax = __uint_as_float(top);
    int e = 0;
    if (amax > 0.0f) frexpf(amax, &e);
    L.e = e;
    L.sh = low_bits(static_cast<int64_t>(L.G / L.D) << kFixedBits);
    L.A = A;
    if (qh) {
        uint16_t* ql = staged_lo(L, buf, vw.rows);
        for (int g = 0; g < L.G; ++g)
            for (int k = threadIdx.x; k < L.n; k += kThreads) {
                const int i = g * L.rnp + k;
                uint32_t h, lo;
                quantize_split(__uint_as_float(qh[i]), e, h, lo);
                qh[i] = h;
                ql[i] = static_cast<uint16_t>(lo);
            }
        L.qh = qh;
        L.ql = ql;
    }
    __syncthreads();
    return true;
}

// ------------------------------------------------------------------ kernel --

template <int DT, bool SM>
__global__ void __launch_bounds__(kThreads, 1)
search_kernel(const float* __restrict__ A_all, int G, int N, int iters, int32_t* __restrict__ head_out,
              int32_t* __restrict__ nu_out, int64_t* __restrict__ score_q_out, double* __restrict__ score_out,
              int32_t* __restrict__ iters_out, int* __restrict__ status_out, int* __restrict__ ws_status,
              uint8_t* __restrict__ gbuf, size_t per_layer, View vw) {
    Shared& sh = shared();
    Team tm = make_team();
    const int layer = blockIdx.x / tm.cl;
    uint8_t* buf = slice_buf<SM>(gbuf, layer, per_layer, vw, DT, tm);
    Layer L;
    layer_view(L, G, N, DT, buf, vw, tm);
    init_shared();
    if (!layer_prologue(L, tm, A_all + static_cast<int64_t>(layer) * G * N + L.k0, buf, vw)) {
        if (threadIdx.x == 0 && tm.rank == 0) {
            status_out[layer] = DTP_ERR_ARG;
            atomicMin(ws_status, static_cast<int>(DTP_ERR_ARG));
        }
        team_sync(tm);
        return;
    }
    if (threadIdx.x < G) sh.h[threadIdx.x] = (threadIdx.x * DT) / G;
    if (threadIdx.x == 0) sh.Jprev = -1;
    __syncthreads();
    if (threadIdx.x < 32) list_heads(sh.h, sh.glist, G, G / DT);
    __syncthreads();

    const Layer S = gains_of_slice(L, vw, tm);
    Team own = make_own(tm);
    int done = 0;
    int64_t total = 0;
    for (int it = 0; it < iters; ++it) {
        build_gain<DT, SM>(S, false, false);
        team_neuron_step<DT, SM>(L, vw, tm, own);
        if (sh.status != DTP_OK) break;
        column_sums<DT, SM>(L, S.nu, tm, G);
        team_sum_i64(G * DT, tm);
        if (it == 0)
            for (int j = 0; j < G * DT; ++j) total += sh.B[j];
        choose_partition<DT>(G);
        done = it + 1;
        const bool stop = sh.J <= sh.Jprev;
        __syncthreads();
        if (threadIdx.x == 0) sh.Jprev = sh.J;
        __syncthreads();
        if (stop) break;
    }
    __syncthreads();
    if (sh.status == DTP_OK)
        for (int k = threadIdx.x; k < L.n; k += kThreads) nu_out[static_cast<int64_t>(layer) * N + L.k0 + k] = S.nu[k];
    team_sync(tm);                     // no block leaves while a peer may still read its shared memory
    if (tm.rank != 0) return;
    if (sh.status != DTP_OK) {
        if (threadIdx.x == 0) {
            status_out[layer] = sh.status;
            atomicMin(ws_status, sh.status);
        }
        return;
    }
    if (threadIdx.x < G) head_out[static_cast<int64_t>(layer) * G + threadIdx.x] = sh.h[threadIdx.x];
    if (threadIdx.x == 0) {
        score_q_out[layer] = sh.J;
        score_out[layer] = total > 0 ? static_cast<double>(sh.J) / static_cast<double>(total) : 0.0;
        iters_out[layer] = done;
        status_out[layer] = DTP_OK;
    }
}

// ------------------------------------------------ global optimum (one layer) --
//
// J of one layer is unchanged when the device labels of h and nu are permuted
// together, so its maximum is the best exact neuron step over the UNLABELLED
// balanced head partitions, G!/((G/D)!^D D!) of them.  Each is taken in its
// canonical labelling (a label first appears after every smaller one), in
// lexicographic order; one team runs the exact neuron step of one (layer,
// partition) item, and a second kernel takes, per layer, the first partition
// with the largest value and recomputes its assignment.

__host__ __device__ inline uint64_t fact_u64(int n) {
    uint64_t f = 1;
    for (int i = 2; i <= n; ++i) f *= static_cast<uint64_t>(i);
    return f;
}

// Completions of a canonical prefix: r heads left, `used` labelled blocks holding the 8-bit counts cnt,
// D - used blocks not yet opened (cap places each, opened in order):
// r! / (prod (cap - cnt)! * cap!^(D-used) * (D-used)!).  r <= 16.
__device__ inline uint64_t rgs_completions(int r, uint64_t cnt, int used, int D, int cap) {
    uint64_t n = fact_u64(r);
    for (int l = 0; l < used; ++l) n /= fact_u64(cap - static_cast<int>((cnt >> (8 * l)) & 255u));
    const int u = D - used;
    const uint64_t fc = fact_u64(cap);
    for (int i = 0; i < u; ++i) n /= fc;
    return n / fact_u64(u);
}

// The idx-th canonical balanced labelling in lexicographic order.
__device__ inline bool unrank_canonical(uint64_t idx, int G, int D, int* h) {
    const int cap = G / D;
    uint64_t cnt = 0;                  // heads placed per block, 8 bits each
    int used = 0;
    for (int k = 0; k < G; ++k) {
        bool placed = false;
        for (int l = 0; l <= used && l < D; ++l) {
            if (static_cast<int>((cnt >> (8 * l)) & 255u) == cap) continue;
            const uint64_t cnt2 = cnt + (uint64_t(1) << (8 * l));
            const int used2 = l == used ? used + 1 : used;
            const uint64_t c = rgs_completions(G - k - 1, cnt2, used2, D, cap);
            if (idx < c) {
                h[k] = l;
                cnt = cnt2;
                used = used2;
                placed = true;
                break;
            }
            idx -= c;
        }
        if (!placed) return false;
    }
    return true;
}

int64_t unlabelled_count(int G, int D);

// The value of the assignment (labels true) or the sum of all gains, after a neuron step; on gathered
// gains only block 0 knows it.
template <int DT, bool SM>
__device__ int64_t sum_gains(const Layer& L, bool labels, Team& tm) {
    Shared& sh = shared();
    int64_t part = 0;
    for (int k = threadIdx.x; k < L.n; k += kThreads) {
        if (labels) part += gain_at<SM>(L, nu_of<SM>(L)[k], k);
        else
            for (int l = 0; l < DT; ++l) part += gain_at<SM>(L, l, k);
    }
    part = block_sum_i64(part);
    if (threadIdx.x == 0) sh.xl[tm.lph][0] = part;
    team_sum_i64(1, tm);
    const int64_t v = sh.B[0];
    __syncthreads();
    return v;
}
template <int DT, bool SM>
__device__ int64_t team_sum_gains(const Layer& L, const View& vw, bool labels, Team& tm, Team& own) {
    Shared& sh = shared();
    if (!vw.gathered) return sum_gains<DT, SM>(L, labels, tm);
    return tm.rank == 0 ? sum_gains<DT, SM>(whole_layer(L), labels, own) : 0;
}

// The canonical partition pidx into sh.h and sh.glist.  False: no such partition.
static __device__ bool set_partition(int64_t pidx, int G, int D) {
    Shared& sh = shared();
    __syncthreads();
    if (threadIdx.x == 0) sh.flag = unrank_canonical(static_cast<uint64_t>(pidx), G, D, sh.h);
    __syncthreads();
    const bool ok = sh.flag != 0;
    if (ok && threadIdx.x < 32) list_heads(sh.h, sh.glist, G, G / D);
    __syncthreads();
    return ok;
}

template <int DT, bool SM>
__global__ void __launch_bounds__(kThreads, 1)
global_items_kernel(const float* __restrict__ A_all, int layers, int G, int N, int64_t n_unl,
                    int64_t* __restrict__ values, int* __restrict__ ws_status, uint8_t* __restrict__ gbuf,
                    size_t per_team, View vw) {
    Shared& sh = shared();
    Team tm = make_team();
    const int64_t team = blockIdx.x / tm.cl, teams = gridDim.x / tm.cl;
    uint8_t* buf = slice_buf<SM>(gbuf, team, per_team, vw, DT, tm);
    const int64_t items = static_cast<int64_t>(layers) * n_unl;
    Team own = make_own(tm);
    init_shared();
    __syncthreads();
    for (int64_t item = team; item < items; item += teams) {
        const int layer = static_cast<int>(item / n_unl);
        const int64_t pidx = item - static_cast<int64_t>(layer) * n_unl;
        Layer L;
        layer_view(L, G, N, DT, buf, vw, tm);
        if (threadIdx.x == 0) sh.status = DTP_OK;
        if (threadIdx.x < DMAX) sh.pi[threadIdx.x] = 0;
        if (!set_partition(pidx, G, DT)) {
            if (threadIdx.x == 0 && tm.rank == 0) {
                values[item] = -1;
                atomicMin(ws_status, static_cast<int>(DTP_ERR_NOT_CONVERGED));
            }
            continue;
        }
        if (!layer_prologue(L, tm, A_all + static_cast<int64_t>(layer) * G * N + L.k0, buf, vw)) {
            if (threadIdx.x == 0 && tm.rank == 0) {
                values[item] = -1;
                atomicMin(ws_status, static_cast<int>(DTP_ERR_ARG));
            }
            continue;
        }
        build_gain<DT, SM>(gains_of_slice(L, vw, tm), false, false);
        team_neuron_step<DT, SM>(L, vw, tm, own);
        if (sh.status != DTP_OK) {
            if (threadIdx.x == 0 && tm.rank == 0) {
                values[item] = -1;
                atomicMin(ws_status, sh.status);
            }
            team_sync(tm);             // the peers have read block 0's status: the next item resets it
            continue;
        }
        const int64_t v = team_sum_gains<DT, SM>(L, vw, true, tm, own);
        if (threadIdx.x == 0 && tm.rank == 0) values[item] = v;
        team_sync(tm);                 // block 0's gains are free for the next item
    }
    team_sync(tm);                     // no block leaves while a peer may still read its shared memory
}

// (score, index) with the larger score, then the smaller index.
__device__ __forceinline__ void better(int64_t& s, int& i, int64_t s2, int i2) {
    if (s2 > s || (s2 == s && i2 < i)) s = s2, i = i2;
}

template <int DT, bool SM>
__global__ void __launch_bounds__(kThreads, 1)
global_pick_kernel(const float* __restrict__ A_all, int G, int N, int64_t n_unl, const int64_t* __restrict__ values,
                   int32_t* __restrict__ head_out, int32_t* __restrict__ nu_out, int64_t* __restrict__ score_q_out,
                   double* __restrict__ score_out, int* __restrict__ ws_status, uint8_t* __restrict__ gbuf,
                   size_t per_team, View vw) {
    Shared& sh = shared();
    Team tm = make_team();
    const int layer = blockIdx.x / tm.cl;
    const int64_t* vals = values + static_cast<int64_t>(layer) * n_unl;
    // first index of the largest value (values < 0 mark failed items); every block for itself
    int64_t best = -1;
    int best_idx = 0x7FFFFFFF;
    for (int64_t i = threadIdx.x; i < n_unl; i += kThreads) better(best, best_idx, vals[i], static_cast<int>(i));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const int64_t s2 = __shfl_xor_sync(0xFFFFFFFFu, best, o);
        const int i2 = __shfl_xor_sync(0xFFFFFFFFu, best_idx, o);
        better(best, best_idx, s2, i2);
    }
    if (lane == 0) sh.red_i64[warp] = best, sh.red_int[warp] = best_idx;
    init_shared();
    __syncthreads();
    if (warp == 0) {
        int64_t b = lane < kWarps ? sh.red_i64[lane] : -1;
        int bi = lane < kWarps ? sh.red_int[lane] : 0x7FFFFFFF;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const int64_t s2 = __shfl_xor_sync(0xFFFFFFFFu, b, o);
            const int i2 = __shfl_xor_sync(0xFFFFFFFFu, bi, o);
            better(b, bi, s2, i2);
        }
        if (lane == 0) {
            sh.Jprev = b;
            sh.best_idx = bi;
        }
    }
    __syncthreads();
    if (sh.Jprev < 0) {                                   // every item failed: already reported
        if (threadIdx.x == 0) atomicMin(ws_status, static_cast<int>(DTP_ERR_ARG));
        return;
    }
    uint8_t* buf = slice_buf<SM>(gbuf, layer, per_team, vw, DT, tm);
    Layer L;
    layer_view(L, G, N, DT, buf, vw, tm);
    set_partition(sh.best_idx, G, DT);
    layer_prologue(L, tm, A_all + static_cast<int64_t>(layer) * G * N + L.k0, buf, vw);
    const Layer S = gains_of_slice(L, vw, tm);
    Team own = make_own(tm);
    build_gain<DT, SM>(S, false, false);
    team_neuron_step<DT, SM>(L, vw, tm, own);
    if (sh.status != DTP_OK) {
        if (threadIdx.x == 0) atomicMin(ws_status, sh.status);
        team_sync(tm);
        return;
    }
    const int64_t v = team_sum_gains<DT, SM>(L, vw, true, tm, own);
    const int64_t total = team_sum_gains<DT, SM>(L, vw, false, tm, own);
    for (int k = threadIdx.x; k < L.n; k += kThreads) nu_out[static_cast<int64_t>(layer) * N + L.k0 + k] = S.nu[k];
    team_sync(tm);
    if (tm.rank != 0) return;
    if (threadIdx.x < G) head_out[static_cast<int64_t>(layer) * G + threadIdx.x] = sh.h[threadIdx.x];
    if (threadIdx.x == 0) {
        score_q_out[layer] = v;
        score_out[layer] = total > 0 ? static_cast<double>(v) / static_cast<double>(total) : 0.0;
        if (v != sh.Jprev) atomicMin(ws_status, static_cast<int>(DTP_ERR_NOT_CONVERGED));   // must recompute equal
    }
}

// ------------------------------------------------------- whole-model search --
//
// Eq. objective with both sums: J = sum_i up_i + sum_{i<L-1} down_i, each matrix
// in its exact unit-mass form n = floor(q 2^43 / total), q = floor(S 2^(40-e)).
// One iteration = every layer's neuron step given all head partitions (gain from
// h_i for the up edge and h_{i+1} for the down edge), then every layer's head
// step given all neuron assignments (column sums over nu_i for the up edge and
// nu_{i-1} for the down edge), then the score.  Each step maximises J exactly
// given the other block, so layers run in parallel, one team each.  A device
// flag stops later iterations after the first one (after the first) without a
// strict increase, so the host never waits.
//
// One launch runs all iterations where every team can be resident (a cooperative launch: the teams wait
// for each iteration's score; the scores' matrices stay in shared memory), else one iteration each.  A
// layer's team also sums the columns that its new
// assignment contributes to its own head step (up edge) and to the next layer's
// (down edge); whichever of the two teams that feed a head step arrives second
// (a counter per layer) runs it, and the last head step adds the score.
//
// Ablations (Sec. 3 "Optimiser", Table 4): per-layer flags freeze a layer's
// heads or neurons at the contiguous start, and `minimize` minimises J.  A
// minimising step maximises R - gain with R the per-neuron (per-head) sum of
// the gains over devices: every neuron (head) sits on exactly one device, so
// the offset shifts all assignments' totals equally and leaves the set of
// optimal assignments (hence the canonical one) unchanged, while keeping every
// gain non-negative and below 2^44 as the exact steps require.

constexpr int kNormBits = 43;   // gains (one up + one down matrix) stay below 2^44
constexpr int kNormPreBits = 40;

struct ChainState {
    int done;      // written only by the last block of an iteration (or before the first)
    int iters;
    int failed;    // a team of this iteration reported an error
    int heads;     // head steps of this iteration finished
    int64_t prev;
    int epoch;     // iterations scored, published after everything above and the head partitions
    int beat;      // counts on while some team is in a long repair
};

struct ChainArgs {
    int Lyr, G, N;
    const int64_t* nbuf;
    const int64_t* top;     // [2 Lyr - 1]: each matrix's largest entry
    int32_t* head;
    int32_t* nu;
    int64_t* prices;        // [Lyr][DMAX]
    int64_t* up_sums;       // [Lyr][GMAX * DMAX]: columns of layer i's up edge over nu_i
    int64_t* down_sums;     // [Lyr][GMAX * DMAX]: columns of its down edge over nu_i
    int* arrived;           // [Lyr]: teams that have fed layer i's head step
    int64_t* layer_score;   // [Lyr]
    ChainState* st;
    int* ws_status;
    uint8_t* gbuf;
    size_t per_layer;
    View vw;
    const uint8_t* move_neurons;
    const uint8_t* move_heads;
    int minimize;
    int64_t* J_q;
    double* J;
    int32_t* iters_done;
    int rounds;             // iterations of this launch; above 1 every team is resident
};

// Head step of layer i from the sums of layers i and i - 1; the last one of the iteration adds the score.
template <int DT, bool SM>
__device__ void chain_head_step(const ChainArgs& c, int i) {
    Shared& sh = shared();
    const int G = c.G, tid = threadIdx.x;
    __shared__ int last;
    // another team may set the flag at any time: one thread reads it, and the whole block takes one side
    const bool failed = __syncthreads_or(tid == 0 && *reinterpret_cast<volatile int*>(&c.st->failed) != 0);
    if (!failed) {
        if (tid < G * DT) {
            int64_t b = __ldcg(c.up_sums + static_cast<int64_t>(i) * GMAX * DMAX + tid);
            if (i > 0) b += __ldcg(c.down_sums + static_cast<int64_t>(i - 1) * GMAX * DMAX + tid);
            sh.B[tid] = b;
        }
        __syncthreads();
        if (c.move_heads && !c.move_heads[i]) {            // frozen: score the current (contiguous) partition
            if (tid == 0) {
                int64_t sc = 0;
                for (int g = 0; g < G; ++g) sc += sh.B[g * DT + c.head[i * G + g]];
                c.layer_score[i] = c.minimize ? -sc : sc;
            }
        } else {
            int64_t R = 0;                                  // sum_g R_g, held by thread 0
            if (c.minimize) {
                if (tid < G) {
                    int64_t r = 0;
#pragma unroll
                    for (int l = 0; l < DT; ++l) r += sh.B[tid * DT + l];
#pragma unroll
                    for (int l = 0; l < DT; ++l) sh.B[tid * DT + l] = r - sh.B[tid * DT + l];
                    sh.red_i64[tid] = r;
                }
                __syncthreads();
                if (tid == 0)
                    for (int g = 0; g < G; ++g) R += sh.red_i64[g];
            }
            choose_partition<DT>(G);
            if (tid < G) c.head[i * G + tid] = sh.h[tid];
            if (tid == 0) c.layer_score[i] = sh.J - R;      // minimising: -(J of this layer) = J' - sum_g R_g
        }
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) last = atomicAdd(&c.st->heads, 1) == c.Lyr - 1;
    __syncthreads();
    if (!last) return;
    // every team has arrived and every head step is done
    __threadfence();
    int64_t part = 0;
    for (int j = tid; j < c.Lyr; j += kThreads) {
        part += __ldcg(c.layer_score + j);
        c.arrived[j] = 0;
    }
    __threadfence();
    const int64_t total = block_sum_i64(part);
    if (tid == 0) {
        ChainState* st = c.st;
        st->heads = 0;
        if (*reinterpret_cast<volatile int*>(&st->failed)) {
            st->done = 1;
        } else {
            st->iters += 1;
            *c.iters_done = st->iters;
            const int64_t jq = c.minimize ? -total : total;
            *c.J_q = jq;
            *c.J = ldexp(static_cast<double>(jq), -kNormBits);
            if (total <= st->prev) st->done = 1;
            else st->prev = total;
        }
        __threadfence();
        atomicAdd(&st->epoch, 1);
    }
    __syncthreads();
}

// Thread 0 of a team: waits until iteration `epoch` (counted from this call's start) has been scored.
// Gives up after kWaitLimitNs without a sign of progress.  True: another iteration follows.
__device__ __forceinline__ bool wait_scored(const ChainArgs& c, int epoch) {
    auto load = [](const int* p) {
        int v;
        asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
        return v;
    };
    uint64_t t0 = globaltimer_ns();
    int beat = load(&c.st->beat);
    while (load(&c.st->epoch) < epoch) {
        __nanosleep(100);
        const int now = load(&c.st->beat);
        if (now != beat) {
            beat = now;
            t0 = globaltimer_ns();
        } else if (globaltimer_ns() - t0 > kWaitLimitNs) {
            atomicMin(c.ws_status, static_cast<int>(DTP_ERR_NOT_CONVERGED));
            return false;
        }
    }
    return load(&c.st->done) == 0;
}

template <int DT, bool SM>
__global__ void __launch_bounds__(kThreads, 1) chain_iteration_kernel(const ChainArgs c) {
    Shared& sh = shared();
    __shared__ int second[2];
    __shared__ int go;
    // between launches done is written only after every block of an iteration has read it, so a team's
    // blocks agree
    if (*reinterpret_cast<volatile int*>(&c.st->done)) return;
    Team tm = make_team();
    const int i = blockIdx.x / tm.cl;
    const int G = c.G, N = c.N, tid = threadIdx.x;
    const int64_t GN = static_cast<int64_t>(G) * N;
    uint8_t* buf = slice_buf<SM>(c.gbuf, i, c.per_layer, c.vw, DT, tm);
    Layer L;
    layer_view(L, G, N, DT, buf, c.vw, tm);
    init_shared();
    const bool has_down = i + 1 < c.Lyr;
    const bool move = !c.move_neurons || c.move_neurons[i];
    const int rows = has_down ? 2 * G : G;
    // a gain is a sum over one device's heads, minimising over all others'
    L.sh = low_bits((c.top[i] + (has_down ? c.top[c.Lyr + i] : 0)) * (c.minimize ? G : G / DT));
    team_sync(tm);                     // every block of the team has started: its shared memory may be written
    if (tid == 0) sh.beat = &c.st->beat;
    if (tid < DMAX) sh.pi[tid] = c.prices[i * DMAX + tid];
    L.nU = c.nbuf + i * GN + L.k0;
    L.nD = has_down ? c.nbuf + (c.Lyr + i) * GN + L.k0 : nullptr;
    if (c.vw.rows) {
        uint32_t* qh = staged_hi(L, buf);
        uint16_t* ql = staged_lo(L, buf, c.vw.rows);
        for (int k = tid; k < L.n; k += kThreads)
#pragma unroll 8
            for (int r = 0; r < rows; ++r) {
                const int64_t v = (r < G ? L.nU + static_cast<int64_t>(r) * N
                                         : L.nD + static_cast<int64_t>(r - G) * N)[k];
                qh[r * L.rnp + k] = static_cast<uint32_t>(v >> kLoBits);
                ql[r * L.rnp + k] = static_cast<uint16_t>(v & ((1 << kLoBits) - 1));
            }
        L.qh = qh;
        L.ql = ql;
    }
    const Layer S = gains_of_slice(L, c.vw, tm);
    Team own = make_own(tm);
    for (int round = 0; round < c.rounds; ++round) {
        __syncthreads();
        if (tid < G) {
            sh.h[tid] = __ldcg(c.head + i * G + tid);
            sh.hn[tid] = has_down ? __ldcg(c.head + (i + 1) * G + tid) : -1;
        }
        __syncthreads();
        if (tid < 32) list_heads(sh.h, sh.glist, G, G / DT);
        else if (tid < 64 && has_down) list_heads(sh.hn, sh.gnlist, G, G / DT);
        __syncthreads();
        if (move) {
            build_gain<DT, SM>(S, has_down, c.minimize != 0);
            team_neuron_step<DT, SM>(L, c.vw, tm, own);
            if (sh.status == DTP_OK)
                for (int k = tid; k < L.n; k += kThreads) c.nu[static_cast<int64_t>(i) * N + L.k0 + k] = S.nu[k];
        } else {                                            // frozen: nu_i stays contiguous
            for (int k = tid; k < L.n; k += kThreads)
                S.nu[k] = static_cast<uint8_t>((static_cast<int64_t>(L.k0 + k) * DT) / N);
            __syncthreads();
        }
        const bool ok = sh.status == DTP_OK;
        if (ok) {
            column_sums<DT, SM>(L, S.nu, tm, rows);
            team_sum_i64(rows * DT, tm);
            if (tm.rank == 0 && tid < rows * DT) {
                const int r = tid / DT, l = tid % DT;
                int64_t* to = r < G ? c.up_sums : c.down_sums;
                to[static_cast<int64_t>(i) * GMAX * DMAX + (r < G ? r : r - G) * DT + l] = sh.B[tid];
            }
        }
        if (tm.rank == 0) {
            if (tid == 0 && !ok) {
                atomicMin(c.ws_status, sh.status);
                atomicExch(&c.st->failed, 1);
            }
            __threadfence();
            __syncthreads();
            if (tid == 0) {
                second[0] = atomicAdd(&c.arrived[i], 1) == (i > 0 ? 1 : 0);
                second[1] = has_down && atomicAdd(&c.arrived[i + 1], 1) == 1;
            }
            __syncthreads();
            __threadfence();
            if (second[0]) chain_head_step<DT, SM>(c, i);
            if (second[1]) chain_head_step<DT, SM>(c, i + 1);
            if (tid == 0) go = round + 1 < c.rounds && wait_scored(c, round + 1);
        }
        team_sync(tm);                 // also: no block goes on while a peer may still read its shared memory
        const int more = *at_rank(&go, 0);
        team_sync(tm);
        if (!more) break;
    }
    if (tm.rank == 0 && tid < DMAX) c.prices[i * DMAX + tid] = sh.pi[tid];
}

// The kernels for one device count, on layers in shared memory or (larger than 16 blocks can hold) in
// the workspace: two translation units, compiled side by side.
struct Kernels {
    void (*search)(const float*, int, int, int, int32_t*, int32_t*, int64_t*, double*, int32_t*, int*, int*, uint8_t*,
                   size_t, View);
    void (*items)(const float*, int, int, int, int64_t, int64_t*, int*, uint8_t*, size_t, View);
    void (*pick)(const float*, int, int, int64_t, const int64_t*, int32_t*, int32_t*, int64_t*, double*, int*,
                 uint8_t*, size_t, View);
    void (*chain)(ChainArgs);
};
Kernels kernels_in_shared(int D);
Kernels kernels_in_global(int D);

template <bool SM>
Kernels kernels_for(int D) {
#define DTP_KERNELS(DV) \
    case DV: return {search_kernel<DV, SM>, global_items_kernel<DV, SM>, global_pick_kernel<DV, SM>, chain_iteration_kernel<DV, SM>};
    switch (D) {
        DTP_KERNELS(2)
        DTP_KERNELS(3)
        DTP_KERNELS(4)
        DTP_KERNELS(5)
        DTP_KERNELS(6)
        DTP_KERNELS(7)
        DTP_KERNELS(8)
        default: return {};
    }
#undef DTP_KERNELS
}

}  // namespace search
}  // namespace dtp
