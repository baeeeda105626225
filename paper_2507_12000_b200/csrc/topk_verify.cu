// Truncated-support (top-k) verification round for sm_100a: the sampler of the paper's
// experiments (Section 4) applied to Algorithm 2.
//
//   topk_select_kernel  one CTA per run of one target row (16 to 64 KB of logits): the run's k best entries.
//                       The threads' maxima over the first tile, taken in 32 groups, give a threshold: the
//                       k-th largest group maximum is a lower bound on the run's k-th largest logit
//                       (k <= 32).  Vectors that reach it are taken apart, their entries that reach it become
//                       candidates - a dozen per tile - and the candidates are ranked by counting.
//   topk_fold_kernel    one CTA per sequence, a warp per row: merges the lists of the row's runs, turns the k
//                       logits into probabilities in float64, evaluates the acceptance test; the first
//                       rejection gives n, and the warp that holds row n writes its pairs.
//
// A key is 64 bits: the logit mapped to an unsigned integer that sorts like the float (with -0 folded
// into +0), then the complemented index - larger key = earlier in the order (logit descending, index
// ascending), and all keys of a row are distinct.  Input that defeats the threshold (masks, runs of
// equal or of ascending logits) overflows the candidate buffer; the CTA then goes over its run again with a bound from the
// whole run, ties in index order, and where even that lets too many through it selects step by step, at most
// one entry per thread and step, cutting the buffer back to its k best whenever it fills: slow, never wrong.
// The end of a kernel is the only synchronisation; nothing in the workspace has to be cleared.
//
// Device kernel: one warp per sequence, everything in registers and shuffles, sums strictly
// sequential in float64 so that the draw is reproducible bit for bit.
#include "topk_verify.h"

#include <math.h>

#include "dssd_device.cuh"
#include "launch.h"

namespace dssd {
namespace {

// Tiles per CTA of the selection kernel: one in small launches, so that all SMs share the work; from four
// waves of CTAs on two, from sixteen on four: every run ranks its candidates once.  Measured (us a round,
// 1 / 2 / 4 tiles): B = 256 gamma = 4 V = 151936 bf16 (24 320 tiles) 87.9 / 71.9 / 69.9, B = 1 gamma = 8
// V = 50272 float32 (117) 10.8 / 10.7 / 11.9.
constexpr unsigned long long kSelTwoTiles = 4700, kSelFourTiles = 19000;

constexpr int kSelThreads = 128;
constexpr int kSelLoads = 8;                         // 16-byte loads a thread has in flight
constexpr int kSelTile = kSelThreads * kSelLoads;    // 16-byte vectors of one pass over the CTA (16 KB)
constexpr int kCand = 1024;                          // candidates that a CTA can hold
// The first threshold: the k-th of 32 groups' maxima is tight and cheap for small k (k = 10: about 12 candidates per tile)
// but near its smallest group for large ones (k = 32: 110 candidates, and ranking m of them costs m * m), where a bound
// from all threads' maxima leaves 50.  More than kRefine candidates are cut back once more by the maxima over the whole
// run.  B = 256 gamma = 4 V = 151936 bf16 k = 32: 85 us against 553 without both.
constexpr int kGroupsUpTo = 12;
constexpr int kRefine = 96;
constexpr int kFoldWarps = 16;                       // most warps (rows at a time) of the fold kernel
constexpr int kFoldTurns = 2;                        // most turns; beyond, topk_rows_kernel
constexpr int kMergeCap = 256;                       // keys that a warp ranks when it merges a row's runs
constexpr int kMergeLists = 64;                      // lists that it notes before it looks at their keys
constexpr unsigned long long kBadList = ~0ull;       // every key of a run that held a NaN or +inf
constexpr unsigned kFullMask = 0xffffffffu;

__device__ __forceinline__ float max_nan(float a, float b)
{
    float r;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}

__device__ __forceinline__ uint32_t max_nan_bf16x2(uint32_t a, uint32_t b)
{
    uint32_t r;
    asm("max.NaN.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}

// unsigned integers that sort like the floats they come from (NaN excluded by the callers)
__device__ __forceinline__ uint32_t ord(float f)
{
    uint32_t b = __float_as_uint(f);
    if (b == 0x80000000u) b = 0u;  // -0 and +0 are the same logit
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

__device__ __forceinline__ float unord(uint32_t o)
{
    return __uint_as_float((o & 0x80000000u) ? (o & 0x7fffffffu) : ~o);
}

__device__ __forceinline__ unsigned long long make_key(float f, int idx)
{
    return ((unsigned long long)ord(f) << 32) | (unsigned long long)(~(uint32_t)idx);
}

__device__ __forceinline__ int key_index(unsigned long long key) { return (int)(~(uint32_t)key); }
__device__ __forceinline__ float key_value(unsigned long long key) { return unord((uint32_t)(key >> 32)); }

template <int DT>
struct Vec;
template <>
struct Vec<DSSD_F32> {
    static constexpr int E = 4;
    static constexpr int kEsz = 4;
    __device__ static __forceinline__ uint4 fill() { return make_uint4(0xff800000u, 0xff800000u, 0xff800000u, 0xff800000u); }
    __device__ static __forceinline__ float vmax(const uint4 &v)
    {
        return max_nan(max_nan(__uint_as_float(v.x), __uint_as_float(v.y)),
                       max_nan(__uint_as_float(v.z), __uint_as_float(v.w)));
    }
    __device__ static __forceinline__ float load(const void *row, int64_t i) { return reinterpret_cast<const float *>(row)[i]; }
    // element j of the vector (j < E)
    __device__ static __forceinline__ float elem(const uint4 &v, int j)
    {
        return __uint_as_float(j < 2 ? (j == 0 ? v.x : v.y) : (j == 2 ? v.z : v.w));
    }
};
template <>
struct Vec<DSSD_BF16> {
    static constexpr int E = 8;
    static constexpr int kEsz = 2;
    __device__ static __forceinline__ uint4 fill() { return make_uint4(0xff80ff80u, 0xff80ff80u, 0xff80ff80u, 0xff80ff80u); }
    __device__ static __forceinline__ float vmax(const uint4 &v)
    {
        const uint32_t w = max_nan_bf16x2(max_nan_bf16x2(v.x, v.y), max_nan_bf16x2(v.z, v.w));
        return max_nan(bf16_lo(w), bf16_hi(w));
    }
    __device__ static __forceinline__ float load(const void *row, int64_t i)
    {
        return __uint_as_float((uint32_t)reinterpret_cast<const unsigned short *>(row)[i] << 16);
    }
    __device__ static __forceinline__ float elem(const uint4 &v, int j)
    {
        const uint32_t w = j < 4 ? (j < 2 ? v.x : v.y) : (j < 6 ? v.z : v.w);
        return (j & 1) ? bf16_hi(w) : bf16_lo(w);
    }
};

struct SelectShared {
    unsigned long long key[kCand];
    unsigned long long top[32];
    uint4 grp[kSelThreads / 4];  // thresholds are taken from these maxima: of 32 groups, or of the threads
    uint32_t tau[kSelThreads / 32];
    unsigned count;  // candidates found (more than kCand: some were dropped)
    int bad;         // the run holds a NaN or +inf
};

__device__ __forceinline__ void push(SelectShared &sh, unsigned long long key)
{
    const unsigned at = atomicAdd(&sh.count, 1u);
    if (at < (unsigned)kCand) sh.key[at] = key;
}

// A lower bound on the k-th largest of the threads' values x, each of which is an entry of its own: the smallest over
// the warps of the ceil(k / 4)-th largest in the warp (k <= 32).  Cheaper than the k-th largest itself: the values
// are compared within a warp only, as integers that carry the lane in their last bits.
__device__ __forceinline__ float bound_of_threads(SelectShared &sh, float x, int k)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t mine = (ord(x) & ~31u) | (uint32_t)lane;
    reinterpret_cast<uint32_t *>(sh.grp)[tid] = mine;
    __syncwarp();
    int rank = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const uint4 o = sh.grp[warp * 8 + j];
        rank += (o.x > mine) + (o.y > mine) + (o.z > mine) + (o.w > mine);
    }
    if (rank == (k - 1) / 4) sh.tau[warp] = mine & ~31u;
    __syncthreads();
    uint32_t t = sh.tau[0];
#pragma unroll
    for (int w = 1; w < kSelThreads / 32; ++w) t = min(t, sh.tau[w]);
    return t <= ord(DSSD_NEG_INF) ? DSSD_NEG_INF : unord(t);  // (below -inf there are NaNs)
}

// The k largest of the m keys in sh.key, best first, to sh.top (0 where there are fewer); by the whole CTA.
__device__ __forceinline__ void rank_keys(SelectShared &sh, int m, int k)
{
    const int tid = threadIdx.x;
    if (tid < 32) sh.top[tid] = 0ull;
    __syncthreads();
    for (int i = tid; i < m; i += kSelThreads) {
        const unsigned long long x = sh.key[i];
        int rank = 0;
        for (int j = 0; j < m; ++j) rank += sh.key[j] > x;
        if (rank < k) sh.top[rank] = x;
    }
    __syncthreads();
}

// Drops candidates that cannot be among the k best: the k-th largest of the threads' maxima over the whole run bounds
// the k-th logit much more tightly than the first tile's did, and ranking costs the square of what is left.
__device__ __noinline__ int refine(SelectShared &sh, int m, float top, int k)
{
    const int tid = threadIdx.x;
    const float tau = bound_of_threads(sh, top == top ? top : DSSD_NEG_INF, k);
    unsigned long long held[kCand / kSelThreads];
#pragma unroll
    for (int i = 0; i < kCand / kSelThreads; ++i) {
        held[i] = 0ull;
        if (i * kSelThreads + tid < m) held[i] = sh.key[i * kSelThreads + tid];
    }
    if (tid == 0) sh.count = 0;
    __syncthreads();
    const unsigned long long floor = (unsigned long long)ord(tau) << 32;
#pragma unroll
    for (int i = 0; i < kCand / kSelThreads; ++i)
        if (held[i] != 0ull && held[i] >= floor) sh.key[atomicAdd(&sh.count, 1u)] = held[i];
    __syncthreads();
    return (int)sh.count;
}

// The candidates did not fit: the threshold of the first tile was too low for what came after it, or more entries equal it than a
// CTA can hold (a mask, equal logits).  The threads' maxima over the whole run give a better bound t, this time exactly: at
// least k entries reach it.  Those above t are candidates; where they are fewer than k, the first ones that equal t follow, found
// vector by vector in index order.  Two passes over the run at most, from L2.  B = 256 gamma = 4 V = 32000 bf16,
// nine tenths masked, k = 10: 61 us, entry by entry (select_slowly) 791; ascending rows 267 and 6592.  false: more are above t than fit.
template <int DT>
__device__ __noinline__ bool select_again(SelectShared &sh, const char *rowp, int idx0, int v0, int v1, int e0, int e1, float top, int k)
{
    constexpr int E = Vec<DT>::E;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint4 *src = reinterpret_cast<const uint4 *>(rowp + (size_t)idx0 * Vec<DT>::kEsz);
    const int ev0 = idx0 + v0 * E, ev1 = idx0 + v1 * E;  // the entries in vectors
    const uint32_t mine = ord(top == top ? top : DSSD_NEG_INF);
    int rank = 0;
    for (int j = 0; j < 32; ++j) {
        const uint32_t o = __shfl_sync(kFullMask, mine, j);
        rank += o > mine || (o == mine && j < lane);
    }
    __syncthreads();  // the number of candidates has been read
    if (rank == (k - 1) / 4) sh.tau[warp] = mine;
    if (tid == 0) sh.count = 0;
    __syncthreads();
    uint32_t least = sh.tau[0];
#pragma unroll
    for (int w = 1; w < kSelThreads / 32; ++w) least = min(least, sh.tau[w]);
    const float t = unord(least);
    for (int i = v0 + tid; i < v1; i += kSelThreads) {
        const uint4 v = ld_stream16(src + i);
        if (!(Vec<DT>::vmax(v) > t)) continue;
#pragma unroll
        for (int j = 0; j < E; ++j)
            if (Vec<DT>::elem(v, j) > t) push(sh, make_key(Vec<DT>::elem(v, j), idx0 + i * E + j));
    }
    const int outside = tid < 32 ? e0 + tid : ev1 + tid - 32;  // the entries before and after the vectors: fewer than eight each
    const bool has = tid < 32 ? outside < ev0 : outside < e1;
    const float f = has ? Vec<DT>::load(rowp, outside) : DSSD_NEG_INF;
    if (has && f > t) push(sh, make_key(f, outside));
    __syncthreads();
    const unsigned above = sh.count;
    if (above > (unsigned)kCand) return false;
    int found = 0;  // entries that equal t so far, in index order; the same in all threads
    const int want = k - (int)above;
    auto take = [&](unsigned mask, int first) {  // this thread's: bit j is entry first + j; threads in index order
        unsigned incl = __popc(mask);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned up = __shfl_up_sync(kFullMask, incl, o);
            if (lane >= o) incl += up;
        }
        __syncthreads();
        if (lane == 31) sh.tau[warp] = incl;
        __syncthreads();
        int at = found + (int)incl - __popc(mask);
#pragma unroll
        for (int w = 0; w < kSelThreads / 32; ++w) {
            if (w < warp) at += (int)sh.tau[w];
            found += (int)sh.tau[w];
        }
        for (; mask && at < want; mask &= mask - 1u, ++at) sh.key[above + at] = make_key(t, first + __ffs(mask) - 1);
    };
    if (want > 0) take(tid < 32 && has && f == t ? 1u : 0u, outside);
    for (int base = v0; base < v1 && found < want; base += kSelThreads) {
        unsigned mask = 0;
        if (base + tid < v1) {
            const uint4 v = ld_stream16(src + base + tid);
#pragma unroll
            for (int j = 0; j < E; ++j) mask |= Vec<DT>::elem(v, j) == t ? 1u << j : 0u;
        }
        take(mask, idx0 + (base + tid) * E);
    }
    if (found < want) take(tid >= 32 && has && f == t ? 1u : 0u, outside);
    __syncthreads();
    if (tid == 0) sh.count = above + (unsigned)(want <= 0 ? 0 : found < want ? found : want);
    __syncthreads();
    return true;
}

// The run again, where that did not do either: entry by entry, at most one per thread and step.
template <int DT>
__device__ __noinline__ void select_slowly(SelectShared &sh, const char *rowp, int e0, int e1, int k)
{
    const int tid = threadIdx.x;
    unsigned long long floor = 0ull;  // keys up to here are not among the k best
    __syncthreads();
    if (tid == 0) sh.count = 0;
    __syncthreads();
    for (int first = e0; first < e1; first += kSelThreads) {
        const int e = first + tid;
        if (e < e1) {
            const float f = Vec<DT>::load(rowp, e);
            if (!(f < INFINITY)) sh.bad = 1;
            const unsigned long long key = make_key(f, e);
            if (key > floor) push(sh, key);
        }
        __syncthreads();
        if (sh.count > (unsigned)(kCand - kSelThreads)) {
            rank_keys(sh, (int)sh.count, k);
            floor = sh.top[k - 1];
            if (tid < k) sh.key[tid] = sh.top[tid];
            if (tid == 0) sh.count = (unsigned)k;
        }
        __syncthreads();
    }
}

// Bound by HBM: B = 256 gamma = 4 V = 151936 bf16 (389 MB) in 61.5 us, 6.3 TB/s, k = 10; the persistent kernel it
// replaces (a ring per CTA, one selection warp that inserted candidates one by one, rows judged in the
// same warp) took 79 us for this and the fold together, and 18.8 us at B = 1 gamma = 8 V = 50272 where
// both kernels now take 7.7.  Ten CTAs per SM (48 registers); eight 61.9, twelve 65 us (spills).
// One CTA per (row, run).  A row's vectors start at
// its first 16-byte boundary; the entries before it belong to the first run, those after the last whole
// vector to the last run.
template <int DT>
__global__ void __launch_bounds__(kSelThreads, 10) topk_select_kernel(const __grid_constant__ TopkParams P)
{
    constexpr int E = Vec<DT>::E, kEsz = Vec<DT>::kEsz;
    __shared__ SelectShared sh;
    const int tid = threadIdx.x, lane = tid & 31, k = P.k;
    const unsigned row = blockIdx.x / (unsigned)P.runs;
    const int run = (int)(blockIdx.x - row * (unsigned)P.runs);
    const char *rowp = static_cast<const char *>(P.logits) + (size_t)row * (size_t)P.row_stride * kEsz;
    const long long rowbytes = (long long)P.V * kEsz;
    int head = (int)((16u - (unsigned)(reinterpret_cast<uintptr_t>(rowp) & 15u)) & 15u);
    if (head > rowbytes) head = (int)rowbytes;
    const int nvec = (int)((rowbytes - head) >> 4);
    const int v0 = min(nvec, run * P.run_vecs), v1 = run + 1 == P.runs ? nvec : min(nvec, v0 + P.run_vecs);
    const uint4 *src = reinterpret_cast<const uint4 *>(rowp + head);
    const int idx0 = head / kEsz;  // index of the first vector's first entry
    if (tid == 0) {
        sh.count = 0;
        sh.bad = 0;
    }
    pdl_wait();
    pdl_trigger();
    // the entries outside the vectors: at most one per thread
    int extra_at = -1;
    if (run == 0 && tid < idx0) extra_at = tid;
    if (run + 1 == P.runs && tid >= 32) {
        const int e = idx0 + nvec * E + tid - 32;
        if (e < P.V) extra_at = e;
    }
    float extra = DSSD_NEG_INF;
    if (extra_at >= 0) extra = Vec<DT>::load(rowp, extra_at);
    float tau = DSSD_NEG_INF;
    float top = extra;  // NaN-propagating maximum of all that this thread has seen
    bool first = true;
    for (int base = v0; base < v1 || first; base += kSelTile) {
        float vm[kSelLoads];
        {
            uint4 v[kSelLoads];
#pragma unroll
            for (int u = 0; u < kSelLoads; ++u) {
                v[u] = Vec<DT>::fill();
                if (base + tid + u * kSelThreads < v1) v[u] = ld_stream16(src + base + tid + u * kSelThreads);
            }
#pragma unroll
            for (int u = 0; u < kSelLoads; ++u) vm[u] = Vec<DT>::vmax(v[u]);
        }
        float tm = vm[0];
#pragma unroll
        for (int u = 1; u < kSelLoads; ++u) tm = max_nan(tm, vm[u]);
        top = max_nan(top, tm);
        unsigned hot = 0;
        if (first) {
            const float x = tm == tm ? tm : DSSD_NEG_INF;
            if (k > kGroupsUpTo) {
                tau = bound_of_threads(sh, x, k);
            } else {
                // 32 groups of four threads: each group's maximum is one distinct entry
                float g = fmaxf(x, __shfl_xor_sync(kFullMask, x, 1));
                g = fmaxf(g, __shfl_xor_sync(kFullMask, g, 2));
                float *grp = reinterpret_cast<float *>(sh.grp);
                if ((tid & 3) == 0) grp[tid >> 2] = g;
                __syncthreads();
                const float mine = grp[lane];
                int rank = 0;
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                    const float o = grp[j];
                    rank += (o > mine) || (o == mine && j < lane);
                }
                const unsigned hit = __ballot_sync(kFullMask, rank == k - 1);
                tau = __shfl_sync(kFullMask, mine, __ffs(hit) - 1);
            }
            if (extra_at >= 0 && extra >= tau) push(sh, make_key(extra, extra_at));
#pragma unroll
            for (int u = 0; u < kSelLoads; ++u) hot |= vm[u] >= tau && base + tid + u * kSelThreads < v1 ? 1u << u : 0u;
        } else {
            // k entries of the first tile reach tau and come before every entry that equals it here
#pragma unroll
            for (int u = 0; u < kSelLoads; ++u) hot |= vm[u] > tau ? 1u << u : 0u;
        }
        while (hot) {
            const int at = base + tid + (__ffs(hot) - 1) * kSelThreads;
            hot &= hot - 1u;
            const uint4 v = ld_stream16(src + at);  // from L2: the registers have moved on
            unsigned mask = 0;
#pragma unroll
            for (int j = 0; j < E; ++j) {
                const float f = Vec<DT>::elem(v, j);
                mask |= (first ? f >= tau : f > tau) ? 1u << j : 0u;
            }
            unsigned to = atomicAdd(&sh.count, (unsigned)__popc(mask));
#pragma unroll
            for (int j = 0; j < E; ++j) {
                if (!(mask >> j & 1u)) continue;
                if (to < (unsigned)kCand) sh.key[to] = make_key(Vec<DT>::elem(v, j), idx0 + at * E + j);
                ++to;
            }
        }
        first = false;
    }
    if (!(top < INFINITY)) sh.bad = 1;
    __syncthreads();
    int m = (int)sh.count;
    if (m > kCand) {
        const int e0 = run == 0 ? 0 : idx0 + v0 * E, e1 = run + 1 == P.runs ? P.V : idx0 + v1 * E;
        if (!select_again<DT>(sh, rowp, idx0, v0, v1, e0, e1, top, k)) select_slowly<DT>(sh, rowp, e0, e1, k);
        m = (int)sh.count;
    }
    if (m > kRefine) m = refine(sh, m, top, k);
    rank_keys(sh, m, k);
    if (tid < k) {
        unsigned long long key = sh.top[tid];
        if (sh.bad) key = kBadList;
        P.lists[(size_t)blockIdx.x * k + tid] = key;
    }
}

// The sum of a row's weights: up to this k one after the other, beyond by halves, a chain of five additions with two shuffles each (the
// edge call at B = 1 gamma = 8 V = 50272 float32 k = 10 7.8 us; 8.1 with this sum one after the other and with the other chains below as they were).
constexpr int kChain = 8;

struct RowDist {   // per lane r < k: entry r of the row's support, best first
    int idx;
    double prob;
    bool bad;      // the row has no distribution (warp-uniform)
};

// One warp: lane r < k holds key r of a row's support (best first; kBadList in lane 0 marks a
// row with a NaN or +inf).  Turns the k logits into probabilities in float64.
__device__ __forceinline__ RowDist dist_from_keys(const TopkParams &P, unsigned long long key)
{
    const int lane = threadIdx.x & 31, k = P.k;
    RowDist d;
    d.idx = -1;
    d.prob = NAN;
    const float val = key_value(key);
    const float best = __shfl_sync(kFullMask, val, 0);
    d.bad = __shfl_sync(kFullMask, key, 0) == kBadList || !(best > -INFINITY);  // nothing above -inf
    if (d.bad) return d;
    const double T = (double)P.temperature;
    const double z = (double)val / T;
    const double mx = __shfl_sync(kFullMask, z, 0);
    const double e = lane < k ? exp(z - mx) : 0.0;
    double S = 0.0;  // the lanes beyond k add 0
    if (k > kChain) {
        S = warp_sum(e);
    } else {
        for (int r = 0; r < k; r += 4) {
#pragma unroll
            for (int j = 0; j < 4; ++j) S += __shfl_sync(kFullMask, e, r + j);
        }
    }
    d.idx = lane < k ? key_index(key) : -1;
    d.prob = e / S;
    return d;
}

__device__ __forceinline__ unsigned long long warp_max_u64(unsigned long long x)
{
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        const unsigned long long y = __shfl_xor_sync(kFullMask, x, o);
        x = y > x ? y : x;
    }
    return x;
}

struct MergeShared {
    unsigned long long key[kMergeCap + 8];
    unsigned long long top[32];
    int list[kMergeLists];
};

// One warp: the k largest of the c <= kMergeCap keys in sh.key (at least k), best first, to sh.top.
__device__ __forceinline__ void rank_merged(MergeShared &sh, int c, int k)
{
    const int lane = threadIdx.x & 31;
    if (lane < 8) sh.key[c + lane] = 0ull;  // the ranking goes in steps of eight
    __syncwarp();
    for (int i = lane; i < c; i += 32) {
        const unsigned long long y = sh.key[i];
        int rank = 0;
        for (int j0 = 0; j0 < c; j0 += 8) {
#pragma unroll
            for (int j = 0; j < 8; ++j) rank += sh.key[j0 + j] > y;
        }
        if (rank < k) sh.top[rank] = y;
    }
    __syncwarp();
}

// One warp: merges the lists of a row of many runs; returns key r of the row's support in lane r (kBadList in lane 0 marks a
// row with a NaN or +inf).  Of the lists' j-th keys - one per lane, the largest of the lane's lists - the r-th largest,
// r * j >= k, bounds the row's k-th key from below: r lists hold j keys each that reach it.  So does the largest of their last
// keys, the better bound where one run holds most of the row's best (masked and ascending rows).  The keys that
// reach it are few more than k, ranked by counting; if more come than fit, those that have come are cut back to their k best,
// the last of which is a better bound.  All keys are looked at where they are few (four round trips), else only the
// lists whose first key reaches the bound, hardly ever more than k of the hundreds.
// (With the lists' last keys alone for a bound, far lower where many lists interleave, the edge call took
// 75 us at k = 32 B = 1 gamma = 4 V = 128256 float32, 32 lists per row, now 12.1; k = 10 B = 1 gamma = 2 V = 4194304 217, now 30.)
__device__ __forceinline__ unsigned long long merge_many(const unsigned long long *src, int runs, int k, MergeShared &sh)
{
    const int lane = threadIdx.x & 31, m = runs * k;
    const bool all = m <= 1024;
    // one round trip for the first 256 keys and what the bound is taken from
    unsigned long long x[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) x[u] = all && 32 * u + lane < m ? ld_after(src + 32 * u + lane) : 0ull;
    const int half = ((runs < 32 ? runs : 32) + 1) / 2;
    const int j = (k + half - 1) / half, r = (k + j - 1) / j;
    unsigned long long best = 0ull, last = 0ull;
    bool bad = false;
    for (int q0 = lane; q0 < runs; q0 += 256) {
        unsigned long long y[8], z[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const bool there = q0 + 32 * u < runs;
            y[u] = there ? ld_after(src + (size_t)(q0 + 32 * u) * k + j - 1) : 0ull;
            z[u] = there ? ld_after(src + (size_t)(q0 + 32 * u) * k + k - 1) : 0ull;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            bad |= y[u] == kBadList;
            best = y[u] > best ? y[u] : best;
            last = z[u] > last ? z[u] : last;
        }
    }
    if (__any_sync(kFullMask, bad)) return lane == 0 ? kBadList : 0ull;
    sh.top[lane] = best;
    __syncwarp();
    int place = 0;
#pragma unroll
    for (int i = 0; i < 32; ++i) {
        const unsigned long long o = sh.top[i];
        place += o > best || (o == best && i < lane);
    }
    unsigned long long bound = __shfl_sync(kFullMask, best, __ffs(__ballot_sync(kFullMask, place == r - 1)) - 1);
    last = warp_max_u64(last);
    if (last > bound) bound = last;
    if (bound == 0ull) bound = 1ull;  // too few lists of j keys: every key counts, empty slots do not
    int c = 0;
    auto append = [&](unsigned long long y) {
        unsigned keep = __ballot_sync(kFullMask, y >= bound);
        if (!keep) return;
        if (c + __popc(keep) > kMergeCap) {
            __syncwarp();
            rank_merged(sh, c, k);
            bound = sh.top[k - 1];
            if (lane < k) sh.key[lane] = sh.top[lane];
            __syncwarp();
            c = k;
            keep = __ballot_sync(kFullMask, y >= bound);
        }
        if (y >= bound) sh.key[c + __popc(keep & ((1u << lane) - 1u))] = y;
        c += __popc(keep);
    };
    if (all) {
        for (int i0 = 0;;) {
#pragma unroll
            for (int u = 0; u < 8; ++u) append(x[u]);
            i0 += 256;
            if (i0 >= m) break;
#pragma unroll
            for (int u = 0; u < 8; ++u) x[u] = i0 + 32 * u + lane < m ? ld_after(src + i0 + 32 * u + lane) : 0ull;
        }
    } else {
        int lists = 0;  // noted in sh.list, their keys not looked at yet
        auto take = [&]() {
            __syncwarp();
            for (int i0 = 0; i0 < lists * k; i0 += 256) {
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int i = i0 + 32 * u + lane;
                    x[u] = i < lists * k ? ld_after(src + (size_t)sh.list[i / k] * k + i % k) : 0ull;
                }
#pragma unroll
                for (int u = 0; u < 8; ++u) append(x[u]);
            }
            lists = 0;
            __syncwarp();
        };
        for (int q0 = 0; q0 < runs; q0 += 256) {
            unsigned long long y[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) y[u] = q0 + 32 * u + lane < runs ? ld_after(src + (size_t)(q0 + 32 * u + lane) * k) : 0ull;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const unsigned reach = __ballot_sync(kFullMask, y[u] >= bound);
                if (lists + __popc(reach) > kMergeLists) take();
                if (reach >> lane & 1u) sh.list[lists + __popc(reach & ((1u << lane) - 1u))] = q0 + 32 * u + lane;
                lists += __popc(reach);
            }
        }
        take();
    }
    __syncwarp();
    rank_merged(sh, c, k);
    const unsigned long long key = lane < k ? sh.top[lane] : 0ull;
    __syncwarp();
    return key;
}

// The same where the keys fit a warp's registers and k is small: the largest of the lists' last keys is bound enough (7 runs,
// k = 5, B = 32 gamma = 4 V = 50257 bf16: the edge call 10.2 us, with merge_many 11.9; k = 32: 19.1 and 14.4).
// Up to kMergeSmall keys at any k: 4 runs, k = 20, a round of B = 112 gamma = 7 V = 25792 bf16 23.5 us, with merge_many 25.4.
// kFewRegs, where a kernel has 64 registers: the lists' ends are fetched one turn after the other (there is more than one turn from
// 33 runs on only); four turns at once cost it 52 bytes of spills (B = 1024 gamma = 4 V = 8192 k = 20: the edge call 37.5 us, now 36.3;
// B = 1000 gamma = 4 V = 16384 k = 4 59.4 and 58.1), but leave the kernels of 128 registers a shorter chain.
constexpr int kMergeFew = 256, kMergeSmall = 96;
template <bool kFewRegs>
__device__ __forceinline__ unsigned long long merge_few(const unsigned long long *src, int runs, int k, MergeShared &sh)
{
    const int lane = threadIdx.x & 31, m = runs * k;
    // one round trip for the lists' ends and their keys
    unsigned long long x[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) x[u] = 32 * u + lane < m ? ld_after(src + 32 * u + lane) : 0ull;
    // the logit of the largest last key is bound enough, and one instruction finds it (an empty slot has none)
    uint32_t top = 0u;
    if constexpr (kFewRegs) {
#pragma unroll 1
        for (int r = lane; r < runs; r += 32) top = max(top, (uint32_t)(ld_after(src + (size_t)r * k + k - 1) >> 32));
    } else {
        for (int r = lane; r < runs; r += 32) top = max(top, (uint32_t)(ld_after(src + (size_t)r * k + k - 1) >> 32));
    }
    top = __reduce_max_sync(kFullMask, top);
    if (top == (uint32_t)(kBadList >> 32)) return lane == 0 ? kBadList : 0ull;
    // no list is full: every key counts, empty slots do not
    const unsigned long long bound = top ? (unsigned long long)top << 32 : 1ull;
    int c = 0;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const unsigned keep = __ballot_sync(kFullMask, x[u] >= bound);
        if (x[u] >= bound) sh.key[c + __popc(keep & ((1u << lane) - 1u))] = x[u];
        c += __popc(keep);
    }
    __syncwarp();
    rank_merged(sh, c, k);
    const unsigned long long key = lane < k ? sh.top[lane] : 0ull;
    __syncwarp();
    return key;
}

// The acceptance test of one position, as the oracle states it (float64 throughout)
__device__ __forceinline__ bool judge(const TopkParams &P, const RowDist &d, int x, double u, double q, unsigned &fl,
                                      double &p)
{
    const int lane = threadIdx.x & 31;
    const unsigned holds = __ballot_sync(kFullMask, lane < P.k && !d.bad && d.idx == x);
    const double p_in = __shfl_sync(kFullMask, d.prob, holds ? __ffs(holds) - 1 : 0);
    if (x < 0 || x >= P.V) {
        fl |= DSSD_EDGE_FLAG_BAD_TOKEN;
        p = NAN;
        return false;
    }
    p = d.bad ? NAN : (holds ? p_in : 0.0);
    // u < min(1, p / q) as  u < 1  and  u q < p  (u q is exact, and the chain is shorter by a division)
    if (q != q || p != p) return false;
    if (q <= 0.0) return u < (p > 0.0 ? 1.0 : 0.0);
    return u < 1.0 && u * q < p;
}

// One row, by a warp: its support's distribution from the lists of its runs (their merged keys in `key`), the acceptance test if
// a token was drafted for it.  Bit 0 of the result: accepted, flag bits from bit 8 on.
template <bool kMany, bool kFewRegs>
__device__ __forceinline__ unsigned fold_row(const TopkParams &P, int b, int j, MergeShared &sh, RowDist &d, unsigned long long &key)
{
    const int lane = threadIdx.x & 31, k = P.k;
    int x = 0;
    float u = 0.f, q = 0.f;
    if (j < P.gamma) {
        const size_t o = (size_t)b * P.gamma + j;
        x = ld_after(P.draft_tokens + o);
        u = ld_after(P.uniforms + o);
        q = ld_after(P.draft_q_tok + o);
    }
    const unsigned long long *lists = P.lists + ((size_t)b * (P.gamma + 1) + j) * P.runs * k;
    key = P.runs == 1 ? (lane < k ? ld_after(lists + lane) : 0ull) : kMany ? merge_many(lists, P.runs, k, sh) : merge_few<kFewRegs>(lists, P.runs, k, sh);
    d = dist_from_keys(P, key);
    unsigned fl = d.bad ? DSSD_EDGE_FLAG_NONFINITE : 0u;
    bool accept = true;
    if (j < P.gamma) {
        double p;
        accept = judge(P, d, x, (double)u, (double)q, fl, p);
        if (lane == 0 && P.p_tok) P.p_tok[(size_t)b * P.gamma + j] = (float)p;
    }
    return (accept ? 1u : 0u) | (fl << 8);
}

__device__ __forceinline__ void write_pairs(const TopkParams &P, int b, const RowDist &d)
{
    const int lane = threadIdx.x & 31, k = P.k;
    if (lane >= k) return;
    P.p_idx[(size_t)b * k + lane] = d.bad ? -1 : d.idx;
    P.p_val[(size_t)b * k + lane] = d.bad ? NAN : (float)d.prob;
}

// One CTA per sequence, a warp per row (the rows in turns when there are more than kFoldWarps).  Bound by
// latency: one round trip for the lists and the float64 operations that depend on one another.  More sequences than are resident
// at 128 registers run with 64 (kCtas = 2): B = 8192 gamma = 2 V = 4096 k = 4 84 us for the edge call against 93; one wave is
// quicker with 128: B = 256 gamma = 4 V = 151936 k = 10 67.2 against 67.9.
template <bool kMany, int kCtas>
__global__ void __launch_bounds__(32 * kFoldWarps, kCtas) topk_fold_kernel(const __grid_constant__ TopkParams P)
{
    extern __shared__ unsigned char smem[];
    MergeShared *merge = reinterpret_cast<MergeShared *>(smem);
    __shared__ unsigned s_verdict[kFoldWarps];  // bit 0: accepted, flag bits from bit 8 on
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    const int b = blockIdx.x, rows = P.gamma + 1;
    pdl_wait();
    pdl_trigger();
    int n = P.gamma;
    unsigned fl = 0;
    for (int base = 0; base < rows; base += warps) {
        const int j = base + warp;
        RowDist d;
        d.idx = -1;
        d.prob = NAN;
        d.bad = false;
        unsigned mine = 1u;
        if (j < rows) {
            unsigned long long key;
            mine = fold_row<kMany, (kCtas > 1)>(P, b, j, merge[warp], d, key);
        }
        if (lane == 0) s_verdict[warp] = mine;
        __syncthreads();
        const unsigned v = lane < warps ? s_verdict[lane] : 1u;
        fl |= __reduce_or_sync(kFullMask, v >> 8);
        const unsigned rej = __ballot_sync(kFullMask, !(v & 1u));
        const bool open = n == P.gamma;  // no rejection before this batch
        if (rej && open) n = base + __ffs(rej) - 1;
        if (open && n == j) write_pairs(P, b, d);  // row n is this warp's
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        P.accept_len[b] = n;
        if (P.flags) P.flags[b] = fl;
    }
}

// The same in two steps for many positions, which the kernel above takes in turns: a warp per row leaves the row's verdict and, in
// the place of its first list, its merged keys; a warp per sequence finds row n.  B = 2 gamma = 200 V = 32000 k = 10: the edge call
// 17.0 us, in turns 54.5; gamma = 64 12.0 and 21.7; gamma = 31, two turns, 11.8.
template <bool kMany>
__global__ void __launch_bounds__(32 * kFoldWarps, 1) topk_rows_kernel(const __grid_constant__ TopkParams P)
{
    extern __shared__ unsigned char smem[];
    MergeShared *merge = reinterpret_cast<MergeShared *>(smem);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long row = (long long)blockIdx.x * kFoldWarps + warp;
    pdl_wait();
    pdl_trigger();
    if (row >= (long long)P.B * (P.gamma + 1)) return;
    const int b = (int)(row / (P.gamma + 1)), j = (int)(row - (long long)b * (P.gamma + 1));
    RowDist d;
    unsigned long long key;
    const unsigned verdict = fold_row<kMany, false>(P, b, j, merge[warp], d, key);
    if (lane < P.k) P.lists[(size_t)row * P.runs * P.k + lane] = key;
    if (lane == 0) P.verdict[row] = verdict;
}

__global__ void __launch_bounds__(kThreads) topk_first_kernel(const __grid_constant__ TopkParams P)
{
    const int lane = threadIdx.x & 31;
    const long long b = (long long)blockIdx.x * kWarps + (threadIdx.x >> 5);
    pdl_wait();
    pdl_trigger();
    if (b >= P.B) return;
    const size_t row0 = (size_t)b * (P.gamma + 1);
    int n = P.gamma;
    unsigned fl = 0;
    for (int base = 0; base <= P.gamma; base += 32) {
        const unsigned v = base + lane <= P.gamma ? ld_after_u32(P.verdict + row0 + base + lane) : 1u;
        fl |= __reduce_or_sync(kFullMask, v >> 8);
        const unsigned rej = __ballot_sync(kFullMask, !(v & 1u));
        if (rej && n == P.gamma) n = base + __ffs(rej) - 1;
    }
    const RowDist d = dist_from_keys(P, lane < P.k ? ld_after(P.lists + (row0 + n) * P.runs * P.k + lane) : 0ull);
    write_pairs(P, (int)b, d);
    if (lane == 0) {
        P.accept_len[b] = n;
        if (P.flags) P.flags[b] = fl;
    }
}

// ---------------------------------------------------------------------------------------------
// device half: one warp per sequence

// inverse CDF over the warp's k entries (lane e holds r_e, entries in increasing index);
// returns the position, or -1 when the mass is not positive and finite.  The sums are those of a loop over the entries, as dssd.h
// says: a chain of additions, the entries from shared memory, two to a load and eight on their way at a time (the draw at B = 1 k = 10 2.03 us, at k = 32 2.25;
// by shuffles 2.12 and 2.28, a round of B = 4 gamma = 2 V = 100744 bf16 k = 32 12.9 and 13.4.  Sums by halves, 2.14 and 2.25, are other
// sums: entries of far smaller weight than the one before them count there).
__device__ __forceinline__ int warp_inverse_cdf(double r, int k, double u)
{
    __shared__ __align__(16) double s_r[kWarps][32];
    const int lane = threadIdx.x & 31;
    double C = 0.0, mine = 0.0;  // the running mass in index order (lanes beyond k hold 0); this lane's
    double *const row = s_r[threadIdx.x >> 5];
    __syncwarp();
    row[lane] = r;
    __syncwarp();
#pragma unroll
    for (int e0 = 0; e0 < 32; e0 += 8) {
        if (e0 >= k) break;
        double2 v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = reinterpret_cast<const double2 *>(row + e0)[j];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            C += j & 1 ? v[j / 2].y : v[j / 2].x;
            if (lane == e0 + j) mine = C;
        }
    }
    if (!(C > 0.0) || !(C < INFINITY)) return -1;
    const unsigned hit = __ballot_sync(kFullMask, lane < k && mine > u * C);
    const unsigned positive = __ballot_sync(kFullMask, r > 0.0);
    return hit ? __ffs(hit) - 1 : 31 - __clz(positive);
}

__global__ void __launch_bounds__(kThreads) topk_resample_kernel(const __grid_constant__ TopkResampleParams P)
{
    __shared__ int s_idx[kWarps][32];
    __shared__ float s_val[kWarps][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, k = P.k;
    const int b = blockIdx.x * kWarps + warp;
    pdl_wait();
    pdl_trigger();
    if (b >= P.B) return;
    const int n = ld_after(P.accept_len + b);
    const double u = (double)ld_after(P.uniforms + b);
    const int pi = lane < k ? ld_after(P.p_idx + (size_t)b * k + lane) : 0x7fffffff;
    const float pv = lane < k ? ld_after(P.p_val + (size_t)b * k + lane) : 0.f;
    const bool has_row = !__any_sync(kFullMask, lane < k && pi < 0);
    unsigned fl = 0u;
    int tok = -1;
    if (n < 0 || n > P.gamma || !has_row) {
        fl = DSSD_RS_FLAG_INVALID;
    } else {
        // P's entries in increasing vocabulary index (indices are distinct)
        int rank = 0;
        for (int e0 = 0; e0 < k; e0 += 4) {
#pragma unroll
            for (int j = 0; j < 4; ++j) rank += __shfl_sync(kFullMask, pi, e0 + j) < pi;
        }
        if (lane < k) {
            s_idx[warp][rank] = pi;
            s_val[warp][rank] = pv;
        }
        __syncwarp();
        const int sid = lane < k ? s_idx[warp][lane] : -1;
        const double sp = lane < k ? (double)s_val[warp][lane] : 0.0;
        int pos;
        if (n == P.gamma) {
            fl |= DSSD_RS_FLAG_BONUS;
            pos = warp_inverse_cdf(sp, k, u);
        } else {
            const size_t qo = ((size_t)b * P.gamma + n) * (size_t)k;
            const int qi = lane < k ? ld_after(P.q_idx + qo + lane) : -1;
            const float qv = lane < k ? ld_after(P.q_val + qo + lane) : 0.f;
            float sq = 0.f;
            for (int f0 = (k - 1) & ~3; f0 >= 0; f0 -= 4) {  // the first listed match wins
#pragma unroll
                for (int j = 3; j >= 0; --j) {
                    const int fi = __shfl_sync(kFullMask, qi, f0 + j);
                    const float fv = __shfl_sync(kFullMask, qv, f0 + j);
                    if (fi == sid) sq = fv;
                }
            }
            const double r = lane < k ? fmax(0.0, sp - (double)sq) : 0.0;
            pos = warp_inverse_cdf(r, k, u);
            if (pos < 0) {
                fl |= DSSD_RS_FLAG_FALLBACK;
                pos = warp_inverse_cdf(sp, k, u);
            }
        }
        if (pos < 0) fl |= DSSD_RS_FLAG_INVALID;
        else tok = __shfl_sync(kFullMask, sid, pos);
    }
    if (lane == 0) {
        P.token[b] = tok;
        if (P.flags) P.flags[b] = fl;
    }
}

}  // namespace

// runs per row and their length in vectors for one type of logits
static void topk_geometry(int B, int gamma, int V, int esz, int &runs, int &run_vecs)
{
    const long long nvec = (long long)V * esz / 16;
    const unsigned long long tiles =
        (unsigned long long)B * (unsigned long long)(gamma + 1) * (unsigned long long)((nvec + kSelTile - 1) / kSelTile);
    const long long per = tiles < kSelTwoTiles ? 1 : tiles < kSelFourTiles ? 2 : 4;
    const long long r = (nvec + per * kSelTile - 1) / (per * kSelTile);
    runs = (int)(r < 1 ? 1 : r);
    run_vecs = (int)(per * kSelTile);
}

// Enough for every launch of no more sequences, positions, vocabulary entries and k than these, of either type: a
// workspace made for the largest batch serves the smaller ones.  A launch of t tiles keeps t lists below kSelTwoTiles,
// rows * ceil(n / 2) <= t of them below kSelFourTiles (n tiles per row) and rows * ceil(n / 4) beyond; each bound grows with
// rows and n, and so does the largest of the three.
static size_t list_bytes(int B, int gamma, int V, int k)
{
    const unsigned long long rows = (unsigned long long)B * (unsigned long long)(gamma + 1);
    unsigned long long n = ((unsigned long long)V * 4 / 16 + kSelTile - 1) / kSelTile;
    if (n < 1) n = 1;
    auto least = [](unsigned long long a, unsigned long long b) { return a < b ? a : b; };
    unsigned long long lists = least(rows * n, kSelTwoTiles), two = least(rows * ((n + 1) / 2), kSelFourTiles);
    if (two > lists) lists = two;
    if (rows * n >= kSelFourTiles && rows * ((n + 3) / 4) > lists) lists = rows * ((n + 3) / 4);
    return ((size_t)lists * (size_t)k * 8 + 255) & ~(size_t)255;
}

size_t topk_workspace_bytes(int B, int gamma, int V, int k)
{
    return list_bytes(B, gamma, V, k) + (((size_t)B * (size_t)(gamma + 1) * 4 + 255) & ~(size_t)255);
}

cudaError_t topk_verify_launch(TopkParams &P, int dtype, void *workspace, cudaStream_t stream)
{
    topk_geometry(P.B, P.gamma, P.V, dtype == DSSD_BF16 ? 2 : 4, P.runs, P.run_vecs);
    P.lists = static_cast<unsigned long long *>(workspace);
    P.verdict = reinterpret_cast<uint32_t *>(static_cast<char *>(workspace) + list_bytes(P.B, P.gamma, P.V, P.k));
    const unsigned long long grid = (unsigned long long)P.B * (unsigned long long)(P.gamma + 1) * (unsigned long long)P.runs;
    if (grid > 0x7fffffffull) return cudaErrorInvalidConfiguration;
    const cudaError_t e = dtype == DSSD_BF16 ? launch_pdl(topk_select_kernel<DSSD_BF16>, (unsigned)grid, kSelThreads, stream, P)
                                             : launch_pdl(topk_select_kernel<DSSD_F32>, (unsigned)grid, kSelThreads, stream, P);
    if (e != cudaSuccess) return e;
    const int warps = P.gamma + 1 < kFoldWarps ? P.gamma + 1 : kFoldWarps;
    const long long keys = (long long)P.runs * P.k;
    const bool many = keys > kMergeFew || (P.k > kGroupsUpTo && keys > kMergeSmall);
    if (P.gamma + 1 > kFoldTurns * kFoldWarps) {
        const unsigned ctas = (unsigned)(((long long)P.B * (P.gamma + 1) + kFoldWarps - 1) / kFoldWarps);
        const cudaError_t r = launch_pdl(many ? topk_rows_kernel<true> : topk_rows_kernel<false>, ctas, 32u * kFoldWarps, stream, P,
                                         kFoldWarps * sizeof(MergeShared));
        return r != cudaSuccess ? r : launch_pdl(topk_first_kernel, ((unsigned)P.B + kWarps - 1) / kWarps, kThreads, stream, P);
    }
    const bool waves = (long long)P.B * warps > 148 * kFoldWarps;
    return launch_pdl(many ? topk_fold_kernel<true, 1> : waves ? topk_fold_kernel<false, 2> : topk_fold_kernel<false, 1>, (unsigned)P.B,
                      32u * (unsigned)warps, stream, P, (size_t)warps * sizeof(MergeShared));
}

cudaError_t topk_resample_launch(const TopkResampleParams &P, cudaStream_t stream)
{
    return launch_pdl(topk_resample_kernel, (unsigned)((P.B + kWarps - 1) / kWarps), kThreads, stream, P);
}

}  // namespace dssd
