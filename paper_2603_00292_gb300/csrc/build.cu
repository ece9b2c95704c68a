// LBVH construction on the GPU: primitive boxes and centroid bounds, Morton codes, a stable
// LSD radix sort, hierarchy emission and bottom-up fit in blocks of leaves (emit_fit.cuh),
// plus the top-level (instance) build. Refits and the fit after a clustering build walk up
// from the leaves with atomic visit counters (fitKernel).
//
// Method: the paper describes BVH construction, its surface-area cost and refitting
// from child boxes (Sec. 6.2) and the geometry / scene build API (Sec. 7.2-7.3). The
// linear build makes the tree and node numbering of Karras, "Maximizing Parallelism in the
// Construction of BVHs, Octrees, and k-d Trees" (HPG 2012). Builds of one block search each
// node's range and split in the sorted codes; larger ones find them from the leaves upwards.
#include <algorithm>
#include <atomic>
#include <cstring>
#include <mutex>
#include <unordered_map>

#include "cluster.cuh"
#include "emit_fit.cuh"
#include "lbvh_block.cuh"
#include "ploc.cuh"
#include "split.cuh"

namespace grt {

// ======================================================================= radix sort
// Stable least-significant-digit radix sort of (key, value) pairs, 8 bits a pass, one
// launch a pass (Adinolfi and Merrill's single-pass sort, "Onesweep", 2022, over Merrill
// and Garland's decoupled look-back, 2016). The digit histograms of every pass depend on
// the keys alone and are counted once, before the first pass; a pass then takes its tiles
// in order from a ticket, ranks a tile's keys on chip, learns from the tiles before it how
// many of each digit they hold, and writes its own in digit order.
//
// What bounds it: a pass moves 2 x 12 B (8 B with 32-bit keys) a pair, which L2 holds at
// every size that fits it, so the time is the chain load -> rank -> look back -> store of
// one wave of tiles, all of which run at once, and the instructions of ranking. The
// look-back is therefore two levels deep: tiles add their counts to their group's, a tile
// sums the groups before its own and the tiles before it in its group, and a group's first
// tile publishes what lies before the group. Measured on a 1.23 M build with 63-bit codes (8
// passes): groups of 8, 472-478 us; one level 491; groups of 16, 495-511. A pass takes 16 us
// there and 6 at 131,072 32-bit keys. The form before it (a histogram launch, a scan of 256
// counters per block on ONE block, a scatter straight from registers) took 88 us, 55 of them
// in the scan, and 21 us. Tiles of 2,048 keys at four blocks per SM (64 registers): the 603
// tiles of 1.23 M keys run in one wave (tiles of 3,072: 486 us, of 1,024: 509).
constexpr int kSortThreads = 256;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kSortItems = 8;
constexpr int kSortTile = kSortThreads * kSortItems;
constexpr int kRadix = 256;
constexpr int kMaxPasses = 8;
static_assert(kSortThreads == kRadix, "one thread per digit");
// Look-back words, 64 bits each so that a count up to 2^32 and its state are one store: a
// tile's count of a digit with bit 32 set once it is there; a group's count with the number
// of its tiles that have added theirs above it; the count before a group with bit 32 set.
constexpr unsigned long long kLookOne = 1ull << 32;
constexpr uint32_t kLookGroup = 8;          // tiles of a group
constexpr int kLookWindow = 2;              // groups read at a time
constexpr uint32_t kLookSpins = 1u << 22;   // polls of one word, far above any tile's time

// Scratch of a sort: digit counts of every pass, the passes' tile tickets, and two sets of
// look-back words used in turn (a pass clears the next one's). A set: the tiles' words, then
// the groups' counts, then the counts before the groups, kRadix words each.
struct SortScratch {
    uint32_t* hist;             // kMaxPasses x kRadix
    uint32_t* tickets;          // kMaxPasses
    unsigned long long* look[2];
};
constexpr size_t kSortHeadBytes = (size_t)kMaxPasses * kRadix * 4 + 256;
__host__ __device__ inline uint32_t lookGroups(uint32_t tiles) { return (tiles + kLookGroup - 1) / kLookGroup; }
static size_t lookBytes(uint32_t n) {
    const uint32_t tiles = std::max(1u, ceilDiv(n, kSortTile));
    return ((size_t)tiles + 2 * (size_t)lookGroups(tiles)) * kRadix * sizeof(unsigned long long);
}
size_t sortScratchBytes(uint32_t n) { return kSortHeadBytes + 2 * lookBytes(n); }
static SortScratch sortScratch(void* p, uint32_t n) {
    char* c = static_cast<char*>(p);
    SortScratch S;
    S.hist = reinterpret_cast<uint32_t*>(c);
    S.tickets = S.hist + kMaxPasses * kRadix;
    S.look[0] = reinterpret_cast<unsigned long long*>(c + kSortHeadBytes);
    S.look[1] = reinterpret_cast<unsigned long long*>(c + kSortHeadBytes + lookBytes(n));
    return S;
}

__device__ __forceinline__ unsigned long long loadRelaxed(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void storeRelaxed(unsigned long long* p, unsigned long long v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// Word *p, already read as w, once it has reached `ready`. The tile that brings it there
// started before this one, so it always gets there; the limit only ends a wait on a
// corrupted word, and the pass's stores are bounded all the same.
__device__ __forceinline__ uint32_t lookValue(const unsigned long long* p, unsigned long long w,
                                              unsigned long long ready, uint32_t* error) {
    for (uint32_t spin = 0; w < ready; ++spin) {
        if (spin == kLookSpins) {
            latchError(error, GRT_ERROR_TIMEOUT);
            break;
        }
        w = loadRelaxed(p);
    }
    return (uint32_t)w;
}

// Adds key k's digits to the block's histograms h[pass][digit]. A warp whose lanes share a
// digit (the high digits of neighbouring primitives) adds them at once: 32 atomics on one
// word of shared memory would run one after another.
template <typename K>
__device__ __forceinline__ void countDigits(K k, bool valid, int passes, uint32_t (*h)[kRadix]) {
    const unsigned act = __ballot_sync(0xffffffffu, valid);
    if (!act) return;
    const int leader = __ffs(act) - 1;
    for (int p = 0; p < passes; ++p) {
        const uint32_t d = (uint32_t)(k >> (8 * p)) & (kRadix - 1);
        const uint32_t d0 = __shfl_sync(0xffffffffu, d, leader);
        if (__all_sync(0xffffffffu, !valid || d == d0)) {
            if ((int)(threadIdx.x & 31u) == leader) atomicAdd(&h[p][d0], (uint32_t)__popc(act));
        } else if (valid) {
            atomicAdd(&h[p][d], 1u);
        }
    }
}

__device__ __forceinline__ void flushDigits(int passes, const uint32_t (*h)[kRadix], uint32_t* hist) {
    for (int j = threadIdx.x; j < passes * kRadix; j += blockDim.x) {
        const uint32_t c = (&h[0][0])[j];
        if (c) atomicAdd(hist + j, c);
    }
}

// Blocks that count digits are large and few (countBlocks: two per SM fill it): each ends in
// an atomic per nonzero count on the same kMaxPasses x kRadix words. With eight blocks of
// 256 threads per SM the Morton kernel took 20 us at 1.23 M keys, 10 of them there.
constexpr int kCountThreads = 1024;
static unsigned countBlocks(Context* ctx, uint32_t n) {
    return std::min(ceilDiv(n, kCountThreads), 2u * (unsigned)std::max(1, smCount(ctx)));
}

// Digit counts of every pass of n keys (hist zeroed). A single block (one tile of keys, zeroWords
// > 0) needs nothing zeroed: it writes its counts and zeros behind them, the rest of the sort's
// zeroWords (100 keys, one pass: 12.9 us a sort instead of 17.5 with a memset before).
template <typename K>
__global__ void __launch_bounds__(kCountThreads) sortHistogramKernel(const K* __restrict__ keys, uint32_t n, int passes,
                                                                    uint32_t* __restrict__ hist, uint32_t zeroWords) {
    __shared__ uint32_t h[kMaxPasses][kRadix];
    for (int j = threadIdx.x; j < passes * kRadix; j += kCountThreads) (&h[0][0])[j] = 0u;
    __syncthreads();
    for (size_t b = (size_t)blockIdx.x * kCountThreads; b < n; b += (size_t)gridDim.x * kCountThreads) {
        const size_t i = b + threadIdx.x;
        countDigits<K>(i < n ? keys[i] : (K)0, i < n, passes, h);
    }
    __syncthreads();
    if (zeroWords) {
        for (uint32_t j = threadIdx.x; j < zeroWords; j += kCountThreads)
            hist[j] = j < (uint32_t)passes * kRadix ? (&h[0][0])[j] : 0u;
    } else {
        flushDigits(passes, h, hist);
    }
}

// Exclusive prefix sum of one value per thread over the block (every thread calls it).
__device__ __forceinline__ uint32_t blockExclusive(uint32_t v, uint32_t* warpSums) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) warpSums[warp] = incl;
    __syncthreads();
    uint32_t base = 0;
#pragma unroll
    for (int w = 0; w < kSortWarps; ++w) base += w < warp ? warpSums[w] : 0u;
    return base + incl - v;
}

// The lanes (of those with ok) whose low eight bits equal this lane's, one vote per bit: a
// __match_any_sync in its place made ranking the longest part of a pass (0.8 us a key of a
// thread). 0 where ok is false.
__device__ __forceinline__ uint32_t digitPeers(uint32_t d, bool ok) {
    uint32_t peers = __ballot_sync(0xffffffffu, ok);
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        const bool set = (d >> b) & 1u;
        const uint32_t m = __ballot_sync(0xffffffffu, set);
        peers &= set ? m : ~m;
    }
    return ok ? peers : 0u;
}

// One radix pass over one tile. IDENTITY: the values are the positions (a first pass that
// need not read them).
template <typename K, bool IDENTITY>
__global__ void __launch_bounds__(kSortThreads, 4) sortPassKernel(const K* __restrict__ keysIn,
                                                               const uint32_t* __restrict__ valsIn,
                                                               K* __restrict__ keysOut, uint32_t* __restrict__ valsOut,
                                                               uint32_t n, int pass, const uint32_t* __restrict__ hist,
                                                               uint32_t* tickets, unsigned long long* look,
                                                               unsigned long long* lookNext, uint32_t tiles,
                                                               uint32_t* error) {
    __shared__ uint32_t warpHist[kSortWarps][kRadix];
    __shared__ uint32_t outBase[kRadix];
    __shared__ uint32_t sums[2][kSortWarps];
    __shared__ K sKeys[kSortTile];
    __shared__ uint32_t sVals[kSortTile];
    __shared__ uint32_t sTile;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t ltMask = (1u << lane) - 1u;
    const int shift = 8 * pass;
    if (tid == 0) sTile = atomicAdd(tickets + pass, 1u);  // tiles start in order: a tile only waits for running ones
    const uint32_t digitTotal = hist[pass * kRadix + tid];
#pragma unroll
    for (int w = 0; w < kSortWarps; ++w) warpHist[w][tid] = 0u;
    __syncthreads();
    const uint32_t tile = sTile;
    const uint32_t first = tile * (uint32_t)kSortTile;
    const uint32_t count = min((uint32_t)kSortTile, n - first);
    K k[kSortItems];
    uint32_t v[kSortItems], rank[kSortItems];
#pragma unroll
    for (int i = 0; i < kSortItems; ++i) {
        const uint32_t j = (uint32_t)(warp * kSortItems + i) * 32u + (uint32_t)lane;
        const bool ok = j < count;
        k[i] = ok ? keysIn[(size_t)first + j] : (K)0;
        v[i] = IDENTITY ? first + j : ok ? valsIn[(size_t)first + j] : 0u;
    }
    const uint32_t group = tile / kLookGroup;
    const size_t groupsAt = (size_t)tiles * kRadix + tid, beforeAt = groupsAt + (size_t)lookGroups(tiles) * kRadix;
    storeRelaxed(lookNext + (size_t)tile * kRadix + tid, 0ull);
    if (tile % kLookGroup == 0) {
        storeRelaxed(lookNext + groupsAt + (size_t)group * kRadix, 0ull);
        storeRelaxed(lookNext + beforeAt + (size_t)group * kRadix, 0ull);
    }
    uint32_t peers[kSortItems];
#pragma unroll
    for (int i = 0; i < kSortItems; ++i) {
        const bool ok = (uint32_t)(warp * kSortItems + i) * 32u + (uint32_t)lane < count;
        peers[i] = digitPeers((uint32_t)(k[i] >> shift), ok);
    }
#pragma unroll
    for (int i = 0; i < kSortItems; ++i) {
        const uint32_t d = (uint32_t)(k[i] >> shift) & (kRadix - 1);
        const uint32_t b = warpHist[warp][d];
        __syncwarp();
        if (lane == __ffs(peers[i]) - 1) warpHist[warp][d] = b + __popc(peers[i]);
        __syncwarp();
        rank[i] = b + __popc(peers[i] & ltMask);
    }
    __syncthreads();
    // thread = digit: the warps' counts become each warp's first position in the tile's run
    uint32_t total = 0;
#pragma unroll
    for (int w = 0; w < kSortWarps; ++w) {
        const uint32_t c = warpHist[w][tid];
        warpHist[w][tid] = total;
        total += c;
    }
    storeRelaxed(look + (size_t)tile * kRadix + tid, kLookOne | total);
    atomicAdd(look + groupsAt + (size_t)group * kRadix, kLookOne + total);
    const uint32_t digitFirst = blockExclusive(digitTotal, sums[0]);  // over all keys
    const uint32_t tileFirst = blockExclusive(total, sums[1]);        // within the tile
#pragma unroll
    for (int w = 0; w < kSortWarps; ++w) warpHist[w][tid] += tileFirst;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kSortItems; ++i) {
        if ((uint32_t)(warp * kSortItems + i) * 32u + (uint32_t)lane < count) {
            const uint32_t j = warpHist[warp][(uint32_t)(k[i] >> shift) & (kRadix - 1)] + rank[i];
            sKeys[j] = k[i];
            sVals[j] = v[i];
        }
    }
    // the digit's count over the tiles before this one: those of its group, then whole groups
    // back to one whose own count of earlier keys is there
    uint32_t before = 0;
    {
        unsigned long long w[kLookGroup - 1];
        const unsigned long long* p = look + (size_t)group * kLookGroup * kRadix + tid;
        const uint32_t m = tile % kLookGroup;
#pragma unroll
        for (uint32_t j = 0; j + 1 < kLookGroup; ++j) w[j] = j < m ? loadRelaxed(p + (size_t)j * kRadix) : kLookOne;
        uint32_t inGroup = 0;
        bool open = group > 0;
        for (uint32_t g = group; open;) {  // groups g - 1, g - 2, ..
            unsigned long long c[kLookWindow], e[kLookWindow];
#pragma unroll
            for (int j = 0; j < kLookWindow; ++j) {
                const bool in = (uint32_t)j < g;
                c[j] = in ? loadRelaxed(look + groupsAt + (size_t)(g - 1 - j) * kRadix) : 0ull;
                e[j] = in ? loadRelaxed(look + beforeAt + (size_t)(g - 1 - j) * kRadix) : kLookOne;
            }
#pragma unroll
            for (int j = 0; j < kLookWindow; ++j) {
                if (!open) continue;
                before += lookValue(look + groupsAt + (size_t)(g - 1 - j) * kRadix, c[j], kLookGroup * kLookOne, error);
                if ((uint32_t)j + 1 == g) {
                    open = false;
                } else if (e[j] >= kLookOne) {
                    before += (uint32_t)e[j];
                    open = false;
                }
            }
            g -= min(g, (uint32_t)kLookWindow);
        }
        if (m == 0 && group > 0) storeRelaxed(look + beforeAt + (size_t)group * kRadix, kLookOne | before);
#pragma unroll
        for (uint32_t j = 0; j + 1 < kLookGroup; ++j)
            if (j < m) inGroup += lookValue(p + (size_t)j * kRadix, w[j], kLookOne, error);
        before += inGroup;
    }
    outBase[tid] = digitFirst + before - tileFirst;
    __syncthreads();
    for (uint32_t j = tid; j < count; j += kSortThreads) {
        const K key = sKeys[j];
        const uint32_t pos = outBase[(uint32_t)(key >> shift) & (kRadix - 1)] + j;
        if (pos < n) {  // always, unless a wait ran out
            keysOut[pos] = key;
            valsOut[pos] = sVals[j];
        }
    }
}

// The passes over counted digits (scratch.hist) with zeroed tickets and first look-back array.
template <typename K>
static grtError sortPasses(Context* ctx, K* const keys[2], uint32_t* const vals[2], uint32_t n, int passes,
                           const SortScratch& S, bool identity, cudaStream_t s) {
    const unsigned tiles = ceilDiv(n, kSortTile);
    for (int p = 0; p < passes; ++p) {
        const int a = p & 1, b = a ^ 1;
        if (p == 0 && identity)
            sortPassKernel<K, true><<<tiles, kSortThreads, 0, s>>>(keys[a], vals[a], keys[b], vals[b], n, p, S.hist,
                                                                   S.tickets, S.look[a], S.look[b], tiles,
                                                                   &workspace(ctx)->error);
        else
            sortPassKernel<K, false><<<tiles, kSortThreads, 0, s>>>(keys[a], vals[a], keys[b], vals[b], n, p, S.hist,
                                                                    S.tickets, S.look[a], S.look[b], tiles,
                                                                    &workspace(ctx)->error);
        GRT_LAUNCH_CHECK();
    }
    noteLaunches(passes);
    return GRT_SUCCESS;
}

// The pairs of an odd number of passes back in their place, keys and values in one launch.
template <typename K>
__global__ void __launch_bounds__(256) copyPairsKernel(K* __restrict__ keysOut, const K* __restrict__ keysIn,
                                                       uint32_t* __restrict__ valsOut,
                                                       const uint32_t* __restrict__ valsIn, uint32_t n) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        keysOut[i] = keysIn[i];
        valsOut[i] = valsIn[i];
    }
}

template <typename K>
static grtError radixSortT(Context* ctx, K* keys0, K* keys1, uint32_t* vals0, uint32_t* vals1, uint32_t n,
                           int significantBits, void* scratch, cudaStream_t s, int* finalBuf) {
    const int passes = (significantBits + 7) / 8;
    const SortScratch S = sortScratch(scratch, n);
    const size_t zeroed = kSortHeadBytes + lookBytes(n);
    const bool single = n <= (uint32_t)kSortTile;
    if (!single) GRT_CUDA(cudaMemsetAsync(scratch, 0, zeroed, s));
    sortHistogramKernel<K><<<single ? 1u : countBlocks(ctx, n), kCountThreads, 0, s>>>(
        keys0, n, passes, S.hist, single ? (uint32_t)(zeroed / sizeof(uint32_t)) : 0u);
    GRT_LAUNCH_CHECK();
    noteLaunches(1);
    K* const keys[2] = {keys0, keys1};
    uint32_t* const vals[2] = {vals0, vals1};
    *finalBuf = passes & 1;
    return sortPasses<K>(ctx, keys, vals, n, passes, S, false, s);
}

grtError radixSort(Context* ctx, void* keys0, void* keys1, uint32_t* vals0, uint32_t* vals1, uint32_t n, int keyBytes,
                   int significantBits, void* scratch, cudaStream_t s, int* finalBuf) {
    if (n == 0) {
        *finalBuf = 0;
        return GRT_SUCCESS;
    }
    if (keyBytes == 4)
        return radixSortT<uint32_t>(ctx, (uint32_t*)keys0, (uint32_t*)keys1, vals0, vals1, n, significantBits, scratch,
                                    s, finalBuf);
    return radixSortT<unsigned long long>(ctx, (unsigned long long*)keys0, (unsigned long long*)keys1, vals0, vals1, n,
                                          significantBits, scratch, s, finalBuf);
}

// ======================================================================= element kernels (A1-A7)
// Centroids and their bounds. A few blocks per SM loop over the primitives: each block ends
// in six atomics on the same words, which queued behind one another with a block per 256
// primitives.
__global__ void __launch_bounds__(256) primCentroidKernel(PrimSource S, float4* __restrict__ centroids,
                                                          uint32_t* __restrict__ bounds) {
    float mn[3] = {INFINITY, INFINITY, INFINITY}, mx[3] = {-INFINITY, -INFINITY, -INFINITY};
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < S.count; i += (size_t)gridDim.x * blockDim.x) {
        float3 v[3];
        const float3 c = boxCentroid(primBox(S, (uint32_t)i, v));
        centroids[i] = make_float4(c.x, c.y, c.z, 0.f);
        mn[0] = fminf(mn[0], c.x), mn[1] = fminf(mn[1], c.y), mn[2] = fminf(mn[2], c.z);
        mx[0] = fmaxf(mx[0], c.x), mx[1] = fmaxf(mx[1], c.y), mx[2] = fmaxf(mx[2], c.z);
    }
    reduceBoxBounds(mn, mx, bounds);
}

// Morton codes, and the digit counts of every radix pass over them (hist zeroed). The
// values of the pairs are the positions, which the first pass makes itself.
template <typename K, int BITS>
__global__ void __launch_bounds__(kCountThreads) mortonKernel(const float4* __restrict__ centroids, uint32_t n,
                                                             const uint32_t* __restrict__ bounds, K* __restrict__ keys,
                                                             uint32_t* __restrict__ hist) {
    constexpr int kPasses = (3 * BITS + 7) / 8;
    __shared__ uint32_t h[kPasses][kRadix];
    for (int j = threadIdx.x; j < kPasses * kRadix; j += kCountThreads) (&h[0][0])[j] = 0u;
    __syncthreads();
    for (size_t b = (size_t)blockIdx.x * kCountThreads; b < n; b += (size_t)gridDim.x * kCountThreads) {
        const size_t i = b + threadIdx.x;
        K k = 0;
        if (i < n) keys[i] = k = mortonCode<K, BITS>(centroids[i], bounds);
        countDigits<K>(k, i < n, kPasses, h);
    }
    __syncthreads();
    flushDigits(kPasses, h, hist);
}

// A build's scratch before its first kernel: centroid bounds, digit counts, tickets and
// first look-back array of the sort, and the fit's visit counters (only of a fit that counts).
struct BuildInit {
    uint32_t* bounds;
    uint4* sortHead;  // 16-byte words of the sort scratch to clear
    size_t sortWords;
    uint4* flags;
    size_t flagWords;
};
__global__ void __launch_bounds__(256) buildInitKernel(BuildInit I) {
    const size_t at = (size_t)blockIdx.x * blockDim.x + threadIdx.x, step = (size_t)gridDim.x * blockDim.x;
    if (at < 6) I.bounds[at] = at < 3 ? 0xFFFFFFFFu : 0u;  // running minima start at the top, maxima at the bottom
    for (size_t i = at; i < I.sortWords; i += step) I.sortHead[i] = make_uint4(0u, 0u, 0u, 0u);
    for (size_t i = at; i < I.flagWords; i += step) I.flags[i] = make_uint4(0u, 0u, 0u, 0u);
}

// The fit of a hierarchy that is already there (refits, clustering builds, one primitive).
template <int KIND>  // 0 triangles, 1 AABB list
__global__ void __launch_bounds__(256) fitKernel(FitParams P) {
    const uint32_t k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < P.n) fitLeaf<KIND>(P, k);
}

// Quantised form of each of the m 4-wide nodes (the GRT_BUILD_QUANTIZED_NODES layout).
__global__ void __launch_bounds__(256) quantizeKernel(const float4* wide, uint32_t m, float4* qnodes) {
    const uint32_t k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < m) quantizeWideNode(wide + kWideWords * (size_t)k, qnodes + kQuantWords * (size_t)k);
}

// The 8-wide node of each of the m binary nodes of an n-primitive tree (the
// GRT_BUILD_WIDE8_NODES layout). Slots 4s .. 4s+3 are those of child s's 4-wide node, or a
// leaf child and three empty slots, so every row of an 8-wide node is a row of a 4-wide
// one: one thread per row copies it, with whole lines read and written (12 us at 131,072
// triangles; a thread per node that gathered up to seven binary nodes took 18).
__global__ void __launch_bounds__(256) wide8Kernel(const float4* __restrict__ nodes, const float4* __restrict__ wide,
                                                   uint32_t n, uint32_t m, float4* __restrict__ w8) {
    const size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const size_t k = q / kWide8Words;
    if (k >= m) return;
    const uint32_t r = (uint32_t)(q % kWide8Words);
    float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
    if (r < 14) {
        const bool words = r >= 12;
        const uint32_t half = r & 1u, row = words ? 6u : 2 * (r >> 2) + ((r >> 1) & 1u);  // of the 4-wide node
        const uint32_t c = reinterpret_cast<const uint32_t*>(nodes + 4 * k + 3)[half];
        const float none = words ? __uint_as_float(kInvalid) : (row & 1u) ? -INFINITY : INFINITY;
        if (n == 1 && half == 1) {
            o = make_float4(none, none, none, none);
        } else if (c & kLeafBit) {  // binary rows: (lo, hi) of child 0, then of child 1
            const float own =
                words ? __uint_as_float(c)
                      : reinterpret_cast<const float*>(nodes + 4 * k + (row >> 1))[2 * half + (row & 1u)];
            o = make_float4(own, none, none, none);
        } else {
            o = wide[kWideWords * (size_t)c + row];
        }
    }
    w8[q] = o;
}

// The extra node formats of object o, after its fit.
static grtError launchNodeFormats(const BvhObject* o, cudaStream_t s) {
    if (o->qnodes) {
        quantizeKernel<<<ceilDiv(o->nodeCount, 256), 256, 0, s>>>((const float4*)o->wide, o->nodeCount,
                                                                  (float4*)o->qnodes);
        GRT_LAUNCH_CHECK();
        noteLaunches(1);
    }
    if (o->w8nodes) {
        wide8Kernel<<<ceilDiv((size_t)o->nodeCount * kWide8Words, 256), 256, 0, s>>>(
            (const float4*)o->nodes, (const float4*)o->wide, o->leafCount, o->nodeCount, (float4*)o->w8nodes);
        GRT_LAUNCH_CHECK();
        noteLaunches(1);
    }
    return GRT_SUCCESS;
}

// ======================================================================= small builds
// Up to kSmallBuild primitives (kSmallScene instances) a build runs in one block of
// kSmallBuildThreads threads, as one launch, instead of a graph of some nine grid-wide
// launches whose cost is their own latency at this size. The threshold is where the measured
// times of repeated builds cross (us, one block against the graph, 30-bit codes): 512
// triangles 35 / 35, 768 43 / 41, 1,024 49 / 43, 1,280 67 / 45, 2,048 80 / 45. A top level of
// 4,000 instances took 0.61 against 0.15 ms (its FP64 instance setup runs on one SM). Up to
// kSharedFitMax primitives the block keeps the whole build on chip (bitonicSortShared,
// fitLeafShared).
//
// Capturing the graph costs 50 to 70 us, up to kSmallGraph primitives as much as a build: a
// geometry built once paid more for it than the one block took (us, first build of a geometry,
// waited for, one block / graph captured and launched / its launches without a graph: 1,025
// triangles 70 / 112 / 75, 1,280 84 / 126 / 76, 2,048 98 / 125 / 76). There the first builds of a
// description run in one block up to kSmallFirst and as plain launches above, some 15 us longer
// than the graph, which is captured once kDirectBuilds of them have cost what it costs.
constexpr uint32_t kSmallBuild = 1024;
constexpr uint32_t kSmallFirst = 1152;
constexpr uint32_t kSmallGraph = 2048;
constexpr uint32_t kDirectBuilds = 4;
constexpr uint32_t kSmallScene = 1024;
#ifndef GRT_SMALL_BUILD_THREADS
#define GRT_SMALL_BUILD_THREADS 1024
#endif
constexpr int kSmallBuildThreads = GRT_SMALL_BUILD_THREADS;
constexpr int kSmallSceneThreads = 512;  // its FP64 instance setup needs more than 64 registers

// Dynamic shared memory of a single-block build: the radix routines' histograms, or
// the on-chip path's sort pairs, boxes and counters for kSmallFirst primitives.
template <typename K>
constexpr size_t smallBuildSmemBytes() {
    return std::max(blockBuildSmemWords(kSmallBuildThreads) * sizeof(uint32_t),
                    std::max(sharedBuildBytes<K>(kSmallFirst), sharedBuildBytes<K>(kSmallScene)));
}

template <typename K, int BITS>
__global__ void __launch_bounds__(kSmallBuildThreads) smallBuildKernel(BlockBuild B) {
    extern __shared__ uint32_t smem[];
    buildWhole<K, BITS>(B, B.n > 0 ? B.n : 1u, smem, smallBuildSmemBytes<K>());  // one sort chunk
}

// Opts the single-block kernels in to their dynamic shared memory (above the default
// 48 KB for 63-bit codes), once per process and device.
template <class Kern>
static grtError allowSmem(Kern kernel, size_t bytes) {
    int dev = 0;
    GRT_CUDA(cudaGetDevice(&dev));
    static std::mutex m;
    static std::unordered_map<size_t, bool> done;
    const size_t key = (size_t)(void*)kernel ^ ((size_t)dev << 56);
    std::lock_guard<std::mutex> g(m);
    if (done.count(key)) return GRT_SUCCESS;
    GRT_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
    done[key] = true;
    return GRT_SUCCESS;
}

// The device pointers of a build of object o in temporary buffer t.
static BlockBuild blockBuildOf(Context* c, BvhObject* o, const BuildLayout& L, char* t, uint32_t kind) {
    BlockBuild B{};
    B.n = o->leafCount;
    B.bits = o->mortonBits;
    B.sortChunks = 1;
    B.passes = (o->mortonBits + 7) / 8;
    B.kind = kind;
    B.nodes = (float4*)o->nodes;
    B.wide = (float4*)o->wide;
    B.qnodes = (float4*)o->qnodes;
    B.w8nodes = (float4*)o->w8nodes;
    B.leaves = o->leaves;
    B.parents = (uint32_t*)o->parents;
    B.primToLeaf = o->primToLeaf;
    B.header = o->dHeader;
    B.bounds = (uint32_t*)(t + L.bounds);
    B.centroids = (float4*)(t + L.centroids);
    B.keys[0] = t + L.keys[0];
    B.keys[1] = t + L.keys[1];
    B.vals[0] = (uint32_t*)(t + L.vals[0]);
    B.vals[1] = (uint32_t*)(t + L.vals[1]);
    B.counts = (uint32_t*)(t + L.hist);
    B.flags = (uint32_t*)(t + L.flags);
    B.error = &workspace(c)->error;
    return B;
}

static grtError launchSmallBuild(const BlockBuild& B, cudaStream_t s) {
    if (B.bits == 30) {
        const size_t smem = smallBuildSmemBytes<uint32_t>();
        grtError e = allowSmem(smallBuildKernel<uint32_t, 10>, smem);
        if (e != GRT_SUCCESS) return e;
        smallBuildKernel<uint32_t, 10><<<1, kSmallBuildThreads, smem, s>>>(B);
    } else {
        const size_t smem = smallBuildSmemBytes<unsigned long long>();
        grtError e = allowSmem(smallBuildKernel<unsigned long long, 21>, smem);
        if (e != GRT_SUCCESS) return e;
        smallBuildKernel<unsigned long long, 21><<<1, kSmallBuildThreads, smem, s>>>(B);
    }
    GRT_LAUNCH_CHECK();
    noteLaunches(1);
    return GRT_SUCCESS;
}

// ======================================================================= instances (A8)
struct InstanceInput {
    const grtInstance* instances;
    const grtFrameSRT* frames;
    uint32_t count;
    float4* boxes;             // 2 float4 per instance: world lo, hi
    InstanceRecord* records;   // unsorted
    InstanceFrames64* inv64;   // per instance ID
    float4* fwd32;             // kFrameRows rows per instance ID
    float4* centroids;
    uint32_t* bounds;
    uint32_t wide8;            // the scene has 8-wide nodes: so must every instanced geometry
    uint32_t* error;           // the context's device error word
};

// Per instance: frame M = T R S and its inverse S^-1 R^T (x - T) in FP64 (rounded to
// float32), the world box of the bottom level's root box (8 corners through M,
// rounded outward), and the centroid of that box.
__device__ __forceinline__ float3 setupInstance(const InstanceInput& I, uint32_t i) {
    float3 c;
    const grtInstance in = I.instances[i];
    const grtFrameSRT f = I.frames[i];
    const BvhHeader* g = reinterpret_cast<const BvhHeader*>(in.geometry);
    double qx = f.rotation[0], qy = f.rotation[1], qz = f.rotation[2], qw = f.rotation[3];
    const double qn = sqrt(qx * qx + qy * qy + qz * qz + qw * qw);
    qx /= qn, qy /= qn, qz /= qn, qw /= qn;
    const double R[3][3] = {{1 - 2 * (qy * qy + qz * qz), 2 * (qx * qy - qz * qw), 2 * (qx * qz + qy * qw)},
                            {2 * (qx * qy + qz * qw), 1 - 2 * (qx * qx + qz * qz), 2 * (qy * qz - qx * qw)},
                            {2 * (qx * qz - qy * qw), 2 * (qy * qz + qx * qw), 1 - 2 * (qx * qx + qy * qy)}};
    const double S[3] = {f.scale[0], f.scale[1], f.scale[2]};
    const double T[3] = {f.translation[0], f.translation[1], f.translation[2]};
    double F[3][4], G[3][4];
    for (int r = 0; r < 3; ++r) {
        for (int q = 0; q < 3; ++q) {
            F[r][q] = R[r][q] * S[q];
            G[r][q] = R[q][r] / S[r];
        }
        F[r][3] = T[r];
        G[r][3] = -(G[r][0] * T[0] + G[r][1] * T[1] + G[r][2] * T[2]);
    }
    InstanceRecord rec;
    for (int r = 0; r < 3; ++r) {
        rec.inv[r] = make_float4(__double2float_rn(G[r][0]), __double2float_rn(G[r][1]),
                                 __double2float_rn(G[r][2]), __double2float_rn(G[r][3]));
        I.fwd32[kFrameRows * (size_t)i + 3 + r] =
            make_float4(__double2float_rn(G[r][0] - (double)rec.inv[r].x),
                        __double2float_rn(G[r][1] - (double)rec.inv[r].y),
                        __double2float_rn(G[r][2] - (double)rec.inv[r].z),
                        __double2float_rn(G[r][3] - (double)rec.inv[r].w));
        I.fwd32[kFrameRows * (size_t)i + r] = make_float4(__double2float_rn(F[r][0]), __double2float_rn(F[r][1]),
                                                 __double2float_rn(F[r][2]), __double2float_rn(F[r][3]));
        for (int q = 0; q < 4; ++q) I.inv64[i].inv[r][q] = G[r][q];
    }
    // an 8-wide top level walks 8-wide bottom levels; a 4-wide one the geometry's 4-wide
    // (or quantised) nodes. An 8-wide scene instancing a geometry without 8-wide nodes
    // latches GRT_ERROR_INVALID_PARAMETER and leaves that instance empty.
    const bool missing8 = I.wide8 && g->primCount > 0 && g->nodes8 == nullptr;
    if (missing8) latchError(I.error, GRT_ERROR_INVALID_PARAMETER);
    rec.nodes = I.wide8 ? g->nodes8 : g->nodes;
    rec.leaves = g->leaves;
    rec.instanceID = i;
    rec.typeBits = (g->geomType & 0xFFFFFFu) | ((uint32_t)g->primType << 24) |
                   (I.wide8 ? kInstWide8 : g->nodeFormat == 1 ? kInstQuant : 0u) |
                   ((g->flags & kHeaderSplit) ? kInstSplit : 0u) |
                   ((g->primCount == 0 || missing8) ? kInstEmpty : 0u);
    rec.geometry = g;
    double lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    if (g->primCount > 0) {
        for (int cnr = 0; cnr < 8; ++cnr) {
            const double p[3] = {(cnr & 1) ? g->rootHi[0] : g->rootLo[0], (cnr & 2) ? g->rootHi[1] : g->rootLo[1],
                                 (cnr & 4) ? g->rootHi[2] : g->rootLo[2]};
            for (int r = 0; r < 3; ++r) {
                const double w = F[r][0] * p[0] + F[r][1] * p[1] + F[r][2] * p[2] + F[r][3];
                lo[r] = fmin(lo[r], w);
                hi[r] = fmax(hi[r], w);
            }
        }
    } else {
        for (int r = 0; r < 3; ++r) lo[r] = hi[r] = T[r];  // empty: a point box, skipped by traversal
    }
    Box3 b;
    b.lo = make_float3(__double2float_rd(lo[0]), __double2float_rd(lo[1]), __double2float_rd(lo[2]));
    b.hi = make_float3(__double2float_ru(hi[0]), __double2float_ru(hi[1]), __double2float_ru(hi[2]));
    I.boxes[2 * (size_t)i] = make_float4(b.lo.x, b.lo.y, b.lo.z, 0.f);
    I.boxes[2 * (size_t)i + 1] = make_float4(b.hi.x, b.hi.y, b.hi.z, 0.f);
    rec.worldLo = make_float4(b.lo.x, b.lo.y, b.lo.z, 0.f);
    rec.worldHi = make_float4(b.hi.x, b.hi.y, b.hi.z, 0.f);
    rec.mask = in.mask ? in.mask : 0xFFFFFFFFu;
    rec.pad[0] = rec.pad[1] = rec.pad[2] = 0u;
    I.records[i] = rec;
    c = boxCentroid(b);
    I.centroids[i] = make_float4(c.x, c.y, c.z, 0.f);
    return c;
}

__global__ void __launch_bounds__(128) instanceSetupKernel(InstanceInput I) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    const bool valid = i < I.count;
    const float3 c = valid ? setupInstance(I, i) : make_float3(0.f, 0.f, 0.f);
    reduceBounds(c, valid, I.bounds);
}

// A top level of at most kSmallScene instances in one block and one launch: the bounds
// and fit counters initialised, the instance setup, then every LBVH step.
template <typename K, int BITS>
__global__ void __launch_bounds__(kSmallSceneThreads) smallSceneKernel(BlockBuild B, InstanceInput I) {
    extern __shared__ uint32_t smem[];
    if (threadIdx.x == 0) {
        B.bounds[0] = B.bounds[1] = B.bounds[2] = 0xFFFFFFFFu;
        B.bounds[3] = B.bounds[4] = B.bounds[5] = 0u;
    }
    for (uint32_t i = threadIdx.x; i + 1 < B.n; i += blockDim.x) B.flags[i] = 0u;
    __syncthreads();
    float mn[3] = {INFINITY, INFINITY, INFINITY}, mx[3] = {-INFINITY, -INFINITY, -INFINITY};
    for (uint32_t i = threadIdx.x; i < I.count; i += blockDim.x) {
        const float3 c = setupInstance(I, i);
        mn[0] = fminf(mn[0], c.x), mn[1] = fminf(mn[1], c.y), mn[2] = fminf(mn[2], c.z);
        mx[0] = fmaxf(mx[0], c.x), mx[1] = fmaxf(mx[1], c.y), mx[2] = fmaxf(mx[2], c.z);
    }
    reduceBoxBounds(mn, mx, B.bounds);
    __syncthreads();
    buildWhole<K, BITS>(B, B.n, smem, smallBuildSmemBytes<K>());
}

// ======================================================================= host drivers
grtError validateGeometryInput(const grtGeometryBuildInput* in, uint32_t* count) {
    if (!in) return GRT_ERROR_INVALID_PARAMETER;
    if (in->type == GRT_PRIMITIVE_TRIANGLE_MESH) {
        const grtTriangleMeshPrimitive& m = in->triangleMesh;
        if (m.triangleCount && (!m.triangleIndices || !m.vertices || m.triangleStride < 12 || m.vertexStride < 12 ||
                                (m.triangleStride & 3) || (m.vertexStride & 3)))
            return GRT_ERROR_INVALID_PARAMETER;
        if (m.triangleCount >= 0x7FFFFFFFu) return GRT_ERROR_INVALID_PARAMETER;
        *count = m.triangleCount;
        return GRT_SUCCESS;
    }
    if (in->type == GRT_PRIMITIVE_AABB_LIST) {
        const grtAABBListPrimitive& a = in->aabbList;
        if (a.aabbCount && (!a.aabbs || a.aabbStride < 24 || (a.aabbStride & 3))) return GRT_ERROR_INVALID_PARAMETER;
        if (a.aabbCount >= 0x7FFFFFFFu) return GRT_ERROR_INVALID_PARAMETER;
        *count = a.aabbCount;
        return GRT_SUCCESS;
    }
    return GRT_ERROR_INVALID_PARAMETER;
}

PrimSource primSource(const grtGeometryBuildInput* in, uint32_t count) {
    PrimSource S{};
    S.count = count;
    if (in->type == GRT_PRIMITIVE_TRIANGLE_MESH) {
        S.kind = 0;
        S.idx = (const char*)in->triangleMesh.triangleIndices;
        S.idxStride = in->triangleMesh.triangleStride;
        S.verts = (const char*)in->triangleMesh.vertices;
        S.vertStride = in->triangleMesh.vertexStride;
    } else {
        S.kind = 1;
        S.boxes = (const char*)in->aabbList.aabbs;
        S.boxStride = in->aabbList.aabbStride;
    }
    return S;
}

// Live geometries created with GRT_BUILD_QUANTIZED_NODES. While there are none, no
// 4-wide walk can meet quantised nodes, and traces run kernels without that form.
static std::atomic<int> g_quantGeometries{0};
bool anyQuantGeometry() { return g_quantGeometries.load(std::memory_order_relaxed) > 0; }

// count primitives over leafCount leaves (more than count only with split triangles).
static grtError createBvhObject(uint32_t count, uint32_t primType, uint32_t geomType, uint32_t mortonBits,
                                BvhObject** out, bool quant = false, bool wide8 = false, uint32_t leafCount = 0) {
    BvhObject* o = new BvhObject();
    o->primCount = count;
    o->leafCount = count == 0 ? 0 : std::max(leafCount, count);
    o->nodeCount = count == 0 ? 0 : std::max(o->leafCount - 1, 1u);
    o->primType = primType;
    o->geomType = geomType;
    o->mortonBits = mortonBits;
    o->built = false;
    o->quant = quant;
    o->wide8 = wide8;
    size_t leafBytes = primType == GRT_PRIMITIVE_TRIANGLE_MESH ? 48 : (primType == kPrimScene ? 128 : 4);
    cudaError_t e = cudaMalloc(&o->dHeader, sizeof(BvhHeader));
    if (e == cudaSuccess && count) e = cudaMalloc(&o->nodes, (size_t)o->nodeCount * 64);
    if (e == cudaSuccess && count) e = cudaMalloc(&o->wide, (size_t)o->nodeCount * kWideWords * sizeof(float4));
    if (e == cudaSuccess && count && quant)
        e = cudaMalloc(&o->qnodes, (size_t)o->nodeCount * kQuantWords * sizeof(float4));
    if (e == cudaSuccess && count && wide8)
        e = cudaMalloc(&o->w8nodes, (size_t)o->nodeCount * kWide8Words * sizeof(float4));
    if (e == cudaSuccess && count) e = cudaMalloc(&o->leaves, (size_t)o->leafCount * leafBytes);
    if (e == cudaSuccess && count) e = cudaMalloc(&o->parents, (size_t)(2 * (size_t)o->leafCount - 1) * 4);
    if (e == cudaSuccess && count && primType != GRT_PRIMITIVE_AABB_LIST) e = cudaMalloc(&o->primToLeaf, (size_t)count * 4);
    if (e == cudaSuccess && count && primType == kPrimScene) e = cudaMalloc(&o->inv64, (size_t)count * sizeof(InstanceFrames64));
    if (e == cudaSuccess && count && primType == kPrimScene) e = cudaMalloc(&o->fwd32, (size_t)count * kFrameRows * sizeof(float4));
    BvhHeader h{};
    for (int a = 0; a < 3; ++a) h.rootLo[a] = INFINITY, h.rootHi[a] = -INFINITY;
    h.primCount = count;
    h.primType = (uint16_t)primType;
    h.nodeFormat = quant ? 1 : 0;
    h.nodes = (const float4*)(quant ? o->qnodes : o->wide);
    h.nodes8 = (const float4*)o->w8nodes;
    h.leaves = o->leaves;
    h.nodeCount = o->nodeCount;
    h.geomType = geomType;
    h.primToLeaf = o->primToLeaf;
    h.flags = o->leafCount > count ? kHeaderSplit : 0u;
    if (e == cudaSuccess) e = cudaMemcpy(o->dHeader, &h, sizeof(h), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
        cudaFree(o->dHeader);
        cudaFree(o->nodes);
        cudaFree(o->wide);
        cudaFree(o->qnodes);
        cudaFree(o->w8nodes);
        cudaFree(o->leaves);
        cudaFree(o->parents);
        cudaFree(o->primToLeaf);
        cudaFree(o->inv64);
        cudaFree(o->fwd32);
        delete o;
        logf(GRT_LOG_ERROR, "allocation of a BVH with %u primitives failed: %s", count, cudaGetErrorString(e));
        return GRT_ERROR_OUT_OF_MEMORY;
    }
    registerBvh(o);
    if (quant) g_quantGeometries.fetch_add(1, std::memory_order_relaxed);
    *out = o;
    return GRT_SUCCESS;
}

static void destroyBvhObject(BvhObject* o) {
    if (o->quant) g_quantGeometries.fetch_sub(1, std::memory_order_relaxed);
    unregisterBvh(o->dHeader);
    cudaFree(o->dHeader);
    cudaFree(o->nodes);
    cudaFree(o->wide);
    cudaFree(o->qnodes);
    cudaFree(o->w8nodes);
    cudaFree(o->leaves);
    cudaFree(o->parents);
    cudaFree(o->primToLeaf);
    cudaFree(o->inv64);
    cudaFree(o->fwd32);
    delete o;
}

// Morton codes and their sort over the centroids already in temp (count >= 1).
static grtError sortCodes(Context* ctx, BvhObject* o, const BuildLayout& L, char* temp, cudaStream_t s) {
    const uint32_t n = o->leafCount;
    const float4* cen = (const float4*)(temp + L.centroids);
    const uint32_t* bounds = (const uint32_t*)(temp + L.bounds);
    const SortScratch S = sortScratch(temp + L.hist, n);
    uint32_t* const vals[2] = {(uint32_t*)(temp + L.vals[0]), (uint32_t*)(temp + L.vals[1])};
    grtError err;
    if (o->mortonBits == 30) {
        uint32_t* const keys[2] = {(uint32_t*)(temp + L.keys[0]), (uint32_t*)(temp + L.keys[1])};
        mortonKernel<uint32_t, 10><<<countBlocks(ctx, n), kCountThreads, 0, s>>>(cen, n, bounds, keys[0], S.hist);
        GRT_LAUNCH_CHECK();
        err = sortPasses<uint32_t>(ctx, keys, vals, n, L.passes, S, true, s);
    } else {
        unsigned long long* const keys[2] = {(unsigned long long*)(temp + L.keys[0]),
                                             (unsigned long long*)(temp + L.keys[1])};
        mortonKernel<unsigned long long, 21><<<countBlocks(ctx, n), kCountThreads, 0, s>>>(cen, n, bounds, keys[0],
                                                                                         S.hist);
        GRT_LAUNCH_CHECK();
        err = sortPasses<unsigned long long>(ctx, keys, vals, n, L.passes, S, true, s);
    }
    if (err != GRT_SUCCESS) return err;
    noteLaunches(1);
    return GRT_SUCCESS;
}

// The emission's lists: those of the first launch's blocks, then of each further launch's.
static uint32_t emitLists(uint32_t n) {
    uint32_t total = 0;
    for (uint32_t lists = ceilDiv(std::max(n, 1u), kEmitLeaves);; lists = ceilDiv(lists, kTopFan)) {
        total += lists;
        if (lists == 1) return total;
    }
}
size_t emitTopBytes(uint32_t n) { return (size_t)emitLists(n) * (kTopMax * sizeof(uint4) + sizeof(uint4)); }

// Emission and fit over the sorted codes (P.n >= 2, P.sortedPrims their order).
template <typename K, int KIND>
static grtError launchEmitFitT(Context* c, BvhObject* o, const BuildLayout& L, char* temp, const FitParams& P,
                               cudaStream_t s) {
    EmitParams E;
    E.fit = P;
    E.parents = (uint32_t*)o->parents;
    const K* keys = (const K*)(temp + L.keys[L.finalBuf]);
    grtError e = allowSmem(emitTopKernel<K, KIND>, sizeof(TopShared));
    if (e != GRT_SUCCESS) return e;
    uint32_t lists = ceilDiv(P.n, kEmitLeaves);
    TopLists in;
    in.tops = (uint4*)(temp + L.tops);
    in.counts = (uint32_t*)(in.tops + (size_t)emitLists(P.n) * kTopMax);
    emitFitKernel<K, KIND><<<lists, kEmitLeaves, 0, s>>>(E, keys, in);
    GRT_LAUNCH_CHECK();  // a further launch reads the lists and nodes of the one before
    noteLaunches(1);
    while (lists > 1) {
        const TopLists out{in.tops + (size_t)lists * kTopMax, in.counts + lists};
        const uint32_t next = ceilDiv(lists, kTopFan);
        emitTopKernel<K, KIND><<<next, kTopThreads, sizeof(TopShared), s>>>(E, keys, in, lists, out,
                                                                           &workspace(c)->error);
        GRT_LAUNCH_CHECK();
        noteLaunches(1);
        in = out;
        lists = next;
    }
    return GRT_SUCCESS;
}

template <int KIND>
static grtError launchEmitFit(Context* c, BvhObject* o, const BuildLayout& L, char* temp, const FitParams& P,
                              cudaStream_t s) {
    return o->mortonBits == 30 ? launchEmitFitT<uint32_t, KIND>(c, o, L, temp, P, s)
                               : launchEmitFitT<unsigned long long, KIND>(c, o, L, temp, P, s);
}

static grtError resetBuildScratch(Context* ctx, const BuildLayout& L, char* temp, uint32_t n, bool sorts,
                                  bool counts, cudaStream_t s) {
    BuildInit I;
    I.bounds = (uint32_t*)(temp + L.bounds);
    I.sortHead = (uint4*)(temp + L.hist);
    I.sortWords = sorts ? (kSortHeadBytes + lookBytes(n)) / sizeof(uint4) : 0;
    I.flags = (uint4*)(temp + L.flags);
    I.flagWords = counts ? alignUp(4 * (size_t)std::max(n, 1u), 16) / sizeof(uint4) : 0;
    const size_t words = std::max<size_t>(std::max(I.sortWords, I.flagWords), 6);
    buildInitKernel<<<std::min(ceilDiv(words, 256), 8u * (unsigned)std::max(1, smCount(ctx))), 256, 0, s>>>(I);
    GRT_LAUNCH_CHECK();
    noteLaunches(1);
    return GRT_SUCCESS;
}

// ======================================================================= clustering builds
// A geometry's build method is fixed when it is created: 0 = LBVH (GRT_BUILD_PREFER_FAST),
// kSubtreeMethod = clustering inside the LBVH's subtrees (cluster.cuh), else PLOC with
// this search radius (ploc.cuh).
constexpr uint32_t kSubtreeMethod = 0xFFFFu;
static uint32_t buildMethod(const grtBuildOptions* opt) {
    return opt ? opt->buildFlags &
                     ~(uint32_t)(GRT_BUILD_QUANTIZED_NODES | GRT_BUILD_WIDE8_NODES | GRT_BUILD_SPLIT_TRIANGLES)
               : 0u;
}
static bool quantFlag(const grtBuildOptions* opt) { return opt && (opt->buildFlags & GRT_BUILD_QUANTIZED_NODES); }
static bool wide8Flag(const grtBuildOptions* opt) { return opt && (opt->buildFlags & GRT_BUILD_WIDE8_NODES); }
static uint32_t clusterRadius(const grtBuildOptions* opt) {
    const uint32_t m = buildMethod(opt);
    if (m == GRT_BUILD_PREFER_FAST) return 0;
    if (m == GRT_BUILD_CLUSTER_SUBTREES) return kSubtreeMethod;
    return m == GRT_BUILD_PREFER_BALANCED ? 8u : 32u;
}
static bool validBuildFlags(const grtBuildOptions* opt) {
    return !opt || (buildMethod(opt) <= 3u && !(quantFlag(opt) && wide8Flag(opt)));
}
static bool splitFlag(const grtBuildOptions* opt) { return opt && (opt->buildFlags & GRT_BUILD_SPLIT_TRIANGLES); }
// The split bit is for triangle meshes, with a factor in [0, 1] (0 = 0.5).
static bool validSplit(const grtBuildOptions* opt, uint32_t primType) {
    if (!splitFlag(opt)) return true;
    return primType == GRT_PRIMITIVE_TRIANGLE_MESH && opt->splitFactor >= 0.f && opt->splitFactor <= 1.f;
}
// The split factor of a split build (0 selects 0.5), and its extra references for n
// triangles: floor(factor * n).
static double splitFactorOf(const grtBuildOptions* opt) {
    return opt->splitFactor == 0.f ? 0.5 : (double)opt->splitFactor;
}
static uint32_t splitBudgetOf(uint32_t n, const grtBuildOptions* opt) {
    if (!splitFlag(opt)) return 0;
    return (uint32_t)std::floor(splitFactorOf(opt) * (double)n);
}
// Leaf count of a build: the primitives plus the split references; false past 2^31 - 2.
static bool leafCountOf(uint32_t n, const grtBuildOptions* opt, uint32_t* m) {
    const uint64_t total = (uint64_t)n + splitBudgetOf(n, opt);
    if (total >= 0x7FFFFFFFull) return false;
    *m = (uint32_t)total;
    return true;
}

static std::mutex g_methodLock;
static std::unordered_map<const BvhObject*, uint32_t> g_clusterRadius;  // objects with a PLOC build

static uint32_t radiusOf(const BvhObject* o) {
    std::lock_guard<std::mutex> g(g_methodLock);
    auto it = g_clusterRadius.find(o);
    return it == g_clusterRadius.end() ? 0u : it->second;
}

bool buildsBySubtreeClustering(const BvhObject* o) { return radiusOf(o) == kSubtreeMethod; }

// PLOC scratch after the LBVH layout: two cluster arrays (32 B per cluster), the
// per-position neighbour words, per-block counts and the barrier words.
struct PlocLayout {
    size_t clusters, pick, counts, sync, total;
};
static PlocLayout plocLayout(const BuildLayout& L, uint32_t n) {
    PlocLayout P{};
    const size_t m = n ? n : 1;
    P.clusters = alignUp(L.total, 256);
    P.pick = P.clusters + alignUp(2 * 32 * m, 256);
    P.counts = P.pick + alignUp(4 * m, 256);
    P.sync = P.counts + alignUp(8 * (size_t)ceilDiv(m, kPlocThreads), 256);
    P.total = P.sync + 256;
    return P;
}

// Per-geometry build: the LBVH topology into the temporary arrays (one thread per
// internal node), the arrival counters zeroed.
template <typename K>
__global__ void clusterTopologyKernel(ClusterParams C, const K* __restrict__ sortedKeys) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < C.n) karrasTopology<false>(sortedKeys, (int)i, C);
}

constexpr int kClusterThreads = 256;

__global__ void __launch_bounds__(kClusterThreads) clusterWalkKernel(ClusterParams C) {
    __shared__ ClusterWarpList lists[kClusterThreads / 32];
    const uint32_t begin = blockIdx.x * blockDim.x;
    clusterRange(C, begin, min(C.n, begin + blockDim.x), lists);
}

// Subtree-clustering scratch after the LBVH layout: the LBVH's child words, parent
// entries, per-node records (leaf range, clusters passed up), the per-position cluster
// and number arrays and arrival counters (72 B per primitive).
struct SubtreeLayout {
    size_t child, parent, record, clusters, freeIds, flags, total;
};
static SubtreeLayout subtreeLayout(const BuildLayout& L, uint32_t n) {
    SubtreeLayout Q{};
    const size_t m = n ? n : 1;
    Q.child = alignUp(L.total, 256);
    Q.parent = Q.child + alignUp(8 * m, 256);
    Q.record = Q.parent + alignUp(4 * 2 * m, 256);
    Q.clusters = Q.record + alignUp(16 * m, 256);
    Q.freeIds = Q.clusters + alignUp(32 * m, 256);
    Q.flags = Q.freeIds + alignUp(4 * m, 256);
    Q.total = Q.flags + alignUp(4 * m, 256);
    return Q;
}

// The subtree clustering over the sorted leaves (n >= 2): the LBVH topology into the
// scratch, then the bottom-up walk, which writes the final child words and parent links.
static grtError launchSubtreeCluster(Context* c, BvhObject* o, const BuildLayout& L, char* t, const PrimSource& S,
                                     const uint32_t* sorted, const void* sortedKeys, cudaStream_t s) {
    const uint32_t n = o->leafCount;
    const SubtreeLayout Q = subtreeLayout(L, n);
    ClusterParams C{};
    C.src = S;
    C.n = n;
    C.sortedPrims = sorted;
    C.topoChild = (uint2*)(t + Q.child);
    C.topoParent = (uint32_t*)(t + Q.parent);
    C.record = (uint4*)(t + Q.record);
    C.clusters = (float4*)(t + Q.clusters);
    C.freeIds = (uint32_t*)(t + Q.freeIds);
    C.flags = (uint32_t*)(t + Q.flags);
    C.nodes = (float4*)o->nodes;
    C.parents = (uint32_t*)o->parents;
    C.error = &workspace(c)->error;
    if (o->mortonBits == 30)
        clusterTopologyKernel<uint32_t><<<ceilDiv(n, 256), 256, 0, s>>>(C, (const uint32_t*)sortedKeys);
    else
        clusterTopologyKernel<unsigned long long><<<ceilDiv(n, 256), 256, 0, s>>>(
            C, (const unsigned long long*)sortedKeys);
    GRT_LAUNCH_CHECK();
    clusterWalkKernel<<<ceilDiv(n, kClusterThreads), kClusterThreads, 0, s>>>(C);
    GRT_LAUNCH_CHECK();
    noteLaunches(2);
    return GRT_SUCCESS;
}

// The clustering kernel over the sorted leaves: writes child words and parent links.
static grtError launchPloc(Context* c, BvhObject* o, const BuildLayout& L, char* t, const PrimSource& S,
                           const uint32_t* sorted, uint32_t radius, cudaStream_t s) {
    const uint32_t n = o->leafCount;
    const PlocLayout Q = plocLayout(L, n);
    PlocParams P{};
    P.src = S;
    P.n = n;
    P.radius = radius;
    P.sortedPrims = sorted;
    P.clusters[0] = (float4*)(t + Q.clusters);
    P.clusters[1] = P.clusters[0] + 2 * (size_t)n;
    P.pick = (uint32_t*)(t + Q.pick);
    P.blockCounts = (uint2*)(t + Q.counts);
    P.sync = (uint32_t*)(t + Q.sync);
    P.nodes = (float4*)o->nodes;
    P.parents = (uint32_t*)o->parents;
    P.error = &workspace(c)->error;
    P.waitNs = 2000000000ull;
    // below this many clusters one block is faster than the grid: a grid iteration costs
    // about 12 us (r = 8) to 24 us (r = 32) of round trips and barriers, the block's
    // neighbour search about 2r area tests per cluster on one SM
    P.finishAt = std::min<uint32_t>(kPlocFinishMax, 49152u / radius);
    const uint32_t blocks = std::min<uint32_t>(ceilDiv(n, kPlocThreads), 2u * (uint32_t)std::max(smCount(c), 1));
    GRT_CUDA(cudaMemsetAsync(P.sync, 0, 32, s));
    plocKernel<<<blocks, kPlocThreads, plocSmemBytes(radius), s>>>(P);
    GRT_LAUNCH_CHECK();
    plocFinishKernel<<<1, kPlocFinishThreads, plocFinishSmemBytes(), s>>>(P);
    GRT_LAUNCH_CHECK();
    noteLaunches(2);
    return GRT_SUCCESS;
}

// Bytes of the method's temporary layout for leaf count n (the LBVH layout L plus the
// clustering scratch).
static size_t methodTempBytes(const BuildLayout& L, uint32_t n, uint32_t radius) {
    return radius == kSubtreeMethod ? subtreeLayout(L, n).total : radius ? plocLayout(L, n).total : L.total;
}

// Triangle-splitting scratch after the method's: the scene bounds and the two totals,
// per-triangle counts, per-block sums and the references (32 B each).
struct SplitLayout {
    size_t misc, counts, firstSlot, weightSums, blockSums, slotTriangle, refs, total;
};
static SplitLayout splitLayout(size_t base, uint32_t n, uint32_t m) {
    SplitLayout Q{};
    const size_t blocks = ceilDiv(std::max(n, 1u), kSplitThreads);
    Q.misc = alignUp(base, 256);
    Q.counts = Q.misc + 256;
    Q.firstSlot = Q.counts + alignUp(4 * (size_t)std::max(n, 1u), 256);
    Q.weightSums = Q.firstSlot + alignUp(4 * (size_t)std::max(n, 1u), 256);
    Q.blockSums = Q.weightSums + alignUp(8 * blocks, 256);
    Q.slotTriangle = Q.blockSums + alignUp(4 * blocks, 256);
    Q.refs = Q.slotTriangle + alignUp(4 * (size_t)std::max(m, 1u), 256);
    Q.total = Q.refs + alignUp(32 * (size_t)std::max(m, 1u), 256);
    return Q;
}
static SplitLayout splitLayoutOf(const BvhObject* o, const BuildLayout& L, uint32_t radius) {
    return splitLayout(methodTempBytes(L, o->leafCount, radius), o->primCount, o->leafCount);
}

// Splitting kernels of per-geometry builds (split.cuh): a chunk of kSplitThreads
// triangles (references) per block.
__device__ __forceinline__ void chunkOf(uint32_t count, uint32_t* b0, uint32_t* b1) {
    *b0 = blockIdx.x * blockDim.x;
    *b1 = min(count, *b0 + blockDim.x);
}

__global__ void __launch_bounds__(kSplitThreads) splitBoundsKernel(SplitParams P) {
    uint32_t b0, b1;
    chunkOf(P.n, &b0, &b1);
    splitBoundsRange(P, b0, b1);
}

__global__ void __launch_bounds__(kSplitThreads) splitWeightKernel(SplitParams P) {
    uint32_t b0, b1;
    chunkOf(P.n, &b0, &b1);
    splitWeightRange(P, blockIdx.x, b0, b1);
}

__global__ void __launch_bounds__(kSplitScanThreads) splitScanWeightsKernel(SplitParams P) {
    splitScanWeights(P, P.blocks);
}

__global__ void __launch_bounds__(kSplitThreads) splitCountKernel(SplitParams P) {
    uint32_t b0, b1;
    chunkOf(P.n, &b0, &b1);
    splitCountRange(P, blockIdx.x, b0, b1);
}

__global__ void __launch_bounds__(kSplitScanThreads) splitScanKernel(SplitParams P) {
    scanBlockSums<uint32_t>(P.blockSums, P.blocks, nullptr);
}

__global__ void __launch_bounds__(kSplitThreads) splitSlotsKernel(SplitParams P) {
    uint32_t b0, b1;
    chunkOf(P.n, &b0, &b1);
    splitSlotsRange(P, blockIdx.x, b0, b1);
}

__global__ void __launch_bounds__(kSplitThreads) splitEmitKernel(SplitParams P) {
    uint32_t r0, r1;
    chunkOf(P.n + P.budget, &r0, &r1);
    splitEmitRange<true>(P, r0, r1);
}

// The splitting launches of a split build (o->primCount >= 1 triangles): references,
// their centroids and the centroid bounds, in the scratch the rest of the build reads.
static grtError launchSplit(Context* c, BvhObject* o, const BuildLayout& L, char* t, const PrimSource& S,
                            uint32_t radius, cudaStream_t s) {
    const SplitLayout Q = splitLayoutOf(o, L, radius);
    SplitParams P{};
    P.src = S;
    P.n = o->primCount;
    P.budget = o->splitBudget;
    P.sceneBounds = (uint32_t*)(t + Q.misc);
    P.totals = (unsigned long long*)(t + Q.misc + 32);
    P.counts = (uint32_t*)(t + Q.counts);
    P.weightSums = (unsigned long long*)(t + Q.weightSums);
    P.blockSums = (uint32_t*)(t + Q.blockSums);
    P.firstSlot = (uint32_t*)(t + Q.firstSlot);
    P.slotTriangle = (uint32_t*)(t + Q.slotTriangle);
    P.blocks = ceilDiv(P.n, kSplitThreads);
    P.refs = (float4*)(t + Q.refs);
    P.centroids = (float4*)(t + L.centroids);
    P.centroidBounds = (uint32_t*)(t + L.bounds);
    P.error = &workspace(c)->error;
    GRT_CUDA(cudaMemsetAsync(t + Q.misc, 0xFF, 12, s));       // running minima start at the top
    GRT_CUDA(cudaMemsetAsync(t + Q.misc + 12, 0x00, 36, s));  // maxima at the bottom, totals at 0
    splitBoundsKernel<<<P.blocks, kSplitThreads, 0, s>>>(P);
    GRT_LAUNCH_CHECK();
    splitWeightKernel<<<P.blocks, kSplitThreads, 0, s>>>(P);
    GRT_LAUNCH_CHECK();
    splitScanWeightsKernel<<<1, kSplitScanThreads, 0, s>>>(P);
    GRT_LAUNCH_CHECK();
    splitCountKernel<<<P.blocks, kSplitThreads, 0, s>>>(P);
    GRT_LAUNCH_CHECK();
    splitScanKernel<<<1, kSplitScanThreads, 0, s>>>(P);
    GRT_LAUNCH_CHECK();
    splitSlotsKernel<<<P.blocks, kSplitThreads, 0, s>>>(P);
    GRT_LAUNCH_CHECK();
    splitEmitKernel<<<ceilDiv((size_t)P.n + P.budget, kSplitThreads), kSplitThreads, 0, s>>>(P);
    GRT_LAUNCH_CHECK();
    noteLaunches(7);
    return GRT_SUCCESS;
}

// The launch sequence of a geometry BUILD (above kSmallBuild) or UPDATE on stream s:
// scratch reset, centroids and bounds, Morton codes, the radix passes, the hierarchy
// (Karras emission, or PLOC clustering when radius > 0), the fit.
static grtError issueGeometryBuild(Context* c, BvhObject* o, uint32_t op, const grtGeometryBuildInput* input,
                                   const BuildLayout& L, char* t, const PrimSource& S, cudaStream_t s,
                                   uint32_t radius = 0) {
    const uint32_t n = o->leafCount;
    const bool emits = op == GRT_BUILD_OPERATION_BUILD && radius == 0 && n >= 2;
    grtError e = resetBuildScratch(c, L, t, n, op == GRT_BUILD_OPERATION_BUILD, !emits, s);
    if (e != GRT_SUCCESS) return e;
    const uint32_t* sorted = nullptr;
    if (op == GRT_BUILD_OPERATION_BUILD) {
        if (o->split) {
            e = launchSplit(c, o, L, t, S, radius, s);
            if (e != GRT_SUCCESS) return e;
        } else {
            const unsigned blocks = std::min(ceilDiv(n, 256), 8u * (unsigned)std::max(1, smCount(c)));
            primCentroidKernel<<<blocks, 256, 0, s>>>(S, (float4*)(t + L.centroids),
                                                               (uint32_t*)(t + L.bounds));
            GRT_LAUNCH_CHECK();
            noteLaunches(1);
        }
        e = sortCodes(c, o, L, t, s);
        if (e != GRT_SUCCESS) return e;
        sorted = (const uint32_t*)(t + L.vals[L.finalBuf]);
        const void* sortedKeys = t + L.keys[L.finalBuf];
        if (radius == kSubtreeMethod && n >= 2) {
            e = launchSubtreeCluster(c, o, L, t, S, sorted, sortedKeys, s);
            if (e != GRT_SUCCESS) return e;
        } else if (radius != 0 && n >= 2) {
            e = launchPloc(c, o, L, t, S, sorted, radius, s);
            if (e != GRT_SUCCESS) return e;
        }
    }
    FitParams P{};
    P.src = S;
    P.n = n;
    P.sortedPrims = sorted;  // null for UPDATE: IDs come from the leaves
    P.nodes = (float4*)o->nodes;
    P.wide = (float4*)o->wide;
    P.leaves = o->leaves;
    P.primToLeaf = o->primToLeaf;
    P.parents = (const uint32_t*)o->parents;
    P.flags = (uint32_t*)(t + L.flags);
    P.header = o->dHeader;
    if (emits) {
        e = input->type == GRT_PRIMITIVE_TRIANGLE_MESH ? launchEmitFit<0>(c, o, L, t, P, s)
                                                       : launchEmitFit<1>(c, o, L, t, P, s);
        if (e != GRT_SUCCESS) return e;
        return launchNodeFormats(o, s);
    }
    if (input->type == GRT_PRIMITIVE_TRIANGLE_MESH)
        fitKernel<0><<<ceilDiv(n, 256), 256, 0, s>>>(P);
    else
        fitKernel<1><<<ceilDiv(n, 256), 256, 0, s>>>(P);
    GRT_LAUNCH_CHECK();
    noteLaunches(1);
    return launchNodeFormats(o, s);
}

// Repeated BUILDs of a geometry from the same buffers replay a CUDA graph of the launch
// sequence. Every kernel argument is a function of the build input (addresses, strides,
// counts), the temporary buffer, the object's own arrays, the device and the context's
// error word (the sort's and the emission's waits and checks latch there), so a graph
// captured once serves every later build with the same description: new vertex data in
// the same buffers is read by the replay. The graph is captured on a private stream and
// launched on the caller's; a different description captures again, and a caller's
// stream that is itself being captured gets the launches directly.
struct BuildKey {
    grtGeometryBuildInput input;
    const void* temp;
    const uint32_t* error;
    int device;
    uint32_t radius;
    bool operator==(const BuildKey& k) const { return std::memcmp(this, &k, sizeof(*this)) == 0; }
};
struct BuildGraph {
    BuildKey key;
    cudaGraphExec_t exec = nullptr;
    unsigned long long launches = 0;
    uint32_t builds = 0;  // issued without a graph
};
static std::mutex g_buildGraphLock;
static std::unordered_map<const BvhObject*, BuildGraph> g_buildGraphs;
unsigned long long threadLaunches();  // context.cu

static void eraseBuildGraph(std::unordered_map<const BvhObject*, BuildGraph>::iterator it) {
    if (it->second.exec) cudaGraphExecDestroy(it->second.exec);
    g_buildGraphs.erase(it);
}
static void dropBuildGraph(const BvhObject* o) {
    std::lock_guard<std::mutex> g(g_buildGraphLock);
    auto it = g_buildGraphs.find(o);
    if (it != g_buildGraphs.end()) eraseBuildGraph(it);
}

// A build in one block, which initialises its own scratch.
static grtError issueSmallBuild(Context* c, BvhObject* o, const grtGeometryBuildInput* input, const BuildLayout& L,
                                char* t, const PrimSource& S, cudaStream_t s) {
    BlockBuild B = blockBuildOf(c, o, L, t, input->type == GRT_PRIMITIVE_TRIANGLE_MESH ? 0u : 1u);
    B.src = S;
    return launchSmallBuild(B, s);
}

// The graph of a build's launches, counted as launched; null where it cannot be made.
static cudaGraphExec_t captureBuild(Context* c, BvhObject* o, const grtGeometryBuildInput* input, const BuildLayout& L,
                                    char* t, const PrimSource& S, uint32_t radius) {
    cudaStream_t cs = nullptr;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    cudaError_t ce = cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking);
    if (ce == cudaSuccess) {
        ce = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
        grtError e = ce == cudaSuccess
                         ? issueGeometryBuild(c, o, GRT_BUILD_OPERATION_BUILD, input, L, t, S, cs, radius)
                         : GRT_ERROR_CUDA;
        if (ce == cudaSuccess) ce = cudaStreamEndCapture(cs, &graph);
        if (e == GRT_SUCCESS && ce == cudaSuccess) ce = cudaGraphInstantiate(&exec, graph, 0);
        if (graph) cudaGraphDestroy(graph);
        cudaStreamDestroy(cs);
        if (e == GRT_SUCCESS && ce == cudaSuccess) return exec;
    }
    cudaGetLastError();
    if (exec) cudaGraphExecDestroy(exec);
    return nullptr;
}

static grtError replayOrCaptureBuild(Context* c, BvhObject* o, const grtGeometryBuildInput* input,
                                     const BuildLayout& L, char* t, const PrimSource& S, cudaStream_t s,
                                     uint32_t radius) {
    auto issue = [&](bool oneBlock) {
        const grtError e = oneBlock ? issueSmallBuild(c, o, input, L, t, S, s)
                                    : issueGeometryBuild(c, o, GRT_BUILD_OPERATION_BUILD, input, L, t, S, s, radius);
        if (e == GRT_SUCCESS) o->built = true;
        return e;
    };
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (s && cudaStreamIsCapturing(s, &cap) != cudaSuccess) cap = cudaStreamCaptureStatusActive;
    if (cap != cudaStreamCaptureStatusNone) return issue(false);  // the caller is capturing
    BuildKey key;
    std::memset(&key, 0, sizeof(key));
    key.input.type = input->type;  // only the fields the launches read
    if (input->type == GRT_PRIMITIVE_TRIANGLE_MESH)
        key.input.triangleMesh = input->triangleMesh;
    else
        key.input.aabbList = input->aabbList;
    key.temp = t;
    key.error = &workspace(c)->error;
    key.device = deviceOf(c);
    key.radius = radius;
    const bool small = radius == 0 && !o->split && o->leafCount <= kSmallGraph;
    std::lock_guard<std::mutex> g(g_buildGraphLock);
    auto it = g_buildGraphs.find(o);
    if (it != g_buildGraphs.end() && !(it->second.key == key)) {
        eraseBuildGraph(it);
        it = g_buildGraphs.end();
    }
    if (it == g_buildGraphs.end()) {
        BuildGraph bg;
        bg.key = key;
        it = g_buildGraphs.emplace(o, bg).first;
    }
    BuildGraph& G = it->second;
    if (!G.exec) {
        if (small && G.builds < kDirectBuilds) {
            ++G.builds;
            return issue(o->leafCount <= kSmallFirst);
        }
        const unsigned long long before = threadLaunches();
        G.exec = captureBuild(c, o, input, L, t, S, radius);
        if (!G.exec) return issue(false);  // no graph: the launches go straight to s
        G.launches = threadLaunches() - before;  // counted once at capture, for this first replay
    } else {
        noteLaunches((unsigned)G.launches);
    }
    GRT_CUDA(cudaGraphLaunch(G.exec, s));
    o->built = true;
    return GRT_SUCCESS;
}

}  // namespace grt

using namespace grt;

extern "C" {

grtError grtGetGeometryBuildTemporaryBufferSize(grtContext ctx, const grtGeometryBuildInput* input,
                                                const grtBuildOptions* options, size_t* sizeBytes) {
    uint32_t n = 0;
    if (!ctx || !sizeBytes) return GRT_ERROR_INVALID_PARAMETER;
    grtError e = validateGeometryInput(input, &n);
    if (e != GRT_SUCCESS) return e;
    uint32_t m = 0;
    if (!validBuildFlags(options) || !validSplit(options, input->type) || !leafCountOf(n, options, &m))
        return GRT_ERROR_INVALID_PARAMETER;
    const BuildLayout L = buildLayout(m, resolveMortonBits(m, options), false);
    const size_t bytes = methodTempBytes(L, m, clusterRadius(options));
    *sizeBytes = splitFlag(options) ? splitLayout(bytes, n, m).total : bytes;
    return GRT_SUCCESS;
}

grtError grtCreateGeometry(grtContext ctx, const grtGeometryBuildInput* input, const grtBuildOptions* options,
                           grtGeometry* out) {
    uint32_t n = 0;
    if (!ctx || !out) return GRT_ERROR_INVALID_PARAMETER;
    grtError e = validateGeometryInput(input, &n);
    if (e != GRT_SUCCESS) return e;
    uint32_t m = 0;
    if (!validBuildFlags(options) || !validSplit(options, input->type) || !leafCountOf(n, options, &m))
        return GRT_ERROR_INVALID_PARAMETER;
    if (clusterRadius(options) && m > kPlocIndex) return GRT_ERROR_INVALID_PARAMETER;
    BvhObject* o = nullptr;
    e = createBvhObject(n, input->type, input->geomType, resolveMortonBits(m, options), &o, quantFlag(options),
                        wide8Flag(options), m);
    if (e != GRT_SUCCESS) return e;
    o->split = splitFlag(options);
    o->splitFactor = o->split ? (float)splitFactorOf(options) : 0.f;
    o->splitBudget = m - n;
    if (clusterRadius(options)) {
        // the finishing block's shared memory is above the default limit
        cudaError_t ce = cudaFuncSetAttribute(plocFinishKernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)plocFinishSmemBytes());
        if (ce != cudaSuccess) {
            cudaGetLastError();
            destroyBvhObject(o);
            logf(GRT_LOG_ERROR, "clustering build: %s", cudaGetErrorString(ce));
            return GRT_ERROR_CUDA;
        }
        std::lock_guard<std::mutex> g(g_methodLock);
        g_clusterRadius[o] = clusterRadius(options);
    }
    *out = reinterpret_cast<grtGeometry>(o->dHeader);
    return GRT_SUCCESS;
}

grtError grtBuildGeometry(grtContext ctx, uint32_t op, const grtGeometryBuildInput* input,
                          const grtBuildOptions* options, void* temp, void* stream, grtGeometry geom) {
    uint32_t n = 0;
    if (!ctx || !geom) return GRT_ERROR_INVALID_PARAMETER;
    grtError e = validateGeometryInput(input, &n);
    if (e != GRT_SUCCESS) return e;
    BvhObject* o = findBvh(geom);
    if (!o || o->primType == kPrimScene || o->primType != input->type || o->primCount != n)
        return GRT_ERROR_INVALID_PARAMETER;
    if (op != GRT_BUILD_OPERATION_BUILD && op != GRT_BUILD_OPERATION_UPDATE) return GRT_ERROR_INVALID_PARAMETER;
    if (op == GRT_BUILD_OPERATION_UPDATE && !o->built) return GRT_ERROR_NOT_BUILT;
    if (op == GRT_BUILD_OPERATION_UPDATE && o->split) return GRT_ERROR_INVALID_PARAMETER;
    if (n > 0 && (!temp || ((uintptr_t)temp & 15))) return GRT_ERROR_INVALID_PARAMETER;
    if (options && options->mortonBits && resolveMortonBits(o->leafCount, options) != o->mortonBits)
        return GRT_ERROR_INVALID_PARAMETER;
    if (options && (splitFlag(options) != o->split || (o->split && (float)splitFactorOf(options) != o->splitFactor)))
        return GRT_ERROR_INVALID_PARAMETER;
    const uint32_t radius = radiusOf(o);
    if (!validBuildFlags(options) || (options && clusterRadius(options) != radius)) return GRT_ERROR_INVALID_PARAMETER;
    if (options && (quantFlag(options) != o->quant || wide8Flag(options) != o->wide8))
        return GRT_ERROR_INVALID_PARAMETER;
    Context* c = asContext(ctx);
    cudaStream_t s = (cudaStream_t)stream;
    o->geomType = input->geomType;
    if (input->type == GRT_PRIMITIVE_TRIANGLE_MESH) o->vertexCount = input->triangleMesh.vertexCount;
    if (n == 0) {
        o->built = true;
        return GRT_SUCCESS;
    }
    const BuildLayout L = buildLayout(o->leafCount, o->mortonBits, false);
    char* t = (char*)temp;
    PrimSource S = primSource(input, n);
    if (o->split) {  // the build reads the references the splitting writes
        S.kind = 2;
        S.count = o->leafCount;
        S.refs = (const float4*)(t + splitLayoutOf(o, L, radius).refs);
    }
    if (op == GRT_BUILD_OPERATION_BUILD && n <= kSmallBuild && radius == 0 && !o->split) {
        e = issueSmallBuild(c, o, input, L, t, S, s);
        if (e == GRT_SUCCESS) o->built = true;
        return e;
    }
    if (op == GRT_BUILD_OPERATION_BUILD) return replayOrCaptureBuild(c, o, input, L, t, S, s, radius);
    e = issueGeometryBuild(c, o, op, input, L, t, S, s);
    if (e != GRT_SUCCESS) return e;
    o->built = true;
    return GRT_SUCCESS;
}

grtError grtDestroyGeometry(grtContext ctx, grtGeometry geom) {
    BvhObject* o = findBvh(geom);
    if (!ctx || !o || o->primType == kPrimScene) return GRT_ERROR_INVALID_PARAMETER;
    dropBuildGraph(o);
    {
        std::lock_guard<std::mutex> g(g_methodLock);
        g_clusterRadius.erase(o);
    }
    destroyBvhObject(o);
    return GRT_SUCCESS;
}

static grtError validateSceneInput(const grtSceneBuildInput* in) {
    if (!in) return GRT_ERROR_INVALID_PARAMETER;
    if (in->instanceCount != in->frameCount) return GRT_ERROR_INVALID_PARAMETER;
    if (in->instanceCount && (!in->instances || !in->instanceFrames)) return GRT_ERROR_INVALID_PARAMETER;
    if (in->instanceCount >= 0x7FFFFFFFu) return GRT_ERROR_INVALID_PARAMETER;
    return GRT_SUCCESS;
}

grtError grtGetSceneBuildTemporaryBufferSize(grtContext ctx, const grtSceneBuildInput* input,
                                             const grtBuildOptions* options, size_t* sizeBytes) {
    if (!ctx || !sizeBytes) return GRT_ERROR_INVALID_PARAMETER;
    grtError e = validateSceneInput(input);
    if (e != GRT_SUCCESS) return e;
    *sizeBytes = buildLayout(input->instanceCount, resolveMortonBits(input->instanceCount, options), true).total;
    return GRT_SUCCESS;
}

grtError grtCreateScene(grtContext ctx, const grtSceneBuildInput* input, const grtBuildOptions* options,
                        grtScene* out) {
    if (!ctx || !out) return GRT_ERROR_INVALID_PARAMETER;
    grtError e = validateSceneInput(input);
    if (e != GRT_SUCCESS) return e;
    BvhObject* o = nullptr;
    if (!validBuildFlags(options)) return GRT_ERROR_INVALID_PARAMETER;
    e = createBvhObject(input->instanceCount, kPrimScene, 0, resolveMortonBits(input->instanceCount, options), &o,
                        false, wide8Flag(options));
    if (e != GRT_SUCCESS) return e;
    *out = reinterpret_cast<grtScene>(o->dHeader);
    return GRT_SUCCESS;
}

grtError grtBuildScene(grtContext ctx, uint32_t op, const grtSceneBuildInput* input, const grtBuildOptions* options,
                       void* temp, void* stream, grtScene scene) {
    if (!ctx || !scene) return GRT_ERROR_INVALID_PARAMETER;
    grtError e = validateSceneInput(input);
    if (e != GRT_SUCCESS) return e;
    BvhObject* o = findBvh(scene);
    if (!o || o->primType != kPrimScene || o->primCount != input->instanceCount) return GRT_ERROR_INVALID_PARAMETER;
    if (op != GRT_BUILD_OPERATION_BUILD && op != GRT_BUILD_OPERATION_UPDATE) return GRT_ERROR_INVALID_PARAMETER;
    const uint32_t n = o->primCount;
    if (n > 0 && (!temp || ((uintptr_t)temp & 15))) return GRT_ERROR_INVALID_PARAMETER;
    if (options && (!validBuildFlags(options) || wide8Flag(options) != o->wide8)) return GRT_ERROR_INVALID_PARAMETER;
    Context* c = asContext(ctx);
    cudaStream_t s = (cudaStream_t)stream;
    if (n == 0) {
        o->built = true;
        return GRT_SUCCESS;
    }
    // An update of a scene rebuilds its (small) top level: instance frames may move freely.
    const BuildLayout L = buildLayout(n, o->mortonBits, true);
    char* t = (char*)temp;
    InstanceInput I{};
    I.instances = input->instances;
    I.frames = input->instanceFrames;
    I.count = n;
    I.boxes = (float4*)(t + L.extra);
    I.records = (InstanceRecord*)(t + L.extra + alignUp(32 * (size_t)n, 256));
    I.centroids = (float4*)(t + L.centroids);
    I.bounds = (uint32_t*)(t + L.bounds);
    I.inv64 = o->inv64;
    I.fwd32 = o->fwd32;
    I.wide8 = o->wide8 ? 1u : 0u;
    I.error = &workspace(c)->error;
    if (n <= kSmallScene) {
        BlockBuild B = blockBuildOf(c, o, L, t, 2u);
        B.instBoxes = I.boxes;
        B.instRecords = I.records;
        if (B.bits == 30) {
            const size_t smem = smallBuildSmemBytes<uint32_t>();
            e = allowSmem(smallSceneKernel<uint32_t, 10>, smem);
            if (e != GRT_SUCCESS) return e;
            smallSceneKernel<uint32_t, 10><<<1, kSmallSceneThreads, smem, s>>>(B, I);
        } else {
            const size_t smem = smallBuildSmemBytes<unsigned long long>();
            e = allowSmem(smallSceneKernel<unsigned long long, 21>, smem);
            if (e != GRT_SUCCESS) return e;
            smallSceneKernel<unsigned long long, 21><<<1, kSmallSceneThreads, smem, s>>>(B, I);
        }
        GRT_LAUNCH_CHECK();
        noteLaunches(1);
        o->built = true;
        return GRT_SUCCESS;
    }
    e = resetBuildScratch(c, L, t, n, true, false, s);
    if (e != GRT_SUCCESS) return e;
    instanceSetupKernel<<<ceilDiv(n, 128), 128, 0, s>>>(I);
    GRT_LAUNCH_CHECK();
    noteLaunches(1);
    e = sortCodes(c, o, L, t, s);
    if (e != GRT_SUCCESS) return e;
    FitParams P{};
    P.n = n;
    P.sortedPrims = (const uint32_t*)(t + L.vals[L.finalBuf]);
    P.nodes = (float4*)o->nodes;
    P.wide = (float4*)o->wide;
    P.leaves = o->leaves;
    P.header = o->dHeader;
    P.primToLeaf = o->primToLeaf;
    P.instBoxes = I.boxes;
    P.instRecords = I.records;
    e = launchEmitFit<2>(c, o, L, t, P, s);
    if (e != GRT_SUCCESS) return e;
    e = launchNodeFormats(o, s);
    if (e != GRT_SUCCESS) return e;
    o->built = true;
    return GRT_SUCCESS;
}

grtError grtDestroyScene(grtContext ctx, grtScene scene) {
    BvhObject* o = findBvh(scene);
    if (!ctx || !o || o->primType != kPrimScene) return GRT_ERROR_INVALID_PARAMETER;
    destroyBvhObject(o);
    return GRT_SUCCESS;
}

grtError grtSortTemporaryBufferSize(uint32_t count, uint32_t keyBits, size_t* sizeBytes) {
    if (!sizeBytes || (keyBits != 32 && keyBits != 64)) return GRT_ERROR_INVALID_PARAMETER;
    const size_t kb = keyBits / 8;
    *sizeBytes = alignUp(kb * std::max(count, 1u), 256) + alignUp(4 * (size_t)std::max(count, 1u), 256) +
                 sortScratchBytes(count);
    return GRT_SUCCESS;
}

grtError grtSortPairs(grtContext ctx, void* keys, uint32_t* values, uint32_t count, uint32_t keyBits,
                      uint32_t significantBits, void* temp, void* stream) {
    if (!ctx || (keyBits != 32 && keyBits != 64) || significantBits == 0 || significantBits > keyBits)
        return GRT_ERROR_INVALID_PARAMETER;
    if (count == 0) return GRT_SUCCESS;
    if (!keys || !values || !temp || ((uintptr_t)temp & 15)) return GRT_ERROR_INVALID_PARAMETER;
    const size_t kb = keyBits / 8;
    char* t = (char*)temp;
    void* k1 = t;
    uint32_t* v1 = (uint32_t*)(t + alignUp(kb * count, 256));
    void* scratch = t + alignUp(kb * count, 256) + alignUp(4 * (size_t)count, 256);
    cudaStream_t s = (cudaStream_t)stream;
    int fb = 0;
    grtError e = radixSort(asContext(ctx), keys, k1, values, v1, count, (int)kb, (int)significantBits, scratch, s, &fb);
    if (e != GRT_SUCCESS) return e;
    if (fb == 1) {
        const unsigned blocks = std::min(ceilDiv(count, 256), 8u * (unsigned)std::max(1, smCount(asContext(ctx))));
        if (kb == 4)
            copyPairsKernel<<<blocks, 256, 0, s>>>((uint32_t*)keys, (const uint32_t*)k1, values, v1, count);
        else
            copyPairsKernel<<<blocks, 256, 0, s>>>((unsigned long long*)keys, (const unsigned long long*)k1, values, v1,
                                                   count);
        GRT_LAUNCH_CHECK();
        noteLaunches(1);
    }
    return GRT_SUCCESS;
}

}  // extern "C"
