// Hierarchy emission and bottom-up fit of a linear BVH in one pass over the sorted codes, of a
// launch over blocks of leaves and a few that join what remains.
//
// The tree and its numbering are Karras's (HPG 2012), found from the leaves upwards
// (Apetrei, "Fast and Simple Agglomerative LBVH Construction", CGVC 2014). With delta(i) the
// length of the common prefix of the codes at sorted positions i and i + 1 (equal codes
// compared by position), a subtree over positions [l, r] is the left child of its parent
// when delta(r) > delta(l - 1), else the right child; its parent splits after r, or after
// l - 1; and its own number is r, or l (0 for the root). So the two subtrees either side
// of a split meet in that split's word, and the second to arrive, which then knows both
// boxes and both ranges, writes the parent: its binary node, its 4-wide node, the links.
//
// What bounds it: the output, 64 + 128 + 48 + 12 bytes a triangle. A block takes kEmitLeaves
// consecutive leaves and builds every node whose range lies among them in shared memory (a
// node's number is an end of its range, so these nodes lie together in the node arrays
// too) and writes them with whole rows of float4 in order. The subtrees it ends with, whose
// parents reach outside the block, are few: at most one per level of the tree on either
// side (kTopMax). Further launches join the lists of kTopFan blocks the same way, until one
// holds the root. No subtree waits for another and nothing is handed over inside a launch.
//
// Measured, 1,234,567 triangles with 63-bit codes and 131,072 with 30 (launch by launch, cold):
// a search for every node's range, then a walk from every leaf with an acquire-release
// atomic and four dependent loads a level and 8-byte stores into the nodes, 309 and 61 us;
// blocks of 256 whose remaining subtrees met in global memory, 225 and 55 us (390 with 512:
// the climbing threads held their blocks' SMs), 189 and 58 with the climb a launch of its
// own; as it is now 132 + 15 + 17 + 18 and 18 + 14 + 16 us. The first launch writes 2.2
// TB/s; the further ones are one chain of loads, meetings and stores each.
#pragma once

#include "lbvh.cuh"

namespace grt {

// Leaves of a block, one per thread: 512 leave half as many lists as 256 (builds of 331
// against 345 us, 86 against 91 at 131,072 triangles) and still fit three blocks on an SM.
constexpr int kEmitLeaves = 512;
constexpr uint32_t kTopFan = 16;  // lists joined by a block of a further launch
// Subtrees a list can hold: the largest ones inside a range of leaves, at most one per level
// either side. Levels have different common prefixes: below 63 bits of the code, then 32 of
// the position.
constexpr uint32_t kTopMax = 192;
constexpr uint32_t kTopCap = kTopFan * kTopMax;
constexpr int kTopThreads = 1024;

// Lists of subtrees {child word, l, r, 0} in the order of their leaves, kTopMax entries each.
struct TopLists {
    uint4* tops;
    uint32_t* counts;
};

struct EmitParams {
    FitParams fit;  // sortedPrims, nodes, wide, leaves, primToLeaf, header, instances
    uint32_t* parents;
};

// Common prefix of codes a and b at positions i != j.
template <typename K>
__device__ __forceinline__ int prefixOf(K a, K b, uint32_t i, uint32_t j) {
    if (a != b) return sizeof(K) == 4 ? __clz((int)(uint32_t)(a ^ b)) : __clzll((long long)(a ^ b));
    return (int)sizeof(K) * 8 + __clz((int)(i ^ j));
}

// Sorted position k's primitive (an order left incomplete by an expired wait of the sort must
// not lead outside the input).
__device__ __forceinline__ uint32_t sortedItem(const FitParams& P, uint32_t k) {
    return min(P.sortedPrims[k], P.n - 1u);
}

// Box of leaf k; with WRITE its leaf record too.
template <int KIND, bool WRITE>
__device__ __forceinline__ Box3 emitLeaf(const FitParams& P, uint32_t k) {
    const uint32_t item = sortedItem(P, k);
    if constexpr (KIND == 2) {
        const float4 lo = P.instBoxes[2 * (size_t)item], hi = P.instBoxes[2 * (size_t)item + 1];
        if (WRITE) {
            reinterpret_cast<InstanceRecord*>(P.leaves)[k] = P.instRecords[item];
            P.primToLeaf[item] = k;
        }
        return Box3{make_float3(lo.x, lo.y, lo.z), make_float3(hi.x, hi.y, hi.z)};
    } else {
        float3 v[3];
        const Box3 b = primBox(P.src, item, v);
        if (WRITE) {
            if constexpr (KIND == 0)
                writeTriangleLeaf(P, k, item, v);
            else
                reinterpret_cast<uint32_t*>(P.leaves)[k] = item;
        }
        return b;
    }
}

// Box of leaf k, written by an earlier launch: a whole triangle's comes from its leaf record
// in one step, others from the input.
template <int KIND>
__device__ __forceinline__ Box3 leafBox(const FitParams& P, uint32_t k) {
    if (KIND == 0 && P.src.kind == 0) {
        const float4* rec = reinterpret_cast<const float4*>(P.leaves) + 3 * (size_t)k;
        const float4 a = __ldcg(rec), b = __ldcg(rec + 1), c = __ldcg(rec + 2);
        return triangleBox(make_float3(a.x, a.y, a.z), make_float3(b.x, b.y, b.z), make_float3(c.x, c.y, c.z));
    }
    return emitLeaf<KIND, false>(P, k);
}

__device__ __forceinline__ Box3 unionBox(const Box3& a, const Box3& b) {
    return Box3{make_float3(fminf(a.lo.x, b.lo.x), fminf(a.lo.y, b.lo.y), fminf(a.lo.z, b.lo.z)),
                make_float3(fmaxf(a.hi.x, b.hi.x), fmaxf(a.hi.y, b.hi.y), fmaxf(a.hi.z, b.hi.z))};
}

// Box of the subtree of child word w, its node or leaf written by an earlier launch.
template <int KIND>
__device__ __forceinline__ Box3 subtreeBox(const FitParams& P, uint32_t w) {
    if (w & kLeafBit) return leafBox<KIND>(P, w & ~kLeafBit);
    const float4* N = P.nodes + 4 * (size_t)w;
    const float4 x = __ldcg(N), y = __ldcg(N + 1), z = __ldcg(N + 2);
    return Box3{make_float3(fminf(x.x, x.z), fminf(y.x, y.z), fminf(z.x, z.z)),
                make_float3(fmaxf(x.y, x.w), fmaxf(y.y, y.w), fmaxf(z.y, z.w))};
}

// A block's nodes in shared memory, numbered from its first leaf: node p as p - first leaf
// (< C), leaf k as C + k - first leaf.
template <typename K, int C>
struct EmitShared {
    float box[6][2 * C];    // lo.x, hi.x, lo.y, hi.y, lo.z, hi.z
    uint32_t parent[2 * C];  // parent entry (parent << 1 | side), kInvalid until its parent is built here
    uint32_t child[2][C];   // kInvalid until the node is built here
    uint32_t meet[C];
    int16_t delta[C + 1];   // delta[j]: of the leaf before position j and that at j
    uint16_t inside[C];     // the node splitting after position j lies inside the block
    K key[C + 2];
};

template <typename K, int C>
__device__ __forceinline__ Box3 sharedBox(const EmitShared<K, C>& S, uint32_t i) {
    return Box3{make_float3(S.box[0][i], S.box[2][i], S.box[4][i]), make_float3(S.box[1][i], S.box[3][i], S.box[5][i])};
}
template <typename K, int C>
__device__ __forceinline__ void setSharedBox(EmitShared<K, C>& S, uint32_t i, const Box3& b) {
    S.box[0][i] = b.lo.x, S.box[2][i] = b.lo.y, S.box[4][i] = b.lo.z;
    S.box[1][i] = b.hi.x, S.box[3][i] = b.hi.y, S.box[5][i] = b.hi.z;
}

__device__ __forceinline__ void writeRoot(const EmitParams& E, const Box3& b) {
    E.parents[0] = kInvalid;
    BvhHeader* h = E.fit.header;
    h->rootLo[0] = b.lo.x, h->rootLo[1] = b.lo.y, h->rootLo[2] = b.lo.z;
    h->rootHi[0] = b.hi.x, h->rootHi[1] = b.hi.y, h->rootHi[2] = b.hi.z;
}

// First launch: every node inside kEmitLeaves consecutive leaves.
template <typename K, int KIND>  // KIND: 0 triangles, 1 AABB list, 2 instances; n >= 2
__global__ void __launch_bounds__(kEmitLeaves) emitFitKernel(EmitParams E, const K* __restrict__ keys, TopLists out) {
    constexpr uint32_t C = kEmitLeaves;
    __shared__ EmitShared<K, kEmitLeaves> S;
    __shared__ uint32_t topBits[C / 32];  // where the block's remaining subtrees begin
    const FitParams& P = E.fit;
    const uint32_t n = P.n, t = threadIdx.x, b0 = blockIdx.x * C, m = min(C, n - b0);
    for (uint32_t j = t; j < m + 2; j += C) {  // key[j]: of position b0 + j - 1
        const uint32_t at = b0 + j;
        S.key[j] = (at >= 1 && at <= n) ? keys[at - 1] : (K)0;
    }
    S.meet[t] = 0u;
    if (t < C / 32) topBits[t] = 0u;
    S.child[0][t] = kInvalid;
    S.parent[t] = S.parent[C + t] = kInvalid;
    if (t < m) setSharedBox(S, C + t, emitLeaf<KIND, true>(P, b0 + t));
    __syncthreads();
    for (uint32_t j = t; j <= m; j += C) {
        const uint32_t at = b0 + j;  // positions at - 1 and at
        S.delta[j] = (at >= 1 && at < n) ? (int16_t)prefixOf(S.key[j], S.key[j + 1], at - 1, at) : (int16_t)-1;
    }
    {
        // the node splitting after position s reaches below the block when the code before
        // the block shares more with s than s and s + 1 share, and likewise above it
        bool in = t + 1 < m;
        if (in) {
            const uint32_t s = b0 + t;
            const int d = prefixOf(S.key[t + 1], S.key[t + 2], s, s + 1);
            if (b0 > 0 && prefixOf(S.key[0], S.key[t + 1], b0 - 1, s) > d) in = false;
            if (b0 + m < n && prefixOf(S.key[t + 2], S.key[m + 1], s + 1, b0 + m) > d) in = false;
        }
        S.inside[t] = in ? 1 : 0;
    }
    __syncthreads();
    // climb inside the block; a thread that ends with top set holds a subtree whose parent is
    // not built here
    uint32_t id = C + t, l = t, r = t;
    bool top = false;
    if (t < m) {
        int dl = S.delta[l], dr = S.delta[r + 1];
        for (;;) {
            const bool left = dr > dl;
            const uint32_t s = left ? r : l - 1u;
            if ((dl < 0 && dr < 0) || s >= m || !S.inside[s]) {
                top = true;
                break;
            }
            __threadfence_block();
            const uint32_t old = atomicExch(&S.meet[s], 0x80000000u | id << 16 | (left ? l : r));
            if (old == 0u) break;  // the sibling is still on its way up
            __threadfence_block();
            const uint32_t sib = (old >> 16) & 0x7FFFu, end = old & 0xFFFFu;
            const uint32_t a = left ? id : sib, b = left ? sib : id;
            if (left)
                r = end;
            else
                l = end;
            dl = S.delta[l], dr = S.delta[r + 1];
            id = (dl < 0 && dr < 0) ? 0u : dr > dl ? r : l;
            setSharedBox(S, id, unionBox(sharedBox(S, a), sharedBox(S, b)));
            S.child[0][id] = a, S.child[1][id] = b;
            S.parent[a] = (b0 + id) << 1, S.parent[b] = (b0 + id) << 1 | 1u;
        }
    }
    auto word = [&](uint32_t i) { return i < C ? b0 + i : kLeafBit | (b0 + i - C); };
    if (top) atomicOr(&topBits[l >> 5], 1u << (l & 31u));
    __syncthreads();
    if (top) {
        if (gridDim.x == 1) {
            writeRoot(E, sharedBox(S, id));
        } else {
            uint32_t rank = __popc(topBits[l >> 5] & ((1u << (l & 31u)) - 1u));
            for (uint32_t j = 0; j < l >> 5; ++j) rank += __popc(topBits[j]);
            if (rank < kTopMax) out.tops[(size_t)blockIdx.x * kTopMax + rank] = make_uint4(word(id), b0 + l, b0 + r, 0u);
            if (r + 1 == m) out.counts[blockIdx.x] = rank + 1;
        }
    }
    // the block's nodes, one float4 row per thread and step
    for (uint32_t q = t; q < 4 * m; q += C) {
        const uint32_t p = q >> 2, row = q & 3u, a = S.child[0][p], b = S.child[1][p];
        if (a == kInvalid) continue;
        P.nodes[4 * (size_t)b0 + q] =
            row == 3 ? make_float4(__uint_as_float(word(a)), __uint_as_float(word(b)), 0.f, 0.f)
                     : make_float4(S.box[2 * row][a], S.box[2 * row + 1][a], S.box[2 * row][b], S.box[2 * row + 1][b]);
    }
    for (uint32_t q = t; q < kWideWords * m; q += C) {
        const uint32_t p = q / kWideWords, row = q % kWideWords;
        if (S.child[0][p] == kInvalid) continue;
        float o[4] = {0.f, 0.f, 0.f, 0.f};
        if (row < 7) {
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                const uint32_t c = S.child[s][p];
                const bool leaf = c >= C;
                const uint32_t a = leaf ? c : S.child[0][c], b = leaf ? kInvalid : S.child[1][c];
                if (row == 6) {
                    o[2 * s] = __uint_as_float(word(a)), o[2 * s + 1] = __uint_as_float(leaf ? kInvalid : word(b));
                } else {
                    o[2 * s] = S.box[row][a];
                    o[2 * s + 1] = leaf ? ((row & 1u) ? -INFINITY : INFINITY) : S.box[row][b];
                }
            }
        }
        P.wide[kWideWords * (size_t)b0 + q] = make_float4(o[0], o[1], o[2], o[3]);
    }
    if (t < m) {
        if (S.parent[t] != kInvalid) E.parents[b0 + t] = S.parent[t];
        if (S.parent[C + t] != kInvalid) E.parents[n - 1 + b0 + t] = S.parent[C + t];
    }
}

// Shared memory of a further launch: items (a joined list's subtrees) are numbered kTopCap + i,
// the nodes made of them by the item before their split.
struct TopShared {
    float box[6][2 * kTopCap];  // lo.x, hi.x, lo.y, hi.y, lo.z, hi.z
    uint32_t word[kTopCap];     // items: child word
    uint32_t last[kTopCap];     // items: last leaf
    uint32_t number[kTopCap];   // nodes
    uint32_t meet[kTopCap];
    uint16_t child[2][kTopCap];
    int8_t delta[kTopCap + 1];
    uint8_t inside[kTopCap];
    uint32_t bits[kTopCap / 32];
    uint32_t first[kTopFan + 1];  // first item of each list
};

// Joins kTopFan lists: every node whose range lies inside their leaves, from their subtrees.
template <typename K, int KIND>
__global__ void __launch_bounds__(kTopThreads) emitTopKernel(EmitParams E, const K* __restrict__ keys, TopLists in,
                                                             uint32_t lists, TopLists out, uint32_t* error) {
    extern __shared__ uint4 topSmem[];
    TopShared& S = *reinterpret_cast<TopShared*>(topSmem);
    const FitParams& P = E.fit;
    const uint32_t n = P.n, t = threadIdx.x, list0 = blockIdx.x * kTopFan, mine = min(kTopFan, lists - list0);
    if (t < 32) {
        const uint32_t c = t < mine ? min(in.counts[list0 + t], kTopMax) : 0u;
        uint32_t incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t x = __shfl_up_sync(0xffffffffu, incl, o);
            if (t >= (uint32_t)o) incl += x;
        }
        if (t <= kTopFan) S.first[t] = incl - c;
    }
    __syncthreads();
    const uint32_t count = S.first[kTopFan];
    if (count == 0) {  // an empty list cannot be: every block leaves a subtree
        if (t == 0) latchError(error, GRT_ERROR_INTERNAL), out.counts[blockIdx.x] = 0u;
        return;
    }
    for (uint32_t i = t; i < count; i += kTopThreads) {
        uint32_t list = 0;
        for (uint32_t j = 1; j < kTopFan; ++j) list = i >= S.first[j] ? j : list;
        const uint4 top = in.tops[(size_t)(list0 + list) * kTopMax + (i - S.first[list])];
        const Box3 b = subtreeBox<KIND>(P, top.x);
        const uint32_t id = kTopCap + i;
        S.box[0][id] = b.lo.x, S.box[2][id] = b.lo.y, S.box[4][id] = b.lo.z;
        S.box[1][id] = b.hi.x, S.box[3][id] = b.hi.y, S.box[5][id] = b.hi.z;
        S.word[i] = top.x, S.last[i] = top.z;
        S.meet[i] = 0u;
        S.child[0][i] = 0xFFFFu;
    }
    if (t < kTopCap / 32) S.bits[t] = 0u;
    const uint32_t first = in.tops[(size_t)list0 * kTopMax].y;
    __syncthreads();
    const uint32_t last = S.last[count - 1];
    const K before = first > 0 ? keys[first - 1] : (K)0, after = last + 1 < n ? keys[last + 1] : (K)0;
    for (uint32_t i = t; i <= count; i += kTopThreads) {
        const uint32_t at = i ? S.last[i - 1] + 1 : first;  // delta of positions at - 1 and at
        int d = -1;
        if (at > 0 && at < n) {
            const K a = keys[at - 1], b = keys[at];
            d = prefixOf(a, b, at - 1, at);
            if (i > 0 && i < count)
                S.inside[i - 1] = !(first > 0 && prefixOf(before, a, first - 1, at - 1) > d) &&
                                  !(last + 1 < n && prefixOf(b, after, at, last + 1) > d);
        }
        S.delta[i] = (int8_t)d;
    }
    if (t == 0) S.inside[count - 1] = 0;
    __syncthreads();
    auto word = [&](uint32_t id) { return id < kTopCap ? S.number[id] : S.word[id - kTopCap]; };
    auto link = [&](uint32_t id, uint32_t entry) {
        const uint32_t w = word(id);
        E.parents[(w & kLeafBit) ? n - 1u + (w & ~kLeafBit) : w] = entry;
    };
    auto box = [&](uint32_t id) {
        return Box3{make_float3(S.box[0][id], S.box[2][id], S.box[4][id]),
                    make_float3(S.box[1][id], S.box[3][id], S.box[5][id])};
    };
    constexpr int kPer = kTopCap / kTopThreads;
    uint32_t topId[kPer], topL[kPer], topR[kPer];
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        const uint32_t i = t + k * kTopThreads;
        topId[k] = kInvalid;
        if (i >= count) continue;
        uint32_t id = kTopCap + i, l = i, r = i;
        int dl = S.delta[l], dr = S.delta[r + 1];
        for (;;) {
            const bool left = dr > dl;
            const uint32_t s = left ? r : l - 1u;  // the split after item s
            if ((dl < 0 && dr < 0) || s >= count || !S.inside[s]) {
                topId[k] = id, topL[k] = l, topR[k] = r;
                atomicOr(&S.bits[l >> 5], 1u << (l & 31u));
                break;
            }
            __threadfence_block();
            const uint32_t old = atomicExch(&S.meet[s], 0x80000000u | id << 12 | (left ? l : r));
            if (old == 0u) break;  // the sibling is still on its way up
            __threadfence_block();
            const uint32_t sib = (old >> 12) & 0x3FFFu, end = old & 0xFFFu;
            const uint32_t a = left ? id : sib, b = left ? sib : id;
            if (left)
                r = end;
            else
                l = end;
            dl = S.delta[l], dr = S.delta[r + 1];
            const uint32_t num =
                (dl < 0 && dr < 0) ? 0u : dr > dl ? S.last[r] : (l ? S.last[l - 1] + 1 : first);
            const Box3 u = unionBox(box(a), box(b));
            S.box[0][s] = u.lo.x, S.box[2][s] = u.lo.y, S.box[4][s] = u.lo.z;
            S.box[1][s] = u.hi.x, S.box[3][s] = u.hi.y, S.box[5][s] = u.hi.z;
            S.number[s] = num;
            S.child[0][s] = (uint16_t)a, S.child[1][s] = (uint16_t)b;
            link(a, num << 1), link(b, num << 1 | 1u);
            id = s;
        }
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        if (topId[k] == kInvalid) continue;
        if (gridDim.x == 1) {
            writeRoot(E, box(topId[k]));
            continue;
        }
        const uint32_t l = topL[k], r = topR[k];
        uint32_t rank = __popc(S.bits[l >> 5] & ((1u << (l & 31u)) - 1u));
        for (uint32_t j = 0; j < l >> 5; ++j) rank += __popc(S.bits[j]);
        if (rank < kTopMax)
            out.tops[(size_t)blockIdx.x * kTopMax + rank] =
                make_uint4(word(topId[k]), l ? S.last[l - 1] + 1 : first, S.last[r], 0u);
        if (r + 1 == count) out.counts[blockIdx.x] = rank + 1;
    }
    // the new nodes, one float4 row of a binary (0-3) or 4-wide (4-11) node per thread and step
    for (uint32_t q = t; q < 12 * count; q += kTopThreads) {
        const uint32_t s = q / 12, row = q % 12;
        if (S.child[0][s] == 0xFFFFu) continue;
        const size_t num = S.number[s];
        const uint32_t c[2] = {S.child[0][s], S.child[1][s]};
        if (row < 4) {
            P.nodes[4 * num + row] =
                row == 3 ? make_float4(__uint_as_float(word(c[0])), __uint_as_float(word(c[1])), 0.f, 0.f)
                         : make_float4(S.box[2 * row][c[0]], S.box[2 * row + 1][c[0]], S.box[2 * row][c[1]],
                                       S.box[2 * row + 1][c[1]]);
            continue;
        }
        const uint32_t w = row - 4;
        float o[4] = {0.f, 0.f, 0.f, 0.f};
        if (w < 7) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint32_t id = c[h];
                if (id < kTopCap) {  // a node made here
                    const uint32_t a = S.child[0][id], b = S.child[1][id];
                    o[2 * h] = w == 6 ? __uint_as_float(word(a)) : S.box[w][a];
                    o[2 * h + 1] = w == 6 ? __uint_as_float(word(b)) : S.box[w][b];
                } else if (S.word[id - kTopCap] & kLeafBit) {
                    o[2 * h] = w == 6 ? __uint_as_float(S.word[id - kTopCap]) : S.box[w][id];
                    o[2 * h + 1] = w == 6 ? __uint_as_float(kInvalid) : (w & 1u) ? -INFINITY : INFINITY;
                } else {  // a node of an earlier launch: its children are in its binary node
                    const float4 x = __ldcg(P.nodes + 4 * (size_t)S.word[id - kTopCap] + (w >> 1));
                    o[2 * h] = w == 6 || !(w & 1u) ? x.x : x.y;
                    o[2 * h + 1] = w == 6 ? x.y : (w & 1u) ? x.w : x.z;
                }
            }
        }
        P.wide[kWideWords * num + w] = make_float4(o[0], o[1], o[2], o[3]);
    }
}

}  // namespace grt
