// Fully linked octree from the cornerstone array (Sec. 5, steps 1-5), breadth-first.
//
// Node keys: every leaf i gives a node at level L - log8(K_{i+1} - K_i); every adjacent pair
// (K_i, K_{i+1}) whose first differing bit is the leading bit of an octal digit (d % 3 == 0 with
// d the number of equal leading bits of the 3L-bit keys, step 2) gives the internal node at level
// d / 3 that is the lowest common ancestor of the two leaves: the pair straddles the boundary
// between its child 3 and child 4, so each internal node appears exactly once.
//
// Breadth-first order (step 3): taken in array order, leaf i followed by pair i is an in-order
// walk of the tree, so the nodes of any one level already appear in key order. A stable
// partition of that sequence by level therefore gives the breadth-first layout without sorting
// 64-bit keys, and the offsets of the partition are the level offsets LO (step 4). This replaces
// the paper's digit-weight slot mapping of step 2 followed by a radix sort of NK: the final NK
// is the same. The partition is a counting sort with L + 1 buckets: per-tile level counts, one scan
// over (level, tile), and a scatter that ranks items stably inside each tile.
//
// Step 5: the first child of an internal node. In this layout every internal node has its 8
// children together and the sibling groups follow their parents' breadth-first order, so the
// children of the g-th internal node (counting internal nodes only, in breadth-first order) are
// the nodes 8 g + 1 .. 8 g + 8: the child index that the paper's search for the key << 3 in the
// next level finds. The scatter ranks every internal node among the internal nodes with a second
// counting sort of the pairs alone and writes CO (and the parent of every sibling group) directly.
// The sets of a batch go the same way, each from its own first node and internal node.
//
// Node counts in the same pass, where the leaves' particle offsets are at hand (the builds): a node's
// particles are those between the first of its first leaf and the first of the leaf after its last, and
// both leaves are found near the pair (`covered`). This takes the place of a sum over the children level
// by level, whose grid barriers bounded it (upsweep.cu, which still serves callers that have counts only).
// Link and counts together: 512 sets of 1,024 to 1,048,576 particles 640 -> 310 us, 48 of 128 to 4,096
// 88 -> 35, one of 1,048,576 43 -> 25, of 33,554,432 122 -> 63.
#include "common.cuh"

namespace CST_NS {
namespace {

constexpr int kThreads = 256;
// Leaves per thread: 8, and 2 up to kSmallLeaves leaves, where a pass of 8 items in a row is longer than
// the rest of the kernel and most SMs would have no tile (12,000 leaves: scatter 13.5 us with 8, 9.5 with 2).
constexpr int kItemsLarge = 8, kItemsSmall = 2;
constexpr long long kSmallLeaves = 1 << 18;
constexpr int items_of(long long leaves) { return leaves <= kSmallLeaves ? kItemsSmall : kItemsLarge; }
constexpr int kNumLevels = kLevels + 1;  // levels 0..L

__device__ __forceinline__ int leaf_level(Key delta) {  // delta is a power of 8
    return kLevels - key_ffs(delta) / 3;
}

// Level of the internal node implied by the pair (i, i+1), or -1 when d % 3 != 0.
__device__ __forceinline__ int pair_level(Key a, Key b) {
    int d = key_clz(a ^ b) - (kWordBits - kKeyBits);  // equal leading bits of the 3L-bit keys
    return (d >= 0 && d % 3 == 0) ? d / 3 : -1;
}

__device__ __forceinline__ Key placeholder(Key key, int level) {
    return (static_cast<Key>(1) << (3 * level)) | (key >> (3 * (kLevels - level)));
}

// The tile that a block works on: `cnt` leaves from `e0`, of a set whose first leaf is `lo` and whose end
// key is element `hi`; its counters are at first * 22 + level * of + index.
struct Tile {
    u32 e0, cnt, lo, hi;
    u32 first, of, index;
    __device__ __forceinline__ u32 counter(int level) const {
        return first * kNumLevels + static_cast<u32>(level) * of + index;
    }
};

// One counter word per thread and level: all nodes in the low half, internal nodes in the high half (a tile
// has at most 2 * 2048 nodes, so neither its sums nor its ranks overflow a half).
constexpr u32 kLeafOne = 1u, kInternalOne = 0x10001u;
// A row of them has a gap after every 8 threads, so that neither a thread per column nor a lane per 8
// columns meets bank conflicts.
constexpr int kRow = kThreads + kThreads / 8;
__device__ __forceinline__ int column(int thread) { return thread + (thread >> 3); }

// Counts a thread's items by level; `levels` keeps each leaf's level and its pair's (kNoPair: none) << 8.
constexpr u32 kNoPair = 255u;
template <int ITEMS>
__device__ __forceinline__ void count_items(const Key (&key)[ITEMS + 1], u32 i0, const Tile& t,
                                            u32 (*s_rank)[kRow], u32 (&levels)[ITEMS]) {
    const int me = column(threadIdx.x);
#pragma unroll
    for (int l = 0; l < kNumLevels; ++l) s_rank[l][me] = 0;
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
        if (i0 + k >= t.e0 + t.cnt) break;
        const int ll = leaf_level(key[k + 1] - key[k]);
        const int pl = i0 + k + 1 < t.hi ? pair_level(key[k], key[k + 1]) : -1;
        s_rank[ll][me] += kLeafOne;
        if (pl >= 0) s_rank[pl][me] += kInternalOne;
        levels[k] = static_cast<u32>(ll) | (pl >= 0 ? static_cast<u32>(pl) : kNoPair) << 8;
    }
}

template <int ITEMS>
__device__ __forceinline__ void load_items(const Key* __restrict__ K, u32 i0, const Tile& t, Key (&key)[ITEMS + 1]) {
#pragma unroll
    for (int k = 0; k <= ITEMS; ++k) key[k] = i0 + k <= t.e0 + t.cnt ? K[i0 + k] : kKeyEnd;
}

template <int ITEMS>
__device__ __forceinline__ void count_tile(const Key* __restrict__ K, const Tile& t, u32* __restrict__ counts,
                                           u32* __restrict__ pair_counts) {
    __shared__ u32 s_rank[kNumLevels][kRow];
    const u32 i0 = t.e0 + threadIdx.x * ITEMS;
    Key key[ITEMS + 1];
    u32 levels[ITEMS];
    load_items<ITEMS>(K, i0, t, key);
    count_items<ITEMS>(key, i0, t, s_rank, levels);
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int l = warp; l < kNumLevels; l += kThreads / 32) {
        u32 v = 0;
#pragma unroll
        for (int q = 0; q < kThreads / 32; ++q) v += s_rank[l][column(q * 32 + lane)];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) {
            counts[t.counter(l)] = v & 0xffffu;
            pair_counts[t.counter(l)] = v >> 16;
        }
    }
}

// The leaves of the internal node of level `level` whose pair is (i, i + 1): from the first with a key at or
// after its start to the one with a key at or after its end, within the set. When the eight children are
// leaves (nine in ten nodes of a usual tree) they are i - 3 .. i + 4; else the search goes outwards by powers of
// 8 and then bisects. Every index stays within [lo, hi], whatever the keys.
__device__ __forceinline__ uint2 covered(const Key* __restrict__ K, const Tile& t, u32 i, Key a, int level) {
    const Key size = static_cast<Key>(1) << (3 * (kLevels - level));
    const Key start = a & ~(size - 1), end = start + size;
    uint2 r = make_uint2(i - 3, i + 5);
    if (i - t.lo < 3 || K[i - 3] != start) {
        u32 at = i, from = i, step = 8;  // K[at] >= start
        for (;; step <<= 3) {
            from = i - t.lo > step ? i - step : t.lo;
            if (from == t.lo || K[from] < start) break;
            at = from;
        }
        while (from < at) {
            const u32 mid = from + ((at - from) >> 1);
            if (K[mid] < start)
                from = mid + 1;
            else
                at = mid;
        }
        r.x = at;
    }
    if (t.hi - i < 5 || K[i + 5] != end) {
        u32 from = i + 1, at = t.hi, step = 8;
        for (;; step <<= 3) {
            at = t.hi - i > step ? i + step : t.hi;
            if (at == t.hi || K[at] >= end) break;
            from = at;
        }
        while (from < at) {
            const u32 mid = from + ((at - from) >> 1);
            if (K[mid] < end)
                from = mid + 1;
            else
                at = mid;
        }
        r.y = at;
    }
    return r;
}

struct Out {
    u32 n_nodes;              // capacity of the node arrays
    Key* NK;
    int* leaf_to_node;
    int* CO;
    int* parent;              // may be NULL
    const u32* leaf_offsets;  // with COUNTS: first particle of every leaf and end key
    u32* node_counts;
};

// Places a tile's leaves and internal nodes in breadth-first order. Each thread ranks its leaves and pairs
// in in-order sequence (leaf i, then the internal node of pair i). With 8 leaves per thread it lists them by
// level in shared memory, and the nodes are then written from that list, a thread each, so that the lanes of a
// warp write neighbouring nodes: written from the ranking loop, the eight stores of a warp to one sector were
// eight transactions (7.6 million leaves: 204 us, listed 150; 1.7 million 64 and 43). With 2 it writes them as it
// ranks them (the list costs 2 us where the whole takes 10). Six blocks per SM hide the searches' chains of
// loads better than five (43 us against 51). The g-th internal node of the set has its children at 8 g + 1 of the
// set's nodes.
template <int ITEMS, bool COUNTS>
__device__ __forceinline__ void place_tile(const Key* __restrict__ K, const Tile& t, const u32* __restrict__ offsets,
                                           const u32* __restrict__ pair_offsets, const Out& o) {
    constexpr bool kListed = ITEMS > kItemsSmall;
    constexpr u32 kList = kThreads * ITEMS / 8 + 64;
    __shared__ u32 s_rank[kNumLevels][kRow];      // per-thread counts, then per-thread ranks within the tile
    __shared__ u32 s_base[2][kNumLevels];         // the tile's first node and internal node of each level
    __shared__ u32 s_start[kNumLevels];           // nodes of the tile at the levels before
    __shared__ unsigned short s_slot[kListed ? 2 * kThreads * ITEMS : 1];  // by level: 2 x leaf in the tile, + 1: pair
    __shared__ uint2 s_list[kList];               // internal nodes: node, leaf | rank among the level's << 16
    __shared__ u32 s_listed;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, me = column(tid);
    const u32 i0 = t.e0 + tid * ITEMS;
    Key key[ITEMS + 1];
    u32 levels[ITEMS];
    load_items<ITEMS>(K, i0, t, key);
    if (tid == 0) s_listed = 0;
    if (tid < kNumLevels) s_base[0][tid] = offsets[t.counter(tid)];
    if (tid >= 32 && tid < 32 + kNumLevels) s_base[1][tid - 32] = pair_offsets[t.counter(tid - 32)];
    const u32 first_node = offsets[t.first * kNumLevels], first_internal = pair_offsets[t.first * kNumLevels];
    count_items<ITEMS>(key, i0, t, s_rank, levels);
    __syncthreads();
    // exclusive scan of every level row across the threads
    for (int l = warp; l < kNumLevels; l += kThreads / 32) {
        u32 v[kThreads / 32];
        u32 sum = 0;
#pragma unroll
        for (int q = 0; q < kThreads / 32; ++q) {
            v[q] = s_rank[l][column(lane * (kThreads / 32) + q)];
            sum += v[q];
        }
        u32 incl = sum;
        for (int s = 1; s < 32; s <<= 1) {
            const u32 w = __shfl_up_sync(0xffffffffu, incl, s);
            if (lane >= s) incl += w;
        }
        if (kListed && lane == 31) s_start[l] = incl & 0xffffu;
        u32 run = incl - sum;
#pragma unroll
        for (int q = 0; q < kThreads / 32; ++q) {
            s_rank[l][column(lane * (kThreads / 32) + q)] = run;
            run += v[q];
        }
    }
    __syncthreads();
    if (kListed && warp == 0) {  // the levels' totals to their starts
        const u32 own = lane < kNumLevels ? s_start[lane] : 0u;
        u32 incl = own;
        for (int s = 1; s < 32; s <<= 1) {
            const u32 w = __shfl_up_sync(0xffffffffu, incl, s);
            if (lane >= s) incl += w;
        }
        if (lane < kNumLevels) s_start[lane] = incl - own;
    }
    if (kListed) __syncthreads();
    auto leaf = [&](u32 x, u32 i, Key a, int level) {
        if (x >= o.n_nodes) return;
        o.NK[x] = placeholder(a, level);
        o.CO[x] = 0;
        o.leaf_to_node[i] = static_cast<int>(x);
        if (COUNTS) o.node_counts[x] = o.leaf_offsets[i + 1] - o.leaf_offsets[i];
    };
    // CO, parent and count of internal node y of pair i, the r-th internal node of the tile at its level
    auto internal = [&](u32 y, u32 i, Key a, int level, u32 r) {
        if (y >= o.n_nodes) return;
        const u32 g = s_base[1][level] + r - first_internal;
        const u32 c = first_node + 8u * g + 1u;
        const bool inside = c + 7u < o.n_nodes;
        if (!kListed) o.NK[y] = placeholder(a, level);
        o.CO[y] = inside ? static_cast<int>(c) : 0;
        if (o.parent && inside) o.parent[g] = static_cast<int>(y);
        if (COUNTS) {
            const uint2 range = covered(K, t, i, a, level);
            o.node_counts[y] = o.leaf_offsets[range.y] - o.leaf_offsets[range.x];
        }
    };
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
        const u32 i = i0 + k;
        if (i >= t.e0 + t.cnt) break;
        const u32 item = 2u * (tid * ITEMS + k);
        const u32 ll = levels[k] & 255u, pl = levels[k] >> 8;
        const u32 rx = s_rank[ll][me];
        s_rank[ll][me] = rx + kLeafOne;
        if (kListed)
            s_slot[s_start[ll] + (rx & 0xffffu)] = static_cast<unsigned short>(item);
        else
            leaf(s_base[0][ll] + (rx & 0xffffu), i, key[k], static_cast<int>(ll));
        if (pl != kNoPair) {
            const u32 ry = s_rank[pl][me];
            s_rank[pl][me] = ry + kInternalOne;
            if (kListed) s_slot[s_start[pl] + (ry & 0xffffu)] = static_cast<unsigned short>(item + 1u);
            const u32 y = s_base[0][pl] + (ry & 0xffffu);
            const u32 at = atomicAdd(&s_listed, 1u);
            if (at < kList)
                s_list[at] = make_uint2(y, (item >> 1) | (ry & 0xffff0000u));
            else
                internal(y, i, key[k], static_cast<int>(pl), ry >> 16);
        }
    }
    __syncthreads();
    if (kListed) {
        const u32 nodes = s_start[kNumLevels - 1] + (s_rank[kNumLevels - 1][column(kThreads - 1)] & 0xffffu);
        for (u32 p = tid; p < nodes; p += kThreads) {
            const u32 item = s_slot[p], i = t.e0 + (item >> 1);
            const Key a = K[i], b = K[i + 1];
            const int level = (item & 1u) ? pair_level(a, b) : leaf_level(b - a);
            const u32 x = s_base[0][level] + (p - s_start[level]);
            if ((item & 1u) == 0u)
                leaf(x, i, a, level);
            else if (x < o.n_nodes)
                o.NK[x] = placeholder(a, level);
        }
    }
    // the internal nodes (one leaf in seven has one) side by side, not one lane of a warp at a time
    const u32 listed = min(s_listed, kList);
    for (u32 q = tid; q < listed; q += kThreads) {
        const uint2 e = s_list[q];
        const u32 i = t.e0 + (e.y & 0xffffu);
        const Key a = K[i];
        internal(e.x, i, a, pair_level(a, K[i + 1]), e.y >> 16);
    }
}

template <int ITEMS>
__device__ __forceinline__ Tile single_tile(u32 nl) {
    const u32 e0 = blockIdx.x * (kThreads * ITEMS);
    return Tile{e0, min(static_cast<u32>(kThreads * ITEMS), nl - e0), 0u, nl, 0u, gridDim.x, blockIdx.x};
}

template <int ITEMS>
__global__ void __launch_bounds__(kThreads) link_count_kernel(const Key* __restrict__ K, u32 nl,
                                                              u32* __restrict__ counts, u32* __restrict__ pair_counts) {
    count_tile<ITEMS>(K, single_tile<ITEMS>(nl), counts, pair_counts);
}

template <int ITEMS, bool COUNTS>
__global__ void __launch_bounds__(kThreads, 6) link_scatter_kernel(const Key* __restrict__ K, u32 nl,
                                                                const u32* __restrict__ offsets,
                                                                const u32* __restrict__ pair_offsets, Out o) {
    place_tile<ITEMS, COUNTS>(K, single_tile<ITEMS>(nl), offsets, pair_offsets, o);
}

// Exclusive scans of the level-major (level, tile) counts of all nodes (half 0) and of the internal
// nodes alone (half 1), each of `len` entries at a distance of `stride`, in chunks of kScanChunk:
// block (c, h) sums chunk c of half h, then adds the sums of the chunks before it and scans its chunk. LO comes
// from half 0 (LO[l] = offset of (l, 0), LO[22] = total); a total of all nodes different from
// n_expected, or of internal nodes different from (n_expected - 1) / 8, means the input was not a
// cornerstone array. Without LO (the batched (set, level, tile) counts) the total goes to the entry
// after the scanned ones.
constexpr u32 kScanThreads = 1024;
constexpr u32 kScanPer = 4;
constexpr u32 kScanChunk = kScanThreads * kScanPer;

__global__ void __launch_bounds__(kScanThreads) link_scan_reduce_kernel(const u32* __restrict__ counts, u32 len,
                                                                        size_t stride, u32* __restrict__ partial) {
    __shared__ u32 s_warp[kScanThreads / 32];
    const u32 h = blockIdx.y, c = blockIdx.x;
    const u32* a = counts + h * stride;
    u32 sum = 0;
#pragma unroll
    for (u32 j = 0; j < kScanPer; ++j) {
        const u32 i = c * kScanChunk + j * kScanThreads + threadIdx.x;  // coalesced
        if (i < len) sum += a[i];
    }
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if ((threadIdx.x & 31) == 0) s_warp[threadIdx.x >> 5] = sum;
    __syncthreads();
    if (threadIdx.x < 32) {
        u32 v = s_warp[threadIdx.x];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (threadIdx.x == 0) partial[h * gridDim.x + c] = v;
    }
}

__global__ void __launch_bounds__(kScanThreads) link_scan_apply_kernel(u32* __restrict__ counts, u32 len,
                                                                       size_t stride, u32 ntiles,
                                                                       const u32* __restrict__ partial,
                                                                       int* __restrict__ LO, u32 n_expected,
                                                                       WsHeader* hdr) {
    __shared__ u32 s_warp[kScanThreads / 32];
    __shared__ u32 s_carry;
    const u32 h = blockIdx.y, c = blockIdx.x, nchunks = gridDim.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (warp == 0) {  // sums of the chunks before this one (and of all chunks, for the total)
        u32 before = 0, all = 0;
        for (u32 k = lane; k < nchunks; k += 32) {
            const u32 v = partial[h * nchunks + k];
            all += v;
            if (k < c) before += v;
        }
        for (int o = 16; o > 0; o >>= 1) {
            before += __shfl_xor_sync(0xffffffffu, before, o);
            all += __shfl_xor_sync(0xffffffffu, all, o);
        }
        if (lane == 0) {
            s_carry = before;
            if (c == nchunks - 1) {
                if (LO) {
                    const u32 want = h == 0 ? n_expected : (n_expected - 1) / 8;
                    if (h == 0) LO[kNumLevels] = static_cast<int>(all);
                    if (all != want) raise_error(hdr, CSTONE_ERR_INVALID_ARG, all);
                } else {
                    counts[h * stride + len] = all;  // without LO (batched sets): the total after the scan
                }
            }
        }
    }
    __syncthreads();
    u32* a = counts + h * stride;
    // thread t takes the kScanPer consecutive entries c * kScanChunk + t * kScanPer + j
    const u32 i0 = c * kScanChunk + threadIdx.x * kScanPer;
    u32 v[kScanPer], sum = 0;
#pragma unroll
    for (u32 j = 0; j < kScanPer; ++j) {
        v[j] = i0 + j < len ? a[i0 + j] : 0u;
        sum += v[j];
    }
    u32 incl = sum;
    for (int o = 1; o < 32; o <<= 1) {
        const u32 t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        u32 w = s_warp[lane];
        for (int o = 1; o < 32; o <<= 1) {
            const u32 t = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += t;
        }
        s_warp[lane] = w;
    }
    __syncthreads();
    u32 run = s_carry + (warp > 0 ? s_warp[warp - 1] : 0u) + incl - sum;
#pragma unroll
    for (u32 j = 0; j < kScanPer; ++j) {
        const u32 i = i0 + j;
        if (i < len) {
            a[i] = run;
            if (LO && h == 0 && i % ntiles == 0) LO[i / ntiles] = static_cast<int>(run);
        }
        run += v[j];
    }
}

// The largest number of tiles of any array of at most `leaves` leaves.
inline long long most_tiles(long long leaves) {
    const long long small = leaves < kSmallLeaves ? leaves : kSmallLeaves;
    const long long a = (small + kThreads * kItemsSmall - 1) / (kThreads * kItemsSmall);
    const long long b = (leaves + kThreads * kItemsLarge - 1) / (kThreads * kItemsLarge);
    return a > b ? a : b;
}

struct LinkLayout {
    u32* counts;   // [2][ntiles * 22]: all nodes, then internal nodes, per (level, tile)
    u32* partial;  // [2][chunks] chunk sums of the scans
    u32 ntiles;
    u32 chunks;    // scan chunks per half
    size_t bytes;
};

LinkLayout link_layout(void* ws, long long nl) {
    LinkLayout l;
    Carver c(ws);
    const long long tile = kThreads * items_of(nl);
    l.ntiles = static_cast<u32>((nl + tile - 1) / tile);
    if (l.ntiles == 0) l.ntiles = 1;
    const u32 len = l.ntiles * kNumLevels;
    l.chunks = (len + kScanChunk - 1) / kScanChunk;
    // a workspace for more leaves serves fewer: no smaller than the largest that small tiles need
    const size_t held = (size_t)most_tiles(nl) * kNumLevels;
    l.counts = c.take<u32>(2 * held);
    l.partial = c.take<u32>(2 * ((held + kScanChunk - 1) / kScanChunk));
    l.bytes = c.size();
    return l;
}

// ------------------------------------------------------------------ batched sets
// Several cornerstone arrays stored back to back as elements (each set's leaves followed by its end
// key 8^L). Tiles are aligned to sets, so the per-tile level counts of set s are laid out at
// [tile_first[s] * 22 + level * tiles_of_s + k]: one scan over everything then yields, set by set
// and level by level, the node positions of a concatenated node array in which every set's tree is
// one contiguous breadth-first block.
struct LinkSets {
    const long long* elem_offsets;  // [S+1] first element of each set
    u32 tile;                       // leaves per tile
    u32* n_tiles;                   // device scalar
    u32* tile_first;                // [S+1] first tile of each set
    u32* tile_set;                  // [max_tiles]
    u32* tile_elem;                 // [max_tiles] first leaf element of the tile
    u32* tile_count;                // [max_tiles]
    u32* node_first;                // [S+1] expected first node of each set
    int n_sets;
};

__global__ void __launch_bounds__(1024) link_b_setup_kernel(LinkSets ls) {
    __shared__ u32 s_t[1024], s_n[1024];
    const int per = (ls.n_sets + 1023) / 1024;
    const int begin = threadIdx.x * per, end = min(begin + per, ls.n_sets);
    u32 st = 0, sn = 0;
    for (int q = begin; q < end; ++q) {
        const long long nl = ls.elem_offsets[q + 1] - ls.elem_offsets[q] - 1;
        st += static_cast<u32>((nl + ls.tile - 1) / ls.tile);
        sn += static_cast<u32>(nl + (nl - 1) / 7);
    }
    s_t[threadIdx.x] = st;
    s_n[threadIdx.x] = sn;
    __syncthreads();
    for (int o = 1; o < 1024; o <<= 1) {
        const u32 a = threadIdx.x >= (unsigned)o ? s_t[threadIdx.x - o] : 0u;
        const u32 b = threadIdx.x >= (unsigned)o ? s_n[threadIdx.x - o] : 0u;
        __syncthreads();
        s_t[threadIdx.x] += a;
        s_n[threadIdx.x] += b;
        __syncthreads();
    }
    u32 rt = s_t[threadIdx.x] - st, rn = s_n[threadIdx.x] - sn;
    for (int q = begin; q < end; ++q) {
        ls.tile_first[q] = rt;
        ls.node_first[q] = rn;
        const long long nl = ls.elem_offsets[q + 1] - ls.elem_offsets[q] - 1;
        rt += static_cast<u32>((nl + ls.tile - 1) / ls.tile);
        rn += static_cast<u32>(nl + (nl - 1) / 7);
    }
    if (threadIdx.x == 1023) {
        ls.tile_first[ls.n_sets] = s_t[1023];
        ls.node_first[ls.n_sets] = s_n[1023];
        *ls.n_tiles = s_t[1023];
    }
}

__global__ void __launch_bounds__(kThreads) link_b_tiles_kernel(LinkSets ls, u32 max_tiles, u32 elem_cap,
                                                                int* __restrict__ leaf_to_node) {
    // elements between the actual count and the capacity map to no node
    const u32 ne = static_cast<u32>(ls.elem_offsets[ls.n_sets]);
    for (u32 e = ne + blockIdx.x * kThreads + threadIdx.x; e < elem_cap; e += gridDim.x * kThreads)
        leaf_to_node[e] = -1;
    const u32 total = *ls.n_tiles;
    for (u32 t = blockIdx.x * kThreads + threadIdx.x; t < max_tiles; t += gridDim.x * kThreads) {
        if (t >= total) {
            ls.tile_count[t] = 0;
            continue;
        }
        int lo = 0, hi = ls.n_sets;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (ls.tile_first[mid] <= t)
                lo = mid;
            else
                hi = mid;
        }
        const long long e0 = ls.elem_offsets[lo] + (long long)(t - ls.tile_first[lo]) * ls.tile;
        const long long last_leaf_end = ls.elem_offsets[lo + 1] - 1;  // the end key is not a leaf
        ls.tile_set[t] = static_cast<u32>(lo);
        ls.tile_elem[t] = static_cast<u32>(e0);
        ls.tile_count[t] = static_cast<u32>(min((long long)ls.tile, last_leaf_end - e0));
    }
}

__device__ __forceinline__ u32 count_index(const LinkSets& ls, u32 set, int level, u32 k) {
    const u32 tf = ls.tile_first[set], nt = ls.tile_first[set + 1] - tf;
    return tf * kNumLevels + static_cast<u32>(level) * nt + k;
}

__device__ __forceinline__ Tile batched_tile(const LinkSets& ls, u32 tile) {
    const u32 set = ls.tile_set[tile];
    Tile t;
    t.cnt = ls.tile_count[tile];
    t.e0 = ls.tile_elem[tile];
    t.lo = static_cast<u32>(ls.elem_offsets[set]);
    t.hi = static_cast<u32>(ls.elem_offsets[set + 1] - 1);
    t.first = ls.tile_first[set];
    t.of = ls.tile_first[set + 1] - t.first;
    t.index = tile - t.first;
    return t;
}

template <int ITEMS>
__global__ void __launch_bounds__(kThreads) link_b_count_kernel(const Key* __restrict__ K, LinkSets ls,
                                                                u32* __restrict__ counts,
                                                                u32* __restrict__ pair_counts) {
    if (blockIdx.x < *ls.n_tiles) count_tile<ITEMS>(K, batched_tile(ls, blockIdx.x), counts, pair_counts);
}

// Level offsets of every set (global node indices), a size check per set, and -1 for the
// leaf_to_node entries of the end keys.
__global__ void link_b_lo_kernel(const u32* __restrict__ counts, LinkSets ls, int* __restrict__ LO,
                                 int* __restrict__ leaf_to_node, WsHeader* hdr) {
    const u32 total_len = *ls.n_tiles * kNumLevels;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < ls.n_sets * (kNumLevels + 1);
         i += gridDim.x * blockDim.x) {
        const int set = i / (kNumLevels + 1), l = i % (kNumLevels + 1);
        u32 v;
        if (l < kNumLevels)
            v = counts[count_index(ls, set, l, 0)];
        else
            v = set + 1 < ls.n_sets ? counts[count_index(ls, set + 1, 0, 0)] : counts[total_len];
        LO[i] = static_cast<int>(v);
        if (l == kNumLevels) {
            const u32 first = counts[count_index(ls, set, 0, 0)];
            if (v - first != ls.node_first[set + 1] - ls.node_first[set])
                raise_error(hdr, CSTONE_ERR_INVALID_ARG, static_cast<u32>(set));
            leaf_to_node[ls.elem_offsets[set + 1] - 1] = -1;
        }
    }
}

template <int ITEMS, bool COUNTS>
__global__ void __launch_bounds__(kThreads, 6) link_b_scatter_kernel(const Key* __restrict__ K, LinkSets ls,
                                                                  const u32* __restrict__ offsets,
                                                                  const u32* __restrict__ pair_offsets, Out o) {
    if (blockIdx.x < *ls.n_tiles)
        place_tile<ITEMS, COUNTS>(K, batched_tile(ls, blockIdx.x), offsets, pair_offsets, o);
}

struct LinkBLayout {
    LinkSets ls;
    u32* counts;   // 2 x [max_tiles * 22 + 1]: (set, level, tile) counts of all nodes and of internal nodes,
                   // their exclusive scans, the totals
    u32* partial;  // [2][chunks] chunk sums of the scans
    u32 max_tiles;
    u32 chunks;
    size_t bytes;
};

LinkBLayout link_b_layout(void* ws, long long n_elements, int n_sets) {
    LinkBLayout l;
    Carver c(ws);
    l.ls.tile = static_cast<u32>(kThreads * items_of(n_elements));
    l.max_tiles = static_cast<u32>((n_elements + l.ls.tile - 1) / l.ls.tile + n_sets);
    // a workspace for more elements serves fewer: no smaller than the largest that small tiles need
    const size_t held = static_cast<size_t>(most_tiles(n_elements)) + n_sets;
    l.ls.n_tiles = c.take<u32>(1);
    l.ls.tile_first = c.take<u32>((size_t)n_sets + 1);
    l.ls.tile_set = c.take<u32>(held);
    l.ls.tile_elem = c.take<u32>(held);
    l.ls.tile_count = c.take<u32>(held);
    l.ls.node_first = c.take<u32>((size_t)n_sets + 1);
    l.ls.n_sets = n_sets;
    l.ls.elem_offsets = nullptr;
    l.counts = c.take<u32>(2 * (held * kNumLevels + 1));
    l.chunks = static_cast<u32>(((size_t)l.max_tiles * kNumLevels + kScanChunk - 1) / kScanChunk);
    l.partial = c.take<u32>(2 * ((held * kNumLevels + kScanChunk - 1) / kScanChunk));
    l.bytes = c.size();
    return l;
}

}  // namespace

size_t link_batched_ws_bytes(long long n_elements, int n_sets) {
    return link_b_layout(nullptr, n_elements, n_sets).bytes;
}

int launch_link_batched(const Key* K, long long n_elements, const long long* elem_offsets, int n_sets, Key* NK,
                        int* CO, int* LO, int* leaf_to_node, long long n_nodes, const u32* leaf_offsets,
                        u32* node_counts, void* ws, cudaStream_t st) {
    LinkBLayout l = link_b_layout(ws, n_elements, n_sets);
    l.ls.elem_offsets = elem_offsets;
    WsHeader* hdr = reinterpret_cast<WsHeader*>(ws);
    const u32 len = l.max_tiles * kNumLevels;  // unused tail entries are zero
    const size_t stride = (size_t)len + 1;
    CST_CUDA(cudaMemsetAsync(hdr, 0, sizeof(WsHeader), st));
    CST_CUDA(cudaMemsetAsync(l.counts, 0, 2 * stride * sizeof(u32), st));
    link_b_setup_kernel<<<1, 1024, 0, st>>>(l.ls);
    CST_LAUNCHED("link_b_setup_kernel");
    // a thread per tile, and enough threads for the -1 entries of the capacity beyond the elements
    const long long fill = n_elements / 8 > l.max_tiles ? n_elements / 8 : l.max_tiles;
    const long long want = (fill + kThreads - 1) / kThreads;
    const int tgrid = static_cast<int>(want < (long long)sm_count() * 4 ? want : (long long)sm_count() * 4);
    link_b_tiles_kernel<<<tgrid, kThreads, 0, st>>>(l.ls, l.max_tiles, static_cast<u32>(n_elements), leaf_to_node);
    CST_LAUNCHED("link_b_tiles_kernel");
    u32* pairs = l.counts + stride;
    const bool small = l.ls.tile == static_cast<u32>(kThreads * kItemsSmall);
    if (small)
        link_b_count_kernel<kItemsSmall><<<l.max_tiles, kThreads, 0, st>>>(K, l.ls, l.counts, pairs);
    else
        link_b_count_kernel<kItemsLarge><<<l.max_tiles, kThreads, 0, st>>>(K, l.ls, l.counts, pairs);
    CST_LAUNCHED("link_b_count_kernel");
    link_scan_reduce_kernel<<<dim3(l.chunks, 2), kScanThreads, 0, st>>>(l.counts, len, stride, l.partial);
    CST_LAUNCHED("link_scan_reduce_kernel");
    link_scan_apply_kernel<<<dim3(l.chunks, 2), kScanThreads, 0, st>>>(l.counts, len, stride, 1u, l.partial, nullptr,
                                                                        0u, hdr);
    CST_LAUNCHED("link_scan_apply_kernel");
    const int lo_threads = n_sets * (kNumLevels + 1);
    link_b_lo_kernel<<<(lo_threads + 255) / 256, 256, 0, st>>>(l.counts, l.ls, LO, leaf_to_node, hdr);
    CST_LAUNCHED("link_b_lo_kernel");
    const Out o{static_cast<u32>(n_nodes), NK, leaf_to_node, CO, nullptr, leaf_offsets, node_counts};
    auto* scatter = small ? (node_counts ? link_b_scatter_kernel<kItemsSmall, true>
                                         : link_b_scatter_kernel<kItemsSmall, false>)
                          : (node_counts ? link_b_scatter_kernel<kItemsLarge, true>
                                         : link_b_scatter_kernel<kItemsLarge, false>);
    scatter<<<l.max_tiles, kThreads, 0, st>>>(K, l.ls, l.counts, pairs, o);
    CST_LAUNCHED("link_b_scatter_kernel");
    return CSTONE_OK;
}

size_t link_ws_bytes(long long nl) { return link_layout(nullptr, nl).bytes; }

int launch_link(const Key* K, long long nl, Key* NK, int* CO, int* LO, int* leaf_to_node, int* parent,
                const u32* leaf_offsets, u32* node_counts, void* ws, cudaStream_t st) {
    LinkLayout l = link_layout(ws, nl);
    WsHeader* hdr = reinterpret_cast<WsHeader*>(ws);
    CST_CUDA(cudaMemsetAsync(hdr, 0, sizeof(WsHeader), st));
    const u32 n_nodes = static_cast<u32>(nl + (nl - 1) / 7), n = static_cast<u32>(nl);
    const u32 len = l.ntiles * kNumLevels;
    u32* pairs = l.counts + len;
    const bool small = items_of(nl) == kItemsSmall;
    if (small)
        link_count_kernel<kItemsSmall><<<l.ntiles, kThreads, 0, st>>>(K, n, l.counts, pairs);
    else
        link_count_kernel<kItemsLarge><<<l.ntiles, kThreads, 0, st>>>(K, n, l.counts, pairs);
    CST_LAUNCHED("link_count_kernel");
    link_scan_reduce_kernel<<<dim3(l.chunks, 2), kScanThreads, 0, st>>>(l.counts, len, len, l.partial);
    CST_LAUNCHED("link_scan_reduce_kernel");
    link_scan_apply_kernel<<<dim3(l.chunks, 2), kScanThreads, 0, st>>>(l.counts, len, len, l.ntiles, l.partial, LO,
                                                                        n_nodes, hdr);
    CST_LAUNCHED("link_scan_apply_kernel");
    const Out o{n_nodes, NK, leaf_to_node, CO, parent, leaf_offsets, node_counts};
    auto* scatter = small ? (node_counts ? link_scatter_kernel<kItemsSmall, true>
                                         : link_scatter_kernel<kItemsSmall, false>)
                          : (node_counts ? link_scatter_kernel<kItemsLarge, true>
                                         : link_scatter_kernel<kItemsLarge, false>);
    scatter<<<l.ntiles, kThreads, 0, st>>>(K, n, l.counts, pairs, o);
    CST_LAUNCHED("link_scatter_kernel");
    return CSTONE_OK;
}

// The linked tree, with its node counts when node_counts is given (then leaf_offsets [n_leaves + 1] too).
int link_tree(const char* who, const void* leaves, long long n_leaves, void* node_keys, int* child, int* level_offsets,
              int* leaf_to_node, int* parent, const u32* leaf_offsets, u32* node_counts, void* ws, size_t ws_bytes,
              cudaStream_t st) {
    if (n_leaves < 1 || n_leaves > CSTONE_MAX_LEAVES || (n_leaves - 1) % 7 != 0 || !leaves || !node_keys || !child ||
        !level_offsets || !leaf_to_node || (node_counts && !leaf_offsets))
        return cst::fail(CSTONE_ERR_INVALID_ARG, "%s: bad argument (n_leaves=%lld must be 1 + 7k, arrays non-NULL)",
                         who, n_leaves);
    if (int rc = cst::check_ws(ws, ws_bytes, link_ws_bytes(n_leaves), who)) return rc;
    return launch_link(static_cast<const Key*>(leaves), n_leaves, static_cast<Key*>(node_keys), child, level_offsets,
                       leaf_to_node, parent, leaf_offsets, node_counts, ws, st);
}

#ifndef CSTONE_KEY32  // batched builds exist for 63-bit keys only
int link_tree_batched(const char* who, const u64* elements, long long n_elements, const long long* element_offsets,
                      int n_sets, long long n_nodes, u64* node_keys, int* child, int* level_offsets, int* leaf_to_node,
                      const u32* leaf_offsets, u32* node_counts, void* ws, size_t ws_bytes, cudaStream_t st) {
    if (n_sets < 1 || n_sets > (1 << 20) || n_elements < 2 * (long long)n_sets || n_elements > CSTONE_MAX_LEAVES ||
        n_nodes < n_sets || n_nodes > 2 * (long long)CSTONE_MAX_LEAVES || !elements || !element_offsets ||
        !node_keys || !child || !level_offsets || !leaf_to_node || (node_counts && !leaf_offsets))
        return cst::fail(CSTONE_ERR_INVALID_ARG, "%s: bad argument", who);
    if (int rc = cst::check_ws(ws, ws_bytes, link_batched_ws_bytes(n_elements, n_sets), who)) return rc;
    return launch_link_batched(elements, n_elements, element_offsets, n_sets, node_keys, child, level_offsets,
                               leaf_to_node, n_nodes, leaf_offsets, node_counts, ws, st);
}
#endif

}  // namespace CST_NS

extern "C" {

int CSTONE_FN(link_workspace_size)(int64_t n_leaves, size_t* bytes) {
    if (!bytes || n_leaves < 1 || n_leaves > CSTONE_MAX_LEAVES)
        return cst::fail(CSTONE_ERR_INVALID_ARG, CST_STR(CSTONE_FN(link_workspace_size)) ": bad argument");
    *bytes = CST_NS::link_ws_bytes(n_leaves);
    return CSTONE_OK;
}

int CSTONE_FN(link_tree)(const CST_KEY_C* leaves, int64_t n_leaves, CST_KEY_C* node_keys, int32_t* child,
                         int32_t* level_offsets, int32_t* leaf_to_node, int32_t* parent, void* ws, size_t ws_bytes,
                         void* stream) {
    return CST_NS::link_tree(CST_STR(CSTONE_FN(link_tree)), leaves, n_leaves, node_keys, child, level_offsets,
                             leaf_to_node, parent, nullptr, nullptr, ws, ws_bytes, cst::as_stream(stream));
}

#ifndef CSTONE_KEY32  // batched builds exist for 63-bit keys only
int cstone_link_batched_workspace_size(int64_t n_elements, int32_t n_sets, size_t* bytes) {
    if (!bytes || n_sets < 1 || n_sets > (1 << 20) || n_elements < 2 * (int64_t)n_sets ||
        n_elements > CSTONE_MAX_LEAVES)
        return cst::fail(CSTONE_ERR_INVALID_ARG, "cstone_link_batched_workspace_size: bad argument");
    *bytes = cst::link_batched_ws_bytes(n_elements, n_sets);
    return CSTONE_OK;
}

int cstone_link_tree_batched(const uint64_t* elements, int64_t n_elements, const int64_t* element_offsets,
                             int32_t n_sets, int64_t n_nodes, uint64_t* node_keys, int32_t* child,
                             int32_t* level_offsets, int32_t* leaf_to_node, void* ws, size_t ws_bytes, void* stream) {
    return cst::link_tree_batched("cstone_link_tree_batched", reinterpret_cast<const cst::u64*>(elements), n_elements,
                                  reinterpret_cast<const long long*>(element_offsets), n_sets, n_nodes,
                                  reinterpret_cast<cst::u64*>(node_keys), child, level_offsets, leaf_to_node, nullptr,
                                  nullptr, ws, ws_bytes, cst::as_stream(stream));
}

#endif

}  // extern "C"
