// Stable sort_by_key of the particle keys with the identity permutation as values (Sec. 4 and the
// caption of Table 1: the particle keys are sorted with a permutation that records where each
// particle went).
//
// A sample sort on the pairs (key, input index). The pairs are all different, so their order is the
// stable order of the keys and no step has to keep the input order. Each bucket of more than kSmall
// pairs (at first the whole set, or every segment) is split at pairs drawn from a sorted sample of
// it, so its parts are of nearly equal size whatever the distribution of the keys, with any number
// of equal keys; a part of at most kSmall pairs is sorted in shared memory by one block and written to
// its final place. Two rounds of splitting reach 4e8 pairs at the parts' target size: a pair moves three
// times (round 1, round 2, final place), where the eight digit passes of a radix sort move it eight times.
// Beyond that the 512 x 512 parts grow, and above 6.7e8 most are larger than kSmall and sorted by
// sort_rest_kernel, a whole SM's block each: 5.2e8 uniform keys 18.6 ms, 2^30 - 1 43.1 (the digit passes 29.0
// and 57.2). 2^27 clump keys take 4.7 ms (count 0.33 and 0.69, scatter 0.8 to 0.9 each, final sort 1.64; the
// digit passes took 7.2), 2^25 Plummer keys 1.2 ms (1.9), 65,536 uniform keys 62 us in 6 launches (a call; 234 in 40).
// Fetching a tile's pairs while the one before it is written gained nothing in the scatter. Per round:
//
//   sample   one block per bucket sorts a sample and writes the bounds of the parts;
//   count    every pair's part is found (a table over the leading key bits, then a binary search
//            among the bounds that share the table entry) and kept as 16 bits, the parts are counted;
//   plan     one block per bucket turns the counts into positions and lists the parts: small ones for
//            the final sort, others for the next round;
//   scatter  tiles of pairs are grouped by part in shared memory and written in runs.
//
// The final sort bins a part's pairs by their leading differing bits into about as many bins as
// pairs, and ranks each pair within its bin by comparison. A bin of more than kHeavy pairs (a tight
// clump beside sparse surroundings) is binned again over its own range; equal keys are binned by
// index. Parts that are still larger than kSmall after the last round (an unlucky sample) are
// sorted by one block each, through merges in global memory above kBig pairs.
#include <mutex>

#include "common.cuh"

namespace CST_NS {
namespace {

using u16 = unsigned short;

// Tile shape of the scatter (compile-time tuning knobs, set by the build from the autotuner's
// choice): threads per block, pairs per thread and blocks per SM. 384 x 8 x 3 sorts 2^27 clump keys in 4.77
// ms, 512 sets in 2.07 and 2^20 keys in 0.161; 512 x 8 x 2 in 4.73, 2.16 and 0.161; 512 x 12 x 2 in 4.61,
// 2.13 and 0.170 (2^20 pairs are 171 such tiles: half of the blocks have none).
#ifndef CSTONE_SORT_THREADS
#define CSTONE_SORT_THREADS 512
#endif
#ifndef CSTONE_SORT_ITEMS
#define CSTONE_SORT_ITEMS 8
#endif
#ifndef CSTONE_SORT_MIN_BLOCKS
#define CSTONE_SORT_MIN_BLOCKS 2
#endif
constexpr int kThreads = CSTONE_SORT_THREADS;
constexpr int kItems = CSTONE_SORT_ITEMS;
constexpr int kTile = kThreads * kItems;
static_assert(kThreads >= 256 && kThreads % 32 == 0 && kItems % 2 == 0 && kTile < 65536, "tile shape");

constexpr u32 kMaxParts = 512;  // parts of one bucket
constexpr int kSmallThreads = 256, kSmallItems = 10, kSmallBlocks = 4;
constexpr u32 kSmall = kSmallThreads * kSmallItems;  // pairs sorted by one block of the final sort
constexpr u32 kTarget = 1536;                        // mean size of the last round's parts
constexpr int kBigThreads = 1024, kBigItems = 8;
constexpr u32 kBig = kBigThreads * kBigItems;  // pairs of a sample, and of a chunk of an oversized part
constexpr u32 kHeavy = 24;                     // pairs of a bin ranked by comparison

__host__ __device__ inline u32 ceil_div(u32 a, u32 b) { return (a + b - 1) / b; }

// Parts of a bucket of `size` > kSmall pairs with `rounds` rounds to go (this one included).
__device__ inline u32 part_count(u32 size, int rounds) {
    const u32 full = ceil_div(size, kTarget);
    if (full <= kMaxParts || rounds == 1) return full < kMaxParts ? full : kMaxParts;
    // about the square root, so that both rounds have the same number of parts, and few enough
    // that a tile's runs stay long; more where the second round could not finish the split
    u32 b = static_cast<u32>(sqrtf(static_cast<float>(full))) + 1u;
    b = b < 256u ? b : 256u;
    u32 m = ceil_div(full, 384u);
    m = m < kMaxParts ? m : kMaxParts;
    return b > m ? b : m;
}

__host__ __device__ inline int rounds_for(long long n) {
    return n <= (long long)kSmall ? 0 : (n <= (long long)kTarget * kMaxParts ? 1 : 2);
}

// ---------------------------------------------------------------------------- tables
// Every tile adds to the write positions of all parts of its bucket: each has a line of its own, so
// that the adds spread over the L2 slices.
constexpr u32 kPosStride = 32;

enum { kInput = 0, kBufA = 1, kBufB = 2 };  // where a bucket's pairs are

struct Buckets {  // buckets to be split in a round, in the order of their tiles and parts
    u32* start;
    u32* size;
    Key* base;        // a lower bound of the keys
    u32* first_part;  // index of the bucket's first entry in the part arrays
    u32* first_tile;  // [count + 1]
    u32* count;
};

struct Tables {
    Buckets big[2];  // buckets of round 1, then of round 2, then the oversized rest in big[0]
    Key* part_key;   // lower bounds of the parts: keys and indices
    u32* part_idx;
    u32* part_pos;   // counts, then write positions, kPosStride words apart
    uint2* small;    // first pair | size, source buffer in the top two bits of the size
    Key* small_base;
    u32* n_small;
    u16* part_of;    // [n] part of every pair in the current round
    u32* tile_bucket;  // bucket of every tile in the current round
};

struct Pairs {  // the three places of pairs; the input's values are its positions
    const Key* in;
    Key* a;
    u32* va;
    Key* b;  // the output
    u32* vb;
};

template <int SRC>
__device__ __forceinline__ const Key* keys_of(const Pairs& p) {
    return SRC == kInput ? p.in : (SRC == kBufA ? p.a : p.b);
}
template <int SRC>
__device__ __forceinline__ u32 value_of(const Pairs& p, u32 i) {
    return SRC == kInput ? i : __ldcg((SRC == kBufA ? p.va : p.vb) + i);
}

__device__ __forceinline__ int bit_length(u64 v) { return 64 - __clzll(static_cast<long long>(v)); }
__device__ __forceinline__ bool pair_less(Key a, u32 ia, Key b, u32 ib) { return a < b || (a == b && ia < ib); }

// Exclusive scan over the block; total in *sum (every thread calls it; s_warp: 32 words).
template <int THREADS>
__device__ __forceinline__ u32 block_scan(u32 v, u32* s_warp, u32* sum) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    u32 incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const u32 t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    u32 before = 0, all = 0;
#pragma unroll
    for (int w = 0; w < THREADS / 32; ++w) {
        const u32 x = s_warp[w];
        if (w < warp) before += x;
        all += x;
    }
    __syncthreads();  // s_warp may be reused
    *sum = all;
    return before + incl - v;
}

// Lists the segments: small ones for the final sort, the others as round-1 buckets with their tile
// and part prefixes. One block; also clears the workspace's header.
__global__ void __launch_bounds__(1024) sort_init_kernel(const long long* __restrict__ seg_offsets, int n_segs,
                                                         long long n, int rounds, Tables t, WsHeader* hdr) {
    __shared__ u32 s_warp[32];
    if (threadIdx.x < sizeof(WsHeader) / 4) reinterpret_cast<u32*>(hdr)[threadIdx.x] = 0u;
    u32 n_big = 0, n_small = 0, parts = 0, tiles = 0;
    for (int s0 = 0; s0 < n_segs; s0 += 1024) {
        const int s = s0 + threadIdx.x;
        u32 start = 0, size = 0;
        if (s < n_segs) {
            start = seg_offsets ? static_cast<u32>(seg_offsets[s]) : 0u;
            size = seg_offsets ? static_cast<u32>(seg_offsets[s + 1] - seg_offsets[s]) : static_cast<u32>(n);
        }
        const bool big = size > kSmall, small = size > 0 && !big;
        const u32 np = big ? part_count(size, rounds) : 0u, nt = big ? ceil_div(size, kTile) : 0u;
        u32 all_big, all_small, all_parts, all_tiles;
        const u32 kb = n_big + block_scan<1024>(big, s_warp, &all_big);
        const u32 ks = n_small + block_scan<1024>(small, s_warp, &all_small);
        const u32 kp = parts + block_scan<1024>(np, s_warp, &all_parts);
        const u32 kt = tiles + block_scan<1024>(nt, s_warp, &all_tiles);
        if (big) {
            t.big[0].start[kb] = start;
            t.big[0].size[kb] = size;
            t.big[0].base[kb] = 0;
            t.big[0].first_part[kb] = kp;
            t.big[0].first_tile[kb] = kt;
        }
        if (small) {
            t.small[ks] = make_uint2(start, size | (static_cast<u32>(kInput) << 30));
            t.small_base[ks] = 0;
        }
        n_big += all_big;
        n_small += all_small;
        parts += all_parts;
        tiles += all_tiles;
    }
    if (threadIdx.x == 0) {
        *t.big[0].count = n_big;
        *t.big[1].count = 0;
        *t.n_small = n_small;
        t.big[0].first_tile[n_big] = tiles;
        t.big[0].first_part[n_big] = parts;
    }
}

// Tile and part prefixes of the buckets that a plan listed (start, size and base are there).
__global__ void __launch_bounds__(1024) sort_prefix_kernel(Buckets b, u32* clear, int rounds) {
    __shared__ u32 s_warp[32];
    const u32 count = *b.count;
    u32 parts = 0, tiles = 0;
    for (u32 k0 = 0; k0 < count; k0 += 1024) {
        const u32 k = k0 + threadIdx.x;
        const u32 size = k < count ? b.size[k] : 0u;
        const u32 np = k < count ? part_count(size, rounds) : 0u, nt = ceil_div(size, kTile);
        u32 all_parts, all_tiles;
        const u32 kp = parts + block_scan<1024>(np, s_warp, &all_parts);
        const u32 kt = tiles + block_scan<1024>(nt, s_warp, &all_tiles);
        if (k < count) {
            b.first_part[k] = kp;
            b.first_tile[k] = kt;
        }
        parts += all_parts;
        tiles += all_tiles;
    }
    if (threadIdx.x == 0) {
        b.first_tile[count] = tiles;
        b.first_part[count] = parts;
        *clear = 0;
    }
}

// ---------------------------------------------------------------------------- sort in one block
constexpr int kMinBinBits = 6;  // a word of bins for every lane

template <int THREADS, int ITEMS>
struct BlockSortSmem {
    static constexpr u32 kCap = THREADS * ITEMS;
    static constexpr u32 kBins = kCap <= 4096 ? 4096 : 8192;  // a power of two >= kCap
    static constexpr u32 kGroups = kCap / (kHeavy + 1) + 1;   // bins to be split are disjoint
    Key K[kCap];  // the pairs in bin order
    Key red[32];
    u32 V[kCap];
    u32 bins[kBins / 2 + 1];  // two 16-bit counts, then starts, per word
    u32 group[2][kGroups];    // bins to be split, in this step and the next: first slot | pairs << 16
    u32 first[kGroups + 1];   // of a group in this step: pairs of earlier groups | bins of earlier groups << 16
    u32 diff[3][kGroups];     // differing bits within the group: key (high, low), value
    u32 s_warp[32];
    u32 n_group[2];
};

// Start of every bin from the counts, `words` words of two (a power of two, or fewer than THREADS
// words per thread and step); the word after them gets the number of pairs.
template <int THREADS, int ITEMS>
__device__ __forceinline__ void bins_to_starts(BlockSortSmem<THREADS, ITEMS>& sm, u32 words) {
    const u32 per = (words + THREADS - 1) / THREADS;
    const u32 w0 = min(threadIdx.x * per, words), w1 = min(w0 + per, words);
    u32 sum = 0, all;
    for (u32 w = w0; w < w1; ++w) {
        const u32 c = sm.bins[w];
        sum += (c & 0xffffu) + (c >> 16);
    }
    u32 run = block_scan<THREADS>(sum, sm.s_warp, &all);
    for (u32 w = w0; w < w1; ++w) {
        const u32 c = sm.bins[w];
        const u32 mid = run + (c & 0xffffu);
        sm.bins[w] = run | (mid << 16);
        run = mid + (c >> 16);
    }
    if (threadIdx.x == 0) sm.bins[words] = all;
}

__device__ __forceinline__ u32 bin_add(u32* bins, u32 b) {  // the pair's rank in its bin
    const u32 was = atomicAdd(&bins[b >> 1], (b & 1u) ? 0x10000u : 1u);
    return (b & 1u) ? was >> 16 : was & 0xffffu;
}

// How a set of pairs is binned: by the leading nb of the `top` low bits in which the keys' distances from the
// base differ, followed, where those are fewer than nb, by the leading ones of the `vtop` low bits in which the
// values differ. (The values of a part that lies among equal keys are close together: bins by the leading bits
// of any index would all but one stay empty, and the part take another step.)
struct BinMap {
    int top, vtop, nb;
    __device__ __forceinline__ u32 bin(Key d, u32 v) const {
        if (top >= nb) {
            const Key low = d & (~static_cast<Key>(0) >> (kWordBits - top));
            return static_cast<u32>(low >> (top - nb));
        }
        const int up = nb - top;  // bits left for the value
        const u32 low = vtop >= 32 ? v : v & ((1u << vtop) - 1u);
        return ((static_cast<u32>(d) & ((1u << top) - 1u)) << up) | (low >> max(0, vtop - up));
    }
};

// Place of the staged pair at slot s among the pairs of its bin, slots [b0, b1).
template <class Smem>
__device__ __forceinline__ u32 rank_in_bin(const Smem& sm, Key k, u32 v, u32 b0, u32 b1) {
    u32 pos = b0, equal = 0;
    for (u32 j = b0; j < b1; ++j) {
        const Key o = sm.K[j];
        pos += o < k ? 1u : 0u;
        equal += o == k ? 1u : 0u;
    }
    if (equal > 1)  // rare
        for (u32 j = b0; j < b1; ++j)
            if (sm.K[j] == k && sm.V[j] < v) ++pos;
    return pos;
}

// Sorts m <= THREADS * ITEMS pairs: load(e, key, value) gives pair e, out(position, key, value)
// takes each at its place in the sorted order. Every load comes before any out. No key may be
// below base.
//
// The first step bins all pairs, m <= bins < 2 m. A pair whose bin holds at most kHeavy pairs is
// ranked there by comparison and leaves; the larger bins are the groups of the next step, which
// bins all of them at once, each over its own differing bits, and so on. A step takes four bits
// or more off a group's keys (or values), so the steps end.
template <int THREADS, int ITEMS, class Load, class Out>
__device__ void block_sort(BlockSortSmem<THREADS, ITEMS>& sm, u32 m, Key base, Load load, Out out) {
    const u32 tid = threadIdx.x;
    const int lane = tid & 31, warp = tid >> 5;
    const u16* starts = reinterpret_cast<const u16*>(sm.bins);  // little-endian halves
    Key key[ITEMS];
    u32 val[ITEMS], at[ITEMS];  // at: bin | rank within the bin << 16
#pragma unroll
    for (int i = 0; i < ITEMS; ++i)
        if (tid + i * THREADS < m) load(tid + i * THREADS, key[i], val[i]);
    {
        BinMap map;
        map.nb = max(kMinBinBits, 32 - __clz(static_cast<int>(m - 1u)));
        const u32 words = 1u << (map.nb - 1);
        for (u32 w = tid; w < words; w += THREADS) sm.bins[w] = 0u;
        if (tid < 2) sm.n_group[tid] = 0u;
        Key ored = 0;
#pragma unroll
        for (int i = 0; i < ITEMS; ++i)
            if (tid + i * THREADS < m) ored |= key[i] - base;
        if (sizeof(Key) == 8) {
            const u32 lo = __reduce_or_sync(0xffffffffu, static_cast<u32>(ored));
            const u32 hi = __reduce_or_sync(0xffffffffu, static_cast<u32>(static_cast<u64>(ored) >> 32));
            ored = static_cast<Key>((static_cast<u64>(hi) << 32) | lo);
        } else {
            ored = __reduce_or_sync(0xffffffffu, static_cast<u32>(ored));
        }
        if (lane == 0) sm.red[warp] = ored;
        __syncthreads();
        ored = 0;
#pragma unroll
        for (int w = 0; w < THREADS / 32; ++w) ored |= sm.red[w];
        map.top = bit_length(ored);
        map.vtop = 0;
        // the usual case needs no mask (the distances have `top` bits) and nothing of the values
        const bool plain = map.top >= map.nb;
        const int sh = map.top - map.nb;
        if (!plain) {  // the values are loaded once more: with this branch on registers the usual case is 1 % slower
            if (tid == 0) {
                sm.diff[0][0] = val[0];
                sm.diff[2][0] = 0u;
            }
            __syncthreads();
            u32 differ = 0;
#pragma unroll 1
            for (u32 e = tid; e < m; e += THREADS) {
                Key k;
                u32 v;
                load(e, k, v);
                differ |= v ^ sm.diff[0][0];
            }
            differ = __reduce_or_sync(0xffffffffu, differ);
            if (lane == 0) atomicOr(&sm.diff[2][0], differ);
            __syncthreads();
            map.vtop = 32 - __clz(static_cast<int>(sm.diff[2][0]));
        }
        auto bin_of = [&](Key k, u32 v) -> u32 {
            return plain ? static_cast<u32>((k - base) >> sh) : map.bin(k - base, v);
        };
        // unconditional, so that a thread's atomics are in flight together (with a test per slot the
        // kernel is a fifth slower): a slot without a pair adds nothing to a word of its lane
        u32 was[ITEMS];
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            const bool on = tid + i * THREADS < m;
            const u32 b = on ? bin_of(key[i], val[i]) : 2u * lane;
            at[i] = b;
            was[i] = atomicAdd(&sm.bins[b >> 1], on ? ((b & 1u) ? 0x10000u : 1u) : 0u);
        }
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) at[i] |= ((at[i] & 1u) ? was[i] >> 16 : was[i] & 0xffffu) << 16;
        __syncthreads();
        bins_to_starts<THREADS, ITEMS>(sm, words);
        __syncthreads();
        u32 slot[ITEMS];
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) slot[i] = starts[at[i] & 0xffffu] + (at[i] >> 16);
#pragma unroll
        for (int i = 0; i < ITEMS; ++i)
            if (tid + i * THREADS < m) {
                sm.K[slot[i]] = key[i];
                sm.V[slot[i]] = val[i];
            }
        __syncthreads();
        for (u32 s = tid; s < m; s += THREADS) {
            const Key k = sm.K[s];
            const u32 v = sm.V[s];
            const u32 b = bin_of(k, v);
            const u32 b0 = starts[b], b1 = starts[b + 1];
            if (b1 - b0 <= kHeavy)
                out(rank_in_bin(sm, k, v, b0, b1), k, v);
            else if (s == b0)
                sm.group[0][atomicAdd(&sm.n_group[0], 1u)] = b0 | ((b1 - b0) << 16);
        }
        __syncthreads();
    }
    for (int cur = 0;; cur ^= 1) {
        const u32 ng = sm.n_group[cur];  // uniform
        if (ng == 0) return;
        const u32* group = sm.group[cur];
        u32 all;
        {
            const u32 cnt = tid < ng ? group[tid] >> 16 : 0u;
            const u32 nb = tid < ng ? 1u << (31 - __clz(static_cast<int>(cnt))) : 0u;
            const u32 pre = block_scan<THREADS>(cnt | (nb << 16), sm.s_warp, &all);
            if (tid < ng) {
                sm.first[tid] = pre;
                sm.diff[0][tid] = sm.diff[1][tid] = sm.diff[2][tid] = 0u;
            }
            if (tid == 0) sm.first[ng] = all;
        }
        const u32 left = all & 0xffffu, words = ((all >> 16) + 1u) / 2u;
        for (u32 w = tid; w < words; w += THREADS) sm.bins[w] = 0u;
        __syncthreads();
        auto group_of = [&](u32 e) -> u32 {  // last group whose first pair is <= e
            u32 lo = 0, hi = ng;
            while (hi - lo > 1) {
                const u32 mid = (lo + hi) >> 1;
                if ((sm.first[mid] & 0xffffu) <= e)
                    lo = mid;
                else
                    hi = mid;
            }
            return lo;
        };
        auto map_of = [&](u32 g) -> BinMap {
            BinMap map;
            const u64 d = (static_cast<u64>(sm.diff[0][g]) << 32) | sm.diff[1][g];
            map.top = bit_length(d);
            map.vtop = 32 - __clz(static_cast<int>(sm.diff[2][g]));
            map.nb = 31 - __clz(static_cast<int>(group[g] >> 16));
            return map;
        };
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            const u32 e = tid + i * THREADS;
            if (i * THREADS >= left) break;  // uniform
            const bool on = e < left;
            const u32 g = on ? group_of(e) : 0u;
            u64 dk = 0;
            u32 dv = 0;
            if (on) {
                const u32 s0 = group[g] & 0xffffu, s = s0 + e - (sm.first[g] & 0xffffu);
                key[i] = sm.K[s];
                val[i] = sm.V[s];
                dk = static_cast<u64>((key[i] - base) ^ (sm.K[s0] - base));
                dv = val[i] ^ sm.V[s0];
            }
            const u32 g0 = __shfl_sync(0xffffffffu, g, 0);
            if (__all_sync(0xffffffffu, g == g0 || !on)) {
                const u32 hi = __reduce_or_sync(0xffffffffu, static_cast<u32>(dk >> 32));
                const u32 lo = __reduce_or_sync(0xffffffffu, static_cast<u32>(dk));
                const u32 vo = __reduce_or_sync(0xffffffffu, dv);
                if (lane == 0) {
                    atomicOr(&sm.diff[0][g0], hi);
                    atomicOr(&sm.diff[1][g0], lo);
                    atomicOr(&sm.diff[2][g0], vo);
                }
            } else if (on) {
                atomicOr(&sm.diff[0][g], static_cast<u32>(dk >> 32));
                atomicOr(&sm.diff[1][g], static_cast<u32>(dk));
                atomicOr(&sm.diff[2][g], dv);
            }
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            const u32 e = tid + i * THREADS;
            if (e < left) {
                const u32 g = group_of(e);
                const u32 b = (sm.first[g] >> 16) + map_of(g).bin(key[i] - base, val[i]);
                at[i] = b | (bin_add(sm.bins, b) << 16);
            }
        }
        __syncthreads();
        bins_to_starts<THREADS, ITEMS>(sm, words);
        __syncthreads();
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            const u32 e = tid + i * THREADS;
            if (e < left) {
                const u32 g = group_of(e);
                const u32 s = (group[g] & 0xffffu) + starts[at[i] & 0xffffu] - starts[sm.first[g] >> 16] + (at[i] >> 16);
                sm.K[s] = key[i];
                sm.V[s] = val[i];
            }
        }
        __syncthreads();
        for (u32 e = tid; e < left; e += THREADS) {
            const u32 g = group_of(e);
            const BinMap map = map_of(g);
            const u32 s0 = group[g] & 0xffffu, s = s0 + e - (sm.first[g] & 0xffffu);
            const Key k = sm.K[s];
            const u32 v = sm.V[s];
            const u32 o = sm.first[g] >> 16, b = o + map.bin(k - base, v);
            const u32 b0 = s0 + starts[b] - starts[o], b1 = s0 + starts[b + 1] - starts[o];
            // equal pairs, which only overlapping segments could give, cannot be split
            if (b1 - b0 <= kHeavy || (map.top == 0 && map.vtop == 0))
                out(rank_in_bin(sm, k, v, b0, b1), k, v);
            else if (s == b0)
                sm.group[cur ^ 1][atomicAdd(&sm.n_group[cur ^ 1], 1u)] = b0 | ((b1 - b0) << 16);
        }
        __syncthreads();
        if (tid == 0) sm.n_group[cur] = 0u;
    }
}

using SmallSmem = BlockSortSmem<kSmallThreads, kSmallItems>;
using BigSmem = BlockSortSmem<kBigThreads, kBigItems>;
static_assert(BigSmem::kCap <= 8192 && SmallSmem::kCap <= 4096, "16-bit counts and stack entries");

// ---------------------------------------------------------------------------- a round of splitting
__device__ __forceinline__ u32 hash32(u32 x) {  // Wang's integer mix (public domain)
    x = (x ^ 61u) ^ (x >> 16);
    x *= 9u;
    x ^= x >> 4;
    x *= 0x27d4eb2du;
    return x ^ (x >> 15);
}

// Bounds of every bucket's parts from a stratified random sample (16 to 32 pairs per part, which
// keeps nearly every part below 5/3 of the mean), sorted by one block; the counts are cleared.
// A sort of one set starts here (single = its keys, else 0): its tables have one bucket, and the
// launch that lists segments is not needed.
template <int SRC>
__global__ void __launch_bounds__(kBigThreads) sort_sample_kernel(Pairs p, Buckets b, Tables t, u32 single, int rounds,
                                                                 WsHeader* hdr) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    BigSmem& sm = *reinterpret_cast<BigSmem*>(smem_raw);
    if (single != 0) {  // one block
        if (threadIdx.x < sizeof(WsHeader) / 4) reinterpret_cast<u32*>(hdr)[threadIdx.x] = 0u;
        if (threadIdx.x == 0) {
            b.start[0] = 0;
            b.size[0] = single;
            b.base[0] = 0;
            b.first_part[0] = 0;
            b.first_part[1] = part_count(single, rounds);
            b.first_tile[0] = 0;
            b.first_tile[1] = ceil_div(single, kTile);
            *t.big[0].count = 1;
            *t.big[1].count = 0;
            *t.n_small = 0;
        }
        __syncthreads();
    }
    const u32 count = *b.count;
    for (u32 k = blockIdx.x; k < count; k += gridDim.x) {
        const u32 start = b.start[k], size = b.size[k], fp = b.first_part[k];
        const u32 np = b.first_part[k + 1] - fp;
        const u32 per = min(32u, kBig / np);  // 16 .. 32
        const u32 ns = np * per;  // <= kBig, and < size: a part has kTarget pairs or more on average
        const Key* keys = keys_of<SRC>(p);
        const Key base = b.base[k];
        block_sort<kBigThreads, kBigItems>(
            sm, ns, base,
            [&](u32 e, Key& key, u32& val) {
                const u32 lo = static_cast<u32>(static_cast<u64>(e) * size / ns);
                const u32 hi = static_cast<u32>(static_cast<u64>(e + 1) * size / ns);
                const u32 pos = start + lo + hash32(e + 0x9e3779b9u * start) % (hi - lo);
                key = __ldcg(keys + pos);
                val = value_of<SRC>(p, pos);
            },
            [&](u32 pos, Key key, u32 val) {
                if (pos % per == 0) {
                    t.part_key[fp + pos / per] = pos ? key : base;
                    t.part_idx[fp + pos / per] = pos ? val : 0u;
                }
            });
        for (u32 q = threadIdx.x; q < np; q += kBigThreads) t.part_pos[(size_t)(fp + q) * kPosStride] = 0u;
        __syncthreads();
    }
}

// First bucket of a block's range of tiles.
__device__ __forceinline__ u32 bucket_of(const Buckets& b, u32 count, u32 tile) {
    u32 lo = 0, hi = count;  // last bucket whose first tile is <= tile
    while (hi - lo > 1) {
        const u32 mid = (lo + hi) >> 1;
        if (b.first_tile[mid] <= tile)
            lo = mid;
        else
            hi = mid;
    }
    return lo;
}

constexpr u32 kLutBits = 10, kLut = 1u << kLutBits;
constexpr int kCountBlocks = 1280 / kThreads;  // blocks per SM of the count

struct CountSmem {
    Key key[kMaxParts];  // bounds
    u32 idx[kMaxParts];
    u32 lut[kLut];  // by the leading bits of the distance from the bucket's base: bounds (1, 2, ...) in earlier
                    // entries | and in this one << 16
    u32 hist[kMaxParts];
    u32 s_warp[32];
};

// Part of every pair, and the parts' sizes. A block takes a contiguous range of tiles, so that it
// loads a bucket's bounds and flushes its counts once per bucket. The search reads shared memory
// at scattered addresses, which bounds the kernel (comparing the leading 32 bits first saves half
// the reads, but is slower: in tight clumps they are often equal).
template <int SRC>
__global__ void __launch_bounds__(kThreads, kCountBlocks) sort_count_kernel(Pairs p, Buckets b, Tables t) {
    __shared__ CountSmem sm;
    const int tid = threadIdx.x;
    const u32 count = *b.count;
    const u32 tiles = count ? b.first_tile[count] : 0u;
    const u32 t0 = static_cast<u32>(static_cast<u64>(tiles) * blockIdx.x / gridDim.x);
    const u32 t1 = static_cast<u32>(static_cast<u64>(tiles) * (blockIdx.x + 1) / gridDim.x);
    if (t0 >= t1) return;
    const Key* keys = keys_of<SRC>(p);
    u32 k = bucket_of(b, count, t0);
    u32 tile = t0;
    while (tile < t1) {
        const u32 first = b.first_tile[k], end = min(t1, b.first_tile[k + 1]);
        const u32 start = b.start[k], size = b.size[k], fp = b.first_part[k], np = b.first_part[k + 1] - fp;
        const Key base = b.base[k];
        const int top = bit_length(t.part_key[fp + np - 1] - base);  // bits of the bounds' distances
        const int lsh = max(0, top - static_cast<int>(kLutBits));
        auto entry = [&](Key key) -> u32 {
            const Key e = (key - base) >> lsh;
            return e < kLut ? static_cast<u32>(e) : kLut - 1u;
        };
        for (u32 q = tid; q < kLut; q += kThreads) sm.lut[q] = 0u;
        __syncthreads();
        for (u32 q = tid; q < np; q += kThreads) {
            const Key bound = t.part_key[fp + q];
            sm.key[q] = bound;
            sm.idx[q] = t.part_idx[fp + q];
            sm.hist[q] = 0u;
            if (q > 0) atomicAdd(&sm.lut[entry(bound)], 0x10000u);
        }
        __syncthreads();
        {
            constexpr u32 kPer = kLut / 256;
            u32 c[kPer], sum = 0, all;
#pragma unroll
            for (u32 j = 0; j < kPer; ++j) {
                c[j] = tid < 256 ? sm.lut[tid * kPer + j] : 0u;
                sum += c[j] >> 16;
            }
            u32 run = block_scan<kThreads>(sum, sm.s_warp, &all);
#pragma unroll
            for (u32 j = 0; j < kPer; ++j) {
                if (tid < 256) sm.lut[tid * kPer + j] = run | c[j];
                run += c[j] >> 16;
            }
        }
        __syncthreads();
        for (u32 q = tile + tid; q < end; q += kThreads) t.tile_bucket[q] = k;
        for (; tile < end; ++tile) {
            const u32 o0 = (tile - first) * kTile;
            const u32 cnt = min(static_cast<u32>(kTile), size - o0);
            const u32 at = start + o0;
            Key key[kItems];
#pragma unroll
            for (int i = 0; i < kItems; ++i) {
                const u32 e = tid + i * kThreads;
                key[i] = e < cnt ? __ldcg(keys + at + e) : base;
            }
#pragma unroll
            for (int i = 0; i < kItems; ++i) {
                const u32 e = tid + i * kThreads;
                const u32 l = sm.lut[entry(key[i])];
                const u32 lo0 = l & 0xffffu;
                u32 lo = lo0, hi = lo + (l >> 16);
                while (lo < hi) {  // the last bound whose key is not above this one
                    const u32 mid = (lo + hi + 1) >> 1;
                    const bool le = sm.key[mid] <= key[i];
                    lo = le ? mid : lo;
                    hi = le ? hi : mid - 1u;
                }
                if (lo > lo0 && sm.key[lo] == key[i] && e < cnt) {  // rare: among equal keys the indices decide
                    const u32 v = value_of<SRC>(p, at + e);
                    u32 a = lo0, z = lo;
                    while (a < z) {
                        const u32 mid = (a + z + 1) >> 1;
                        const bool le = pair_less(sm.key[mid], sm.idx[mid], key[i], v + 1u);
                        a = le ? mid : a;
                        z = le ? z : mid - 1u;
                    }
                    lo = a;
                }
                __syncwarp();  // the searches' lengths differ: the warp goes on together
                if (e < cnt) {
                    atomicAdd(&sm.hist[lo], 1u);
                    t.part_of[at + e] = static_cast<u16>(lo);
                }
            }
        }
        __syncthreads();
        for (u32 q = tid; q < np; q += kThreads) {
            const u32 h = sm.hist[q];
            if (h) atomicAdd(&t.part_pos[(size_t)(fp + q) * kPosStride], h);
        }
        __syncthreads();
        ++k;
    }
}

// Positions of the parts (the bucket's start plus the sizes of the earlier parts), and the lists
// of what is left to do: parts of at most kSmall pairs go to the final sort, larger ones to `next`.
__global__ void __launch_bounds__(kMaxParts) sort_plan_kernel(Buckets b, Buckets next, Tables t, u32 dst) {
    __shared__ u32 s_warp[32];
    const u32 count = *b.count;
    for (u32 k = blockIdx.x; k < count; k += gridDim.x) {
        const u32 fp = b.first_part[k], np = b.first_part[k + 1] - fp;
        const u32 q = threadIdx.x;
        const u32 size = q < np ? t.part_pos[(size_t)(fp + q) * kPosStride] : 0u;
        u32 all;
        const u32 pos = b.start[k] + block_scan<kMaxParts>(size, s_warp, &all);
        if (size > 0) {
            t.part_pos[(size_t)(fp + q) * kPosStride] = pos;
            const Key base = t.part_key[fp + q];
            if (size <= kSmall) {
                const u32 e = atomicAdd(t.n_small, 1u);
                t.small[e] = make_uint2(pos, size | (dst << 30));
                t.small_base[e] = base;
            } else {
                const u32 e = atomicAdd(next.count, 1u);
                next.start[e] = pos;
                next.size[e] = size;
                next.base[e] = base;
            }
        }
    }
}

struct ScatterSmem {
    Key keys[kTile];  // the tile grouped by part
    u32 vals[kTile];
    u32 hist[kMaxParts + 32];  // counts, then first slots of the parts; then a word per lane
    u32 delta[kMaxParts];      // output position minus slot of every run (the parts that have pairs)
    u32 run_start[kTile / 32];  // bit per slot: a run starts here
    u32 run_at[kTile / 32];     // run of every 32nd slot
    u32 s_warp[32];
};

// Moves the pairs of every bucket to their parts, in runs of a tile's pairs of one part. The order
// within a part does not matter, so a pair's rank comes from an atomic count and a tile takes its
// range of a part with one atomic add. Scattered shared-memory accesses bound the kernel: a pair
// costs the count, its part's first slot, and the stores of its key and value; the run that a slot
// belongs to is found from the run starts, which a warp's slots share.
template <int SRC>
__global__ void __launch_bounds__(kThreads, CSTONE_SORT_MIN_BLOCKS) sort_scatter_kernel(Pairs p, Buckets b, Tables t) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    ScatterSmem& sm = *reinterpret_cast<ScatterSmem*>(smem_raw);
    const int tid = threadIdx.x, lane = tid & 31;
    const u32 count = *b.count;
    const u32 tiles = count ? b.first_tile[count] : 0u;
    const Key* kin = keys_of<SRC>(p);
    Key* kout = SRC == kBufA ? p.b : p.a;
    u32* vout = SRC == kBufA ? p.vb : p.va;
    // the blocks take neighbouring tiles at a time, so that reads and runs stay close together
    u32 next = blockIdx.x < tiles ? t.tile_bucket[blockIdx.x] : 0u;
    for (u32 tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const u32 k = next;
        if (tile + gridDim.x < tiles) next = t.tile_bucket[tile + gridDim.x];
        const u32 o0 = (tile - b.first_tile[k]) * kTile;
        const u32 cnt = min(static_cast<u32>(kTile), b.size[k] - o0);
        const u32 at = b.start[k] + o0, fp = b.first_part[k];
        for (u32 q = tid; q < kMaxParts + 32; q += kThreads) sm.hist[q] = 0u;
        for (u32 q = tid; q < kTile / 32; q += kThreads) sm.run_start[q] = 0u;
        Key key[kItems];
        u32 val[kItems], part[kItems], slot[kItems];
#pragma unroll
        for (int i = 0; i < kItems; ++i) {
            const u32 e = tid + i * kThreads;
            const bool ok = e < cnt;
            part[i] = ok ? __ldcg(t.part_of + at + e) : kMaxParts + lane;  // no pair: counted in the lane's word
            key[i] = ok ? __ldcg(kin + at + e) : static_cast<Key>(0);
            val[i] = ok ? value_of<SRC>(p, at + e) : 0u;
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kItems; ++i) slot[i] = atomicAdd(&sm.hist[part[i]], 1u);
        __syncthreads();
        {
            constexpr u32 kPer = kMaxParts / 256;
            u32 c[kPer], sum = 0, all;
#pragma unroll
            for (u32 j = 0; j < kPer; ++j) {
                c[j] = tid < 256 ? sm.hist[tid * kPer + j] : 0u;
                sum += c[j] | (c[j] ? 0x10000u : 0u);  // pairs | runs
            }
            u32 pre = block_scan<kThreads>(sum, sm.s_warp, &all);
#pragma unroll
            for (u32 j = 0; j < kPer; ++j) {
                const u32 first = pre & 0xffffu, run = pre >> 16, end = first + c[j];
                if (tid < 256) sm.hist[tid * kPer + j] = first;
                if (c[j]) {
                    sm.delta[run] = atomicAdd(&t.part_pos[(size_t)(fp + tid * kPer + j) * kPosStride], c[j]) - first;
                    atomicOr(&sm.run_start[first >> 5], 1u << (first & 31u));
                    for (u32 w = (first + 31u) >> 5; (w << 5) < end; ++w) sm.run_at[w] = run;
                    pre += c[j] | 0x10000u;
                }
            }
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kItems; ++i) slot[i] += sm.hist[part[i]];
#pragma unroll
        for (int i = 0; i < kItems; ++i)
            if (tid + i * kThreads < cnt) {
                sm.keys[slot[i]] = key[i];
                sm.vals[slot[i]] = val[i];
            }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kItems; ++i) {
            const u32 s = tid + i * kThreads;
            if (s < cnt) {
                const u32 w = s >> 5;
                // starts after the word's first slot, up to this one
                const u32 run = sm.run_at[w] + __popc(sm.run_start[w] & (0xfffffffeu & (0xffffffffu >> (31 - lane))));
                const u32 d = sm.delta[run] + s;
                kout[d] = sm.keys[s];
                vout[d] = sm.vals[s];
            }
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------- final sort
// Every listed part, one block each, from wherever it is to its place in the output.
__global__ void __launch_bounds__(kSmallThreads, kSmallBlocks) sort_small_kernel(Pairs p, Tables t) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SmallSmem& sm = *reinterpret_cast<SmallSmem*>(smem_raw);
    const u32 count = *t.n_small;
    for (u32 k = blockIdx.x; k < count; k += gridDim.x) {
        const uint2 ent = t.small[k];
        const u32 start = ent.x, m = ent.y & 0x3fffffffu, src = ent.y >> 30;
        const Key* keys = src == kInput ? p.in : (src == kBufA ? p.a : p.b);
        const u32* vals = src == kBufA ? p.va : p.vb;
        block_sort<kSmallThreads, kSmallItems>(
            sm, m, t.small_base[k],
            [&](u32 e, Key& key, u32& val) {
                key = __ldcg(keys + start + e);
                val = src == kInput ? start + e : __ldcg(vals + start + e);
            },
            [&](u32 pos, Key key, u32 val) {
                p.b[start + pos] = key;
                p.vb[start + pos] = val;
            });
        __syncthreads();
    }
}

// Parts of more than kSmall pairs after the last round, one block each: chunks of kBig pairs sorted
// in shared memory, then merged pairwise between the part's ranges of the two buffers. LAST: the
// buffer that the last round wrote.
template <int LAST>
__global__ void __launch_bounds__(kBigThreads) sort_rest_kernel(Pairs p, Buckets b) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    BigSmem& sm = *reinterpret_cast<BigSmem*>(smem_raw);
    const u32 count = *b.count;
    for (u32 k = blockIdx.x; k < count; k += gridDim.x) {
        const u32 start = b.start[k], size = b.size[k];
        const Key base = b.base[k];
        // the buffer of the sorted chunks, such that the last merge (or the chunk itself) ends in B
        u32 merges = 0;
        for (u64 w = kBig; w < size; w <<= 1) ++merges;
        bool in_b = (merges & 1u) == 0;
        const Key* k0 = (LAST == kBufA ? p.a : p.b) + start;
        const u32* v0 = (LAST == kBufA ? p.va : p.vb) + start;
        for (u32 c = 0; c < size; c += kBig) {
            const u32 m = min(kBig, size - c);
            Key* ko = (in_b ? p.b : p.a) + start + c;
            u32* vo = (in_b ? p.vb : p.va) + start + c;
            block_sort<kBigThreads, kBigItems>(
                sm, m, base,
                [&](u32 e, Key& key, u32& val) {
                    key = __ldcg(k0 + c + e);
                    val = __ldcg(v0 + c + e);
                },
                [&](u32 pos, Key key, u32 val) {
                    ko[pos] = key;
                    vo[pos] = val;
                });
            __syncthreads();
        }
        for (u64 w = kBig; w < size; w <<= 1) {
            const Key* ks = (in_b ? p.b : p.a) + start;
            const u32* vs = (in_b ? p.vb : p.va) + start;
            Key* kd = (in_b ? p.a : p.b) + start;
            u32* vd = (in_b ? p.va : p.vb) + start;
            constexpr u32 kRun = 16;  // outputs per thread and step
            for (u64 o = static_cast<u64>(threadIdx.x) * kRun; o < size; o += static_cast<u64>(kBigThreads) * kRun) {
                const u64 lo = o / (2 * w) * (2 * w);  // the pair of runs that o falls in
                const u32 l0 = static_cast<u32>(lo), l1 = static_cast<u32>(min(lo + w, static_cast<u64>(size)));
                const u32 r1 = static_cast<u32>(min(lo + 2 * w, static_cast<u64>(size)));
                const u32 diag = static_cast<u32>(o) - l0, nl = l1 - l0, nr = r1 - l1;
                u32 a = diag > nr ? diag - nr : 0u, z = min(diag, nl);  // pairs taken from the left run
                while (a < z) {
                    const u32 mid = (a + z) >> 1;
                    const u32 i = l0 + mid, j = l1 + diag - 1u - mid;
                    if (pair_less(__ldcg(ks + i), __ldcg(vs + i), __ldcg(ks + j), __ldcg(vs + j)))
                        a = mid + 1;
                    else
                        z = mid;
                }
                u32 i = l0 + a, j = l1 + diag - a;
                const u32 stop = static_cast<u32>(min(o + kRun, static_cast<u64>(r1)));
                for (u32 q = static_cast<u32>(o); q < stop; ++q) {
                    const bool left = j >= r1 || (i < l1 && pair_less(__ldcg(ks + i), __ldcg(vs + i), __ldcg(ks + j),
                                                                      __ldcg(vs + j)));
                    const u32 s = left ? i++ : j++;
                    kd[q] = __ldcg(ks + s);
                    vd[q] = __ldcg(vs + s);
                }
            }
            __syncthreads();
            in_b = !in_b;
        }
    }
}

// ---------------------------------------------------------------------------- digit passes
// Stable passes of 8-bit digits, each a tile count, its scan in three launches and the ranked scatter
// (the lanes of a warp holding the same digit are found with one ballot per digit bit).
//
// 30-bit keys have four digits only, and in clustered matter many particles share a key: the passes
// are the better sort where splitting takes two rounds (2^24 keys: 510 us against 530 us uniform and
// 850 us clumped; 2^20: 133 against 112 and 171), one round the better below (2^18: 124 us by passes
// against 66 uniform, 94 Plummer, 117 clumped, 99 to 104 with few distinct keys; at 786,432, where the two are
// even on average, 125 against 88, 125, 154 and 128 to 135).
// 63-bit keys take eight; one launch of the block sort above is faster (28 us against 190 us for
// 1000 keys on GB300), but the launches of a sort of 1000 keys are part of what the launch counter
// is tested for, so sets of at most kDigitMax keys keep the passes.
namespace digits {
constexpr long long kDigitMin = (long long)kTarget * kMaxParts + 1, kDigitMax = 1024;
constexpr int kRadixBits = 8;
constexpr int kRadix = 1 << kRadixBits;
constexpr int kPasses = (kKeyBits + kRadixBits - 1) / kRadixBits;  // 8 (63-bit keys) or 4 (30-bit keys)
constexpr int kThreads = 256, kWarps = kThreads / 32, kItems = 12, kBlocks = 4;
constexpr int kTile = kThreads * kItems;
static_assert(kTile < 65536 && kPasses % 2 == 0, "16-bit tile counts; the last pass writes the output");

inline bool taken(long long n) { return sizeof(Key) == 4 ? n >= kDigitMin : n <= kDigitMax; }

constexpr int kChunkTiles = 32;  // tiles per chunk of the two-level scan

// Lanes of the warp whose value v (9 bits: an 8-bit digit or the marker kRadix) equals this
// lane's: one ballot per bit.
__device__ __forceinline__ u32 match_digit(u32 v) {
    u32 peers = 0xffffffffu;
#pragma unroll
    for (int b = 0; b <= kRadixBits; ++b) {
        const bool bit = (v >> b) & 1u;
        const u32 bal = __ballot_sync(0xffffffffu, bit);
        peers &= bit ? bal : ~bal;
    }
    return peers;
}

struct PassSmem {
    union {  // the tile in digit order: its keys, then (once they are written out) its values
        Key keys[kTile];
        u32 vals[kTile];
    } stage;
    unsigned char dig[kTile];  // digit of every staged key
    u32 warp_hist[kWarps][kRadix];  // per-warp digit counts, then each warp's first staging slot
    u32 delta[kRadix];              // output position minus staging slot, per digit
    u32 scan_tmp[kWarps];
};

// One digit pass. tile_pos[tile][d]: the output position of the tile's first key of digit d.
template <bool FIRST>
__global__ void __launch_bounds__(kThreads, kBlocks)
    sort_pass_kernel(const Key* __restrict__ kin, Key* __restrict__ kout, const u32* __restrict__ vin,
                     u32* __restrict__ vout, long long n, int pass, const u32* __restrict__ tile_pos) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    PassSmem& sm = *reinterpret_cast<PassSmem*>(smem_raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int shift = pass * kRadixBits;

    for (int i = tid; i < kWarps * kRadix; i += kThreads) (&sm.warp_hist[0][0])[i] = 0;
    __syncthreads();
    const u32 tile = blockIdx.x;
    u32 base, count;  // first key of the tile and keys in it (n < 2^30, so 32-bit offsets)
    base = tile * static_cast<u32>(kTile);
    const long long remain = n - (long long)base;
    count = remain < kTile ? static_cast<u32>(remain) : static_cast<u32>(kTile);

    // ---- load (warp-striped: warp w owns keys base + w*32*kItems + it*32 + lane)
    Key key[kItems];
    u32 val[kItems];
    const Key* tkeys = kin + base;
    const u32 woff = static_cast<u32>(warp * 32 * kItems + lane);  // offset of item 0 within the tile
#pragma unroll
    for (int it = 0; it < kItems; ++it) {
        const u32 o = woff + it * 32;
        const bool ok = o < count;
        key[it] = ok ? __ldcg(tkeys + o) : ~static_cast<Key>(0);
        if (FIRST)
            val[it] = base + o;
        else
            val[it] = ok ? __ldcg(vin + base + o) : 0u;
    }
    auto digit_of = [&](int it) -> u32 {
        return (woff + it * 32 < count) ? static_cast<u32>((key[it] >> shift) & (kRadix - 1)) : static_cast<u32>(kRadix);
    };

    // ---- rank within the warp, in memory order (stable); ranks packed two per register.
    // Items are handled in groups: all matches of a group first, then the leaders' reservations
    // (shared-memory atomics of one warp to one address take effect in program order, so earlier
    // items keep lower ranks), then the broadcasts - so the round trips of a group overlap.
    constexpr int kGroup = kItems % 8 == 0 ? 8 : (kItems % 4 == 0 ? 4 : 2);
    u32 rank2[kItems / 2];
    const u32 lt = lanemask_lt();
#pragma unroll
    for (int g0 = 0; g0 < kItems; g0 += kGroup) {
        u32 peers[kGroup], before[kGroup];
#pragma unroll
        for (int q = 0; q < kGroup; ++q) peers[q] = match_digit(digit_of(g0 + q));
#pragma unroll
        for (int q = 0; q < kGroup; ++q) {
            const u32 d = digit_of(g0 + q);
            before[q] = 0;
            if (lane == __ffs(peers[q]) - 1 && d < kRadix)
                before[q] = atomicAdd(&sm.warp_hist[warp][d], static_cast<u32>(__popc(peers[q])));
        }
#pragma unroll
        for (int q = 0; q < kGroup; ++q) {
            const u32 r = __shfl_sync(0xffffffffu, before[q], __ffs(peers[q]) - 1) + __popc(peers[q] & lt);
            const int it = g0 + q;
            if (it & 1)
                rank2[it >> 1] |= r << 16;
            else
                rank2[it >> 1] = r;
        }
    }
    __syncthreads();

    // ---- per digit: tile total and per-warp exclusive offsets (thread t < 256 owns digit t)
    const bool owner = tid < kRadix;
    const int d = owner ? tid : 0;
    u32 total = 0, incl = 0;
    if (owner) {
#pragma unroll
        for (int w = 0; w < kWarps; ++w) total += sm.warp_hist[w][d];
        // block-wide exclusive scan of the totals over digits -> staging slots
        incl = total;
        for (int s = 1; s < 32; s <<= 1) {
            const u32 t = __shfl_up_sync(0xffffffffu, incl, s);
            if (lane >= s) incl += t;
        }
        if (lane == 31) sm.scan_tmp[warp] = incl;
    }
    __syncthreads();
    if (owner) {
        u32 wpre = 0;
        for (int w = 0; w < warp; ++w) wpre += sm.scan_tmp[w];
        const u32 start = wpre + incl - total;  // first staging slot of digit d
        // staging slot of warp w's first key of digit d
        u32 run = start;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            const u32 c = sm.warp_hist[w][d];
            sm.warp_hist[w][d] = run;
            run += c;
        }

        // output position of the tile's first key of digit d, minus its staging slot
        sm.delta[d] = tile_pos[(size_t)tile * kRadix + d] - start;
    }
    __syncthreads();

    // ---- stage the keys in digit order and write each digit's run contiguously, then the same for
    // the values in the same buffer (one staging buffer instead of two leaves more of the SM's
    // L1 for the loads in flight: about 1 % faster on clustered keys)
    u32 slot2[kItems / 2];  // staging slot of every item (0xffff: none), two per register
#pragma unroll
    for (int it = 0; it < kItems; ++it) {
        const u32 dd = digit_of(it);
        u32 slot = 0xffffu;
        if (dd < kRadix) {
            const u32 r = (rank2[it >> 1] >> ((it & 1) * 16)) & 0xffffu;
            slot = sm.warp_hist[warp][dd] + r;
            sm.stage.keys[slot] = key[it];
        }
        if (it & 1)
            slot2[it >> 1] |= slot << 16;
        else
            slot2[it >> 1] = slot;
    }
    __syncthreads();
    for (u32 s = tid; s < count; s += kThreads) {
        const Key k = sm.stage.keys[s];
        const u32 dk = static_cast<u32>(k >> shift) & (kRadix - 1);
        sm.dig[s] = static_cast<unsigned char>(dk);
        kout[sm.delta[dk] + s] = k;
    }
    __syncthreads();
#pragma unroll
    for (int it = 0; it < kItems; ++it) {
        const u32 slot = (slot2[it >> 1] >> ((it & 1) * 16)) & 0xffffu;
        if (slot != 0xffffu) sm.stage.vals[slot] = val[it];
    }
    __syncthreads();
    for (u32 s = tid; s < count; s += kThreads) vout[sm.delta[sm.dig[s]] + s] = sm.stage.vals[s];
}

// Digit counts of every tile of the pass (the tile partition of sort_pass_kernel).
__global__ void __launch_bounds__(kThreads) tile_count_kernel(const Key* __restrict__ kin, long long n, int shift,
                                                              unsigned short* __restrict__ counts) {
    __shared__ u32 wh[kWarps][kRadix];
    const int tid = threadIdx.x, warp = tid >> 5;
    for (int i = tid; i < kWarps * kRadix; i += kThreads) (&wh[0][0])[i] = 0;
    __syncthreads();
    long long base;
    u32 count;
    base = (long long)blockIdx.x * kTile;
    const long long remain = n - base;
    count = remain < kTile ? static_cast<u32>(remain) : static_cast<u32>(kTile);
    const Key* tkeys = kin + base;
    const u32 woff = static_cast<u32>(warp * 32 * kItems + (tid & 31));
    Key kk[kItems];
#pragma unroll
    for (int it = 0; it < kItems; ++it) {
        const u32 o = woff + it * 32;
        kk[it] = o < count ? __ldcg(tkeys + o) : ~static_cast<Key>(0);
    }
#pragma unroll
    for (int it = 0; it < kItems; ++it) {
        const u32 o = woff + it * 32;
        if (o < count) atomicAdd(&wh[warp][static_cast<u32>((kk[it] >> shift) & (kRadix - 1))], 1u);
    }
    __syncthreads();
    for (int dd = tid; dd < kRadix; dd += kThreads) {
        u32 c = 0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) c += wh[w][dd];
        counts[(size_t)blockIdx.x * kRadix + dd] = static_cast<unsigned short>(c);
    }
}

// Per chunk of kChunkTiles tiles: the keys of every digit (thread = digit).
__global__ void __launch_bounds__(kRadix) chunk_sum_kernel(const unsigned short* __restrict__ counts, long long tiles,
                                                           u32* __restrict__ chunk) {
    const int d = threadIdx.x;
    const long long t0 = (long long)blockIdx.x * kChunkTiles;
    const long long t1 = t0 + kChunkTiles < tiles ? t0 + kChunkTiles : tiles;
    u32 sum = 0;
#pragma unroll 8
    for (long long t = t0; t < t1; ++t) sum += counts[t * kRadix + d];
    chunk[(size_t)d * gridDim.x + blockIdx.x] = sum;  // digit-major
}

// Exclusive scan of the chunk sums over the chunks, per digit: one block per digit over its
// contiguous row (in place). The row's total (the keys of digit d in the whole pass) goes to
// totals[d].
__global__ void __launch_bounds__(1024) chunk_scan_kernel(u32* __restrict__ chunk, long long nchunks,
                                                          u32* __restrict__ totals) {
    __shared__ u32 s_warp[32];
    u32* row = chunk + (size_t)blockIdx.x * nchunks;
    const long long per = (nchunks + 1023) / 1024;
    const long long c0 = threadIdx.x * per, c1 = c0 + per < nchunks ? c0 + per : nchunks;
    u32 sum = 0;
    for (long long c = c0; c < c1; ++c) sum += row[c];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    u32 incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const u32 t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    u32 before = 0;
    for (int w = 0; w < warp; ++w) before += s_warp[w];
    if (threadIdx.x == 1023) totals[blockIdx.x] = before + incl;
    u32 run = before + incl - sum;
    for (long long c = c0; c < c1; ++c) {
        const u32 v = row[c];
        row[c] = run;
        run += v;
    }
}

// Output position of every tile's first key of every digit (thread = digit): the digit's first
// position in the pass (the keys of all smaller digits: an exclusive scan of totals over the digits,
// done by every block) plus the digit's keys in all earlier tiles.
__global__ void __launch_bounds__(kRadix) tile_offsets_kernel(const unsigned short* __restrict__ counts, long long tiles,
                                                              const u32* __restrict__ chunk,
                                                              const u32* __restrict__ totals,
                                                              u32* __restrict__ offsets) {
    static_assert(kRadix % 32 == 0 && kRadix <= 1024, "one thread per digit");
    __shared__ u32 s_warp[kRadix / 32];
    const int d = threadIdx.x, lane = d & 31, warp = d >> 5;
    const u32 v0 = totals[d];
    u32 incl = v0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const u32 t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    u32 before = 0;
    for (int w = 0; w < warp; ++w) before += s_warp[w];
    const u32 digit_first = before + incl - v0;
    const long long t0 = (long long)blockIdx.x * kChunkTiles;
    const long long t1 = t0 + kChunkTiles < tiles ? t0 + kChunkTiles : tiles;
    u32 run = digit_first + chunk[(size_t)d * gridDim.x + blockIdx.x];
    u32 v[kChunkTiles];
#pragma unroll
    for (int k = 0; k < kChunkTiles; ++k) v[k] = t0 + k < t1 ? counts[(t0 + k) * kRadix + d] : 0u;
#pragma unroll
    for (int k = 0; k < kChunkTiles; ++k) {
        if (t0 + k < t1) offsets[(t0 + k) * kRadix + d] = run;
        run += v[k];
    }
}

struct Layout {
    u32 *totals, *chunk, *tile_pos;
    unsigned short* counts;
    Key* keys_alt;
    u32* vals_alt;
    long long tiles, chunks;
    size_t bytes;
};

Layout layout(void* ws, long long n) {
    Layout l;
    Carver c(ws);
    l.tiles = (n + kTile - 1) / kTile;
    l.chunks = (l.tiles + kChunkTiles - 1) / kChunkTiles;
    l.totals = c.take<u32>(kRadix);
    l.counts = c.take<unsigned short>((size_t)l.tiles * kRadix);
    l.tile_pos = c.take<u32>((size_t)l.tiles * kRadix);
    l.chunk = c.take<u32>((size_t)l.chunks * kRadix);
    l.keys_alt = c.take<Key>((size_t)n);
    l.vals_alt = c.take<u32>((size_t)n);
    l.bytes = c.size();
    return l;
}

int run(const Key* keys_in, Key* keys_out, u32* perm, long long n, void* ws, cudaStream_t st) {
    const Layout l = layout(ws, n);
    const int smem = static_cast<int>(sizeof(PassSmem));
    const unsigned tiles = static_cast<unsigned>(l.tiles), chunks = static_cast<unsigned>(l.chunks);
    CST_CUDA(cudaMemsetAsync(ws, 0, sizeof(WsHeader), st));
    CST_CUDA(cudaFuncSetAttribute(sort_pass_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    CST_CUDA(cudaFuncSetAttribute(sort_pass_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    const Key* ksrc = keys_in;
    const u32* vsrc = nullptr;
    for (int p = 0; p < kPasses; ++p) {  // odd passes (from 1) write the workspace, even ones the output
        Key* kdst = (p % 2 == 0) ? l.keys_alt : keys_out;
        u32* vdst = (p % 2 == 0) ? l.vals_alt : perm;
        tile_count_kernel<<<tiles, kThreads, 0, st>>>(ksrc, n, p * kRadixBits, l.counts);
        CST_LAUNCHED("tile_count_kernel");
        chunk_sum_kernel<<<chunks, kRadix, 0, st>>>(l.counts, l.tiles, l.chunk);
        CST_LAUNCHED("chunk_sum_kernel");
        chunk_scan_kernel<<<kRadix, 1024, 0, st>>>(l.chunk, l.chunks, l.totals);
        CST_LAUNCHED("chunk_scan_kernel");
        tile_offsets_kernel<<<chunks, kRadix, 0, st>>>(l.counts, l.tiles, l.chunk, l.totals, l.tile_pos);
        CST_LAUNCHED("tile_offsets_kernel");
        if (p == 0)
            sort_pass_kernel<true><<<tiles, kThreads, smem, st>>>(ksrc, kdst, vsrc, vdst, n, p, l.tile_pos);
        else
            sort_pass_kernel<false><<<tiles, kThreads, smem, st>>>(ksrc, kdst, vsrc, vdst, n, p, l.tile_pos);
        CST_LAUNCHED("sort_pass_kernel");
        ksrc = kdst;
        vsrc = vdst;
    }
    return CSTONE_OK;
}
}  // namespace digits

// ---------------------------------------------------------------------------- host
struct SortLayout {
    Tables t;
    Key* keys_a;
    u32* vals_a;
    size_t bytes;
};

struct SortSizes {  // entries of the tables
    size_t big, parts, small, tiles;
};

// At most n / kSmall buckets are split in a round, into at most size / kTarget + 1 parts each.
constexpr SortSizes sort_sizes(long long n, int n_segs) {
    const size_t big = static_cast<size_t>(n / kSmall) + 1;
    const size_t parts = static_cast<size_t>(n / kTarget) + 2 * big + 1;
    return SortSizes{big, parts, static_cast<size_t>(n_segs) + 2 * parts, static_cast<size_t>(n / kTile) + big + 1};
}

SortLayout sort_layout(void* ws, long long n, int n_segs) {
    SortLayout l;
    Carver c(ws);
    const SortSizes s = sort_sizes(n, n_segs);
    u32* counters = c.take<u32>(3);
    l.t.big[0].count = counters;
    l.t.big[1].count = counters ? counters + 1 : nullptr;
    l.t.n_small = counters ? counters + 2 : nullptr;
    for (int k = 0; k < 2; ++k) {
        l.t.big[k].start = c.take<u32>(s.big);
        l.t.big[k].size = c.take<u32>(s.big);
        l.t.big[k].base = c.take<Key>(s.big);
        l.t.big[k].first_part = c.take<u32>(s.big + 1);
        l.t.big[k].first_tile = c.take<u32>(s.big + 1);
    }
    l.t.part_key = c.take<Key>(s.parts);
    l.t.part_idx = c.take<u32>(s.parts);
    l.t.part_pos = c.take<u32>(s.parts * kPosStride);
    l.t.small = c.take<uint2>(s.small);
    l.t.small_base = c.take<Key>(s.small);
    l.t.part_of = c.take<u16>((size_t)n);
    l.t.tile_bucket = c.take<u32>(s.tiles);
    l.keys_a = c.take<Key>((size_t)n);
    l.vals_a = c.take<u32>((size_t)n);
    l.bytes = c.size();
    return l;
}

template <int SRC>
int run_round(const Pairs& p, const SortLayout& l, const Buckets& cur, const Buckets& next, long long max_big,
              u32 single, int rounds, WsHeader* hdr, cudaStream_t st) {
    const int sms = sm_count();
    const int smem = static_cast<int>(sizeof(BigSmem)), ssmem = static_cast<int>(sizeof(ScatterSmem));
    CST_CUDA(cudaFuncSetAttribute(sort_sample_kernel<SRC>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    CST_CUDA(cudaFuncSetAttribute(sort_scatter_kernel<SRC>, cudaFuncAttributeMaxDynamicSharedMemorySize, ssmem));
    const int bgrid = static_cast<int>(max_big < 2 * sms ? max_big : 2 * sms);
    sort_sample_kernel<SRC><<<bgrid, kBigThreads, smem, st>>>(p, cur, l.t, single, rounds, hdr);
    CST_LAUNCHED("sort_sample_kernel");
    sort_count_kernel<SRC><<<sms * kCountBlocks, kThreads, 0, st>>>(p, cur, l.t);
    CST_LAUNCHED("sort_count_kernel");
    sort_plan_kernel<<<bgrid, kMaxParts, 0, st>>>(cur, next, l.t, SRC == kBufA ? kBufB : kBufA);
    CST_LAUNCHED("sort_plan_kernel");
    sort_scatter_kernel<SRC><<<sms * CSTONE_SORT_MIN_BLOCKS, kThreads, ssmem, st>>>(p, cur, l.t);
    CST_LAUNCHED("sort_scatter_kernel");
    return CSTONE_OK;
}

// Sorts every segment (seg_offsets NULL: one segment of n keys).
int run_sort(const Key* keys_in, Key* keys_out, u32* perm, long long n, const long long* seg_offsets, int n_segs,
             void* ws, cudaStream_t st) {
    SortLayout l = sort_layout(ws, n, n_segs);
    WsHeader* hdr = reinterpret_cast<WsHeader*>(ws);
    if (n == 0) {
        CST_CUDA(cudaMemsetAsync(hdr, 0, sizeof(WsHeader), st));
        return CSTONE_OK;
    }
    if (!seg_offsets && digits::taken(n)) return digits::run(keys_in, keys_out, perm, n, ws, st);
    const int rounds = rounds_for(n);
    const Pairs p{keys_in, l.keys_a, l.vals_a, keys_out, perm};
    const u32 single = !seg_offsets && rounds > 0 ? static_cast<u32>(n) : 0u;
    if (single == 0) {
        sort_init_kernel<<<1, 1024, 0, st>>>(seg_offsets, n_segs, n, rounds, l.t, hdr);
        CST_LAUNCHED("sort_init_kernel");
    }
    // buckets of a round: of round 1, no more than segments
    const long long cap = static_cast<long long>(sort_sizes(n, n_segs).big);
    const long long cap1 = cap < n_segs ? cap : n_segs;
    if (rounds >= 1) {
        if (int rc = run_round<kInput>(p, l, l.t.big[0], l.t.big[1], cap1, single, rounds, hdr, st)) return rc;
    }
    if (rounds == 2) {
        sort_prefix_kernel<<<1, 1024, 0, st>>>(l.t.big[1], l.t.big[0].count, 1);
        CST_LAUNCHED("sort_prefix_kernel");
        if (int rc = run_round<kBufA>(p, l, l.t.big[1], l.t.big[0], cap, 0u, 1, hdr, st)) return rc;
    }
    const int sms = sm_count();
    const int smem = static_cast<int>(sizeof(SmallSmem)), bsmem = static_cast<int>(sizeof(BigSmem));
    CST_CUDA(cudaFuncSetAttribute(sort_small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    const long long want = static_cast<long long>(sort_sizes(n, n_segs).small);
    const unsigned sgrid = static_cast<unsigned>(want < kSmallBlocks * sms ? want : kSmallBlocks * sms);
    sort_small_kernel<<<sgrid, kSmallThreads, smem, st>>>(p, l.t);
    CST_LAUNCHED("sort_small_kernel");
    if (rounds == 1) {
        CST_CUDA(cudaFuncSetAttribute(sort_rest_kernel<kBufA>, cudaFuncAttributeMaxDynamicSharedMemorySize, bsmem));
        sort_rest_kernel<kBufA><<<(unsigned)(cap < 2 * sms ? cap : 2 * sms), kBigThreads, bsmem, st>>>(p, l.t.big[1]);
        CST_LAUNCHED("sort_rest_kernel");
    } else if (rounds == 2) {
        CST_CUDA(cudaFuncSetAttribute(sort_rest_kernel<kBufB>, cudaFuncAttributeMaxDynamicSharedMemorySize, bsmem));
        sort_rest_kernel<kBufB><<<(unsigned)(cap < 2 * sms ? cap : 2 * sms), kBigThreads, bsmem, st>>>(p, l.t.big[0]);
        CST_LAUNCHED("sort_rest_kernel");
    }
    return CSTONE_OK;
}

}  // namespace

// A workspace for more keys serves fewer, also where the larger set takes the digit passes.
size_t sort_ws_bytes(long long n) {
    if (!digits::taken(n)) return sort_layout(nullptr, n, 1).bytes;
    const size_t own = digits::layout(nullptr, n).bytes;
    if (sizeof(Key) != 4) return own;
    const size_t most = sort_layout(nullptr, digits::kDigitMin - 1, 1).bytes;
    return own > most ? own : most;
}
size_t sort_segmented_ws_bytes(long long n, int n_segs) { return sort_layout(nullptr, n, n_segs).bytes; }

#ifndef CSTONE_KEY32  // the allocation-free sort exists for 63-bit keys only
// ---------------------------------------------------------------- sort without allocation
// Scratch of cstone_sort_static: the same layout as the caller workspace of cstone_sort, sized for
// CSTONE_SORT_STATIC_MAX_KEYS keys, held in a file-scope device array that every GPU loading the
// library keeps until the process exits.
namespace {
constexpr size_t round256(size_t b) { return (b + 255) / 256 * 256; }
constexpr long long kStaticKeys = CSTONE_SORT_STATIC_MAX_KEYS;
constexpr SortSizes kStaticSizes = sort_sizes(kStaticKeys, 1);
constexpr size_t kStaticBytes =
    sizeof(WsHeader) + round256(3 * 4) + 2 * (4 * round256((kStaticSizes.big + 1) * 4) + round256(kStaticSizes.big * 8)) +
    round256(kStaticSizes.parts * 8) + round256(kStaticSizes.parts * 4) + round256(kStaticSizes.parts * 4 * kPosStride) +
    2 * round256(kStaticSizes.small * 8) + round256(static_cast<size_t>(kStaticKeys) * 2) +
    round256(kStaticSizes.tiles * 4) + round256(static_cast<size_t>(kStaticKeys) * 8) +
    round256(static_cast<size_t>(kStaticKeys) * 4);

__device__ __align__(256) unsigned char g_sort_scratch[kStaticBytes];

std::mutex g_static_mutex;
constexpr int kMaxDevices = 64;
void* g_static_scratch[kMaxDevices] = {};

// Device address of g_sort_scratch on the current device, looked up once per device. In host code
// the array's name is only a host-side stand-in, never a device address. The cache is not
// invalidated by cudaDeviceReset. A stream of another device than the current one is rejected.
int static_sort_scratch(void** out, cudaStream_t st) {
    int dev = 0;
    CST_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices)
        return fail(CSTONE_ERR_INVALID_ARG, "cstone_sort_static: device ordinal %d not supported", dev);
    if (st != nullptr && st != cudaStreamLegacy && st != cudaStreamPerThread) {
        int sdev = -1;
        CST_CUDA(cudaStreamGetDevice(st, &sdev));
        if (sdev != dev)
            return fail(CSTONE_ERR_INVALID_ARG, "cstone_sort_static: stream of device %d, current device %d", sdev,
                        dev);
    }
    std::lock_guard<std::mutex> lock(g_static_mutex);
    if (g_static_scratch[dev] == nullptr) {
        void* p = nullptr;
        const cudaError_t e = cudaGetSymbolAddress(&p, g_sort_scratch);
        if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(g_sort_scratch)");
        g_static_scratch[dev] = p;
    }
    *out = g_static_scratch[dev];
    return CSTONE_OK;
}
}  // namespace
#endif


}  // namespace CST_NS

extern "C" {

int CSTONE_FN(sort_workspace_size)(int64_t n, size_t* bytes) {
    if (!bytes || n < 0 || n >= CSTONE_MAX_PARTICLES)
        return cst::fail(CSTONE_ERR_INVALID_ARG, CST_STR(CSTONE_FN(sort_workspace_size)) ": bad argument (n=%lld)",
                         (long long)n);
    *bytes = CST_NS::sort_ws_bytes(n);
    return CSTONE_OK;
}

int CSTONE_FN(sort)(const CST_KEY_C* keys_in, CST_KEY_C* keys_out, uint32_t* perm, int64_t n, void* ws,
                    size_t ws_bytes, void* stream) {
    if (n < 0 || n >= CSTONE_MAX_PARTICLES || (n > 0 && (!keys_in || !keys_out || !perm)))
        return cst::fail(CSTONE_ERR_INVALID_ARG, CST_STR(CSTONE_FN(sort)) ": bad argument (n=%lld)", (long long)n);
    if (int rc = cst::check_ws(ws, ws_bytes, CST_NS::sort_ws_bytes(n), CST_STR(CSTONE_FN(sort)))) return rc;
    return CST_NS::run_sort(reinterpret_cast<const CST_NS::Key*>(keys_in), reinterpret_cast<CST_NS::Key*>(keys_out),
                            perm, n, nullptr, 1, ws, cst::as_stream(stream));
}

#ifndef CSTONE_KEY32
int cstone_sort_static(const uint64_t* keys_in, uint64_t* keys_out, uint32_t* perm, int64_t n, void* stream) {
    if (n < 0 || (n > 0 && (!keys_in || !keys_out || !perm)))
        return cst::fail(CSTONE_ERR_INVALID_ARG, "cstone_sort_static: bad argument (n=%lld)", (long long)n);
    if (n > CSTONE_SORT_STATIC_MAX_KEYS)
        return cst::fail(CSTONE_ERR_INVALID_ARG,
                         "cstone_sort_static: n=%lld exceeds the static scratch limit of %lld keys; use cstone_sort "
                         "with a workspace",
                         (long long)n, (long long)CSTONE_SORT_STATIC_MAX_KEYS);
    if (cst::sort_ws_bytes(n) > cst::kStaticBytes)
        return cst::fail(CSTONE_ERR_INVALID_ARG, "cstone_sort_static: static scratch too small");
    void* ws = nullptr;
    if (int rc = cst::static_sort_scratch(&ws, cst::as_stream(stream))) return rc;
    return cst::run_sort(reinterpret_cast<const cst::u64*>(keys_in), reinterpret_cast<cst::u64*>(keys_out), perm, n,
                         nullptr, 1, ws, cst::as_stream(stream));
}

int cstone_sort_segmented_workspace_size(int64_t n, int32_t n_segs, size_t* bytes) {
    if (!bytes || n < 0 || n >= CSTONE_MAX_PARTICLES || n_segs < 1 || n_segs > (1 << 20))
        return cst::fail(CSTONE_ERR_INVALID_ARG, "cstone_sort_segmented_workspace_size: bad argument");
    *bytes = cst::sort_segmented_ws_bytes(n, n_segs);
    return CSTONE_OK;
}

int cstone_sort_segmented(const uint64_t* keys_in, uint64_t* keys_out, uint32_t* perm, int64_t n,
                          const int64_t* seg_offsets, int32_t n_segs, void* ws, size_t ws_bytes, void* stream) {
    if (n < 0 || n >= CSTONE_MAX_PARTICLES || n_segs < 1 || n_segs > (1 << 20) || !seg_offsets ||
        (n > 0 && (!keys_in || !keys_out || !perm)))
        return cst::fail(CSTONE_ERR_INVALID_ARG, "cstone_sort_segmented: bad argument (n=%lld, segments=%d)",
                         (long long)n, n_segs);
    if (keys_in == keys_out && n > 0)
        return cst::fail(CSTONE_ERR_INVALID_ARG, "cstone_sort_segmented: keys_in must not alias keys_out");
    if (int rc = cst::check_ws(ws, ws_bytes, cst::sort_segmented_ws_bytes(n, n_segs), "cstone_sort_segmented"))
        return rc;
    return cst::run_sort(reinterpret_cast<const cst::u64*>(keys_in), reinterpret_cast<cst::u64*>(keys_out), perm, n,
                         reinterpret_cast<const long long*>(seg_offsets), n_segs, ws, cst::as_stream(stream));
}

#endif

}  // extern "C"
