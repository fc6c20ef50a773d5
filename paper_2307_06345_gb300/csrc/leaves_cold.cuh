// The cornerstone leaf array built from the root in one sweep over the sorted keys, for the cold
// start of the leaf loop (leaves.cu, which includes this file). The f / g iteration of Sec. 4 from the
// root ends in the one array whose leaves hold at most N_crit particles (or are single keys) and
// whose internal nodes hold more; this finds that array directly.
//
// With P sorted, a level-l node with more than N_crit particles, the first of them at a, holds the
// particles a .. a + N_crit, so their keys share l digits; and a window of N_crit + 1 particles whose
// keys share l digits lies in one level-l node. With
//   c_i = digits shared by P[i] and P[i + N_crit] (at most L - 1; -1 where the window leaves the set)
//   d_j = digits shared by P[j - 1] and P[j]      (-1 at the first particle of a set)
//   s_j = max of c_i over i in [j - N_crit, j]: the deepest internal level that holds particle j
// the internal nodes that start at j are those of the levels d_j < l <= c_j, and j is the first
// particle of its leaf, at level s_j + 1, where d_j <= s_j. The leaves without particles between
// P[j - 1] and such a j are the later siblings on the way up from the leaf of j - 1 (of level
// s_{j-1} + 1) to the level d_j + 1, those between the two keys there, and the earlier siblings on the
// way down to the leaf of j; so j emits them and its leaf, and one scan over the particles places
// every leaf. A last emission after the last particle closes the array with its end key; in batched
// builds the first particle of a set closes the set before it, with the empty sets between.
//
// One launch reads P and lists the leaf starts (5 % of the particles at N_crit 64), a block scans the
// tiles' totals, one launch emits the leaves and one takes their counts; the loop makes two sweeps over its
// elements and a search of the split ranges per level, which is less where the leaves are few (sweep_taken in
// leaves.cu says where). The window maximum takes log2(N_crit) steps on bytes in shared memory, which holds
// windows of up to kMaxNcrit.
#pragma once

#include "common.cuh"

namespace CST_NS {
namespace {
namespace cold {

constexpr int kThreads = 256, kWarps = kThreads / 32;
constexpr int kItems = 8;
constexpr u32 kTile = kThreads * kItems;  // positions per tile: the particles, and one after the last
constexpr u32 kMaxNcrit = 1024;
constexpr int kBlocks = 6;  // blocks per SM of the sweep
constexpr u32 kDisorder = 0x70001u;  // error detail: keys that are not sorted
static_assert(kTile == 2048 && kLevels < 32, "bits of a listed leaf start");

struct View {  // the sets' particles; offsets == NULL: one set of n
    const long long* offsets;
    int n_sets;
    u32 n;
};

struct Tiles {
    u32* starts;    // [start_cap] leaf starts: position in the tile | level << 11 | level of the previous
                    // particle's leaf << 16 | first of a set or end << 21
    u32 start_cap;  // the capacity of the leaf array, which has room for no more
    u32* n_starts;  // [1] listed so far
    u32* list;      // [tiles] first entry of the tile
    u32* count;     // [tiles] entries of the tile
    u32* elems;     // [tiles] elements of the tile, then the index of the first
    int* levels;    // [kLevels + 2] internal nodes per level, as differences to the level above
    u32 tiles;
};

__host__ __device__ inline u32 tiles_of(long long n) { return static_cast<u32>((n + 1 + kTile - 1) / kTile); }

__device__ __forceinline__ u32 first_of(const View& v) { return v.offsets ? static_cast<u32>(__ldg(v.offsets)) : 0u; }
__device__ __forceinline__ u32 end_of(const View& v) {
    return v.offsets ? min(v.n, static_cast<u32>(__ldg(v.offsets + v.n_sets))) : v.n;
}

__device__ __forceinline__ int shared_digits(Key a, Key b) {  // of two keys, 0 .. kLevels
    const Key x = a ^ b;
    return x ? (key_clz(x) - (kWordBits - kKeyBits)) / 3 : kLevels;
}

// Sum of the octal digits of levels a .. b (from 1; none if a > b) of key.
__device__ __forceinline__ u32 digit_sum(Key key, int a, int b) {
    if (a > b) return 0u;
    const u64 k = (static_cast<u64>(key) >> (3 * (kLevels - b))) & ((1ULL << (3 * (b - a + 1))) - 1ULL);
    constexpr u64 kOnes = 0x1249249249249249ULL;
    return __popcll(k & kOnes) + 2u * __popcll(k & (kOnes << 1)) + 4u * __popcll(k & (kOnes << 2));
}

__device__ __forceinline__ u32 digit_at(Key key, int level) {
    return static_cast<u32>(key >> (3 * (kLevels - level))) & 7u;
}
__device__ __forceinline__ Key prefix(Key key, int level) {
    const int sh = 3 * (kLevels - level);
    return (key >> sh) << sh;
}

// Last set in [lo, hi] that starts at or before particle j (past empty sets).
__device__ __forceinline__ int set_of(const View& v, int lo, int hi, u32 j) {
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (static_cast<u32>(__ldg(v.offsets + mid)) <= j)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// Sets that end, or are empty, between the previous particle's set and position j (first: the first
// particle of any set): {sets before the one of j, of the previous particle or -1}.
__device__ __forceinline__ int2 sets_at(const View& v, u32 j, u32 first, u32 end) {
    if (!v.offsets) return make_int2(j == end ? 1 : 0, j > first ? 0 : -1);
    return make_int2(j == end ? v.n_sets : set_of(v, 0, v.n_sets - 1, j),
                     j > first ? set_of(v, 0, v.n_sets - 1, j - 1) : -1);
}

// Elements that position j emits: inside a set (d >= 0), the leaves without particles since the
// previous particle and the leaf of j; at a set's first particle or the end, the rest of the previous
// set with its end key, two elements per empty set, the way down to the first leaf and that leaf.
__device__ __forceinline__ u32 elements_between(Key prev, Key key, int d, int prev_level, int level) {
    const u32 up = prev_level > d + 1 ? 7u * (prev_level - d - 1) - digit_sum(prev, d + 2, prev_level) : 0u;
    return up + digit_at(key, d + 1) - digit_at(prev, d + 1) + digit_sum(key, d + 2, level);
}
__device__ __forceinline__ u32 elements_at_boundary(const View& v, u32 j, u32 first, u32 end, Key prev, Key key,
                                                    int prev_level, int level) {
    const int2 sets = sets_at(v, j, first, end);
    u32 cnt = 2u * (sets.x - sets.y - 1);
    if (j > first) cnt += 7u * prev_level - digit_sum(prev, 1, prev_level) + 1u;
    if (j < end) cnt += digit_sum(key, 1, level) + 1u;
    return cnt;
}

__device__ __forceinline__ u32 max_u8x4(u32 a, u32 b) {  // bytes below 128
    const u32 ge = (((a | 0x80808080u) - b) & 0x80808080u) >> 7;
    const u32 m = ge * 0xffu;
    return (a & m) | (b & ~m);
}

// Exclusive scan over the block (s: one word per warp), total in all.
__device__ __forceinline__ u32 scan_block(u32 v, u32* s, u32& all) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    u32 incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const u32 t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) s[warp] = incl;
    __syncthreads();
    u32 before = 0;
    all = 0;
    for (int w = 0; w < static_cast<int>(blockDim.x >> 5); ++w) {
        if (w < warp) before += s[w];
        all += s[w];
    }
    __syncthreads();
    return before + incl - v;
}

__host__ __device__ inline u32 halo_of(u32 ncrit) { return (ncrit + 4u) & ~3u; }  // > ncrit, a multiple of 4
inline size_t sweep_smem(u32 ncrit) {
    const size_t h = halo_of(ncrit);
    return (kTile + 2 * h) * sizeof(Key) + kTile * sizeof(u32) + 2 * (kTile + h);
}

// Window and neighbour values are kept as numbers of shared key bits, so that the division into digits
// comes after the maximum: 0 where there is no window, else min(bits, 3 (L - 1) + 2) + 3, so that a
// third of it (rounded down) is the level of the leaf.
__device__ __forceinline__ u32 shared_bits(Key a, Key b) { return key_clz(a ^ b) - (kWordBits - kKeyBits); }
__device__ __forceinline__ int third(u32 v) { return static_cast<int>((v * 171u) >> 9); }  // v < 256
constexpr u32 kMostBits = kKeyBits - 1;

// The sweep: leaf starts and elements of every tile. Dynamic shared memory: the keys from halo before the
// tile to halo after it; the tile's leaf starts; two arrays of bytes for the window maximum, from halo
// before the tile to its end. Most tiles lie inside one set (`plain`) and skip every test on its
// borders; the elements are counted from the list, where a warp has work for all lanes (counting them
// where the starts are found, four particles to a thread, took 1.16 ms for 2^27 clumps, this takes 0.78).
template <bool BATCH>
__global__ void __launch_bounds__(kThreads, kBlocks) starts_kernel(const Key* __restrict__ P, View v, u32 ncrit, Tiles t,
                                                                   WsHeader* hdr) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_levels[kLevels + 2];
    __shared__ u32 s_count[kItems * kWarps];
    __shared__ u32 s_elems;
    __shared__ u32 s_list, s_listed;
    __shared__ int s_sets[2];
    const u32 tid = threadIdx.x;
    const int lane = tid & 31, warp = tid >> 5;
    const u32 halo = halo_of(ncrit), nkeys = kTile + 2u * halo, slots = kTile + halo, words = slots / 4u;
    Key* s_key = reinterpret_cast<Key*>(smem);
    u32* s_start = reinterpret_cast<u32*>(s_key + nkeys);
    u32* s_a = s_start + kTile;
    u32* s_b = s_a + words;
    const u32 p0 = first_of(v), p1 = end_of(v);
    if (tid < kLevels + 2) s_levels[tid] = 0;
    for (u32 tile = blockIdx.x; tile < t.tiles; tile += gridDim.x) {
        const u32 t0 = tile * kTile;
        const long long slot0 = static_cast<long long>(t0) - halo;  // particle of slot 0
        bool plain = slot0 > static_cast<long long>(p0) && t0 + kTile + halo < p1;
        if (tid == 0) s_elems = 0;
        if (BATCH) {  // the sets that the tile and its halos reach
            if (tid < 2) {
                const long long i = tid == 0 ? max(slot0, static_cast<long long>(p0))
                                             : min(static_cast<long long>(t0) + kTile + halo, static_cast<long long>(p1) - 1);
                s_sets[tid] = set_of(v, 0, v.n_sets - 1, i > 0 ? static_cast<u32>(i) : 0u);
            }
            __syncthreads();
            // the whole stretch in one set, and not from its first particle on
            plain = plain && s_sets[0] == s_sets[1] && static_cast<long long>(__ldg(v.offsets + s_sets[0])) < slot0;
        }
        unsigned char* bytes = reinterpret_cast<unsigned char*>(s_a);
        if (plain) {
            const Key* src = P + slot0;
            for (u32 q = tid; q < nkeys; q += kThreads) s_key[q] = __ldcg(src + q);
            __syncthreads();
            for (u32 q = tid; q < slots; q += kThreads)
                bytes[q] = static_cast<unsigned char>(min(shared_bits(s_key[q], s_key[q + ncrit]), kMostBits) + 3u);
        } else {
            auto inside = [&](long long i) { return i >= static_cast<long long>(p0) && i < static_cast<long long>(p1); };
            for (u32 q = tid; q < nkeys; q += kThreads)
                s_key[q] = inside(slot0 + q) ? __ldcg(P + (slot0 + q)) : static_cast<Key>(0);
            __syncthreads();
            for (u32 q = tid; q < slots; q += kThreads) {
                const long long i = slot0 + q;
                u32 bits = 0;
                if (inside(i)) {
                    u32 end = p1;
                    if (BATCH)
                        end = min(p1, static_cast<u32>(__ldg(v.offsets + 1 + set_of(v, s_sets[0], s_sets[1],
                                                                                    static_cast<u32>(i)))));
                    if (ncrit < end - static_cast<u32>(i))
                        bits = min(shared_bits(s_key[q], s_key[q + ncrit]), kMostBits) + 3u;
                }
                bytes[q] = static_cast<unsigned char>(bits);
            }
        }
        __syncthreads();
        // window maximum over [j - ncrit, j] by doubling: the maxima over `width` particles ending at j
        // with those ending `off` earlier. Slots before slot 0 count as zero, which only the halo sees.
        u32 *src = s_a, *dst = s_b;
        for (u32 width = 1; width < ncrit + 1u;) {
            const u32 off = min(width, ncrit + 1u - width), wo = off >> 2, bits = 8u * (off & 3u);
            for (u32 w = tid; w < words; w += kThreads) {
                const u32 hi = w >= wo ? src[w - wo] : 0u, lo = bits && w > wo ? src[w - wo - 1u] : 0u;
                dst[w] = max_u8x4(src[w], __funnelshift_l(lo, hi, bits));
            }
            __syncthreads();
            u32* const swap = src;
            src = dst;
            dst = swap;
            width += off;
        }
        const unsigned char* s_max = reinterpret_cast<const unsigned char*>(src);
        // the leaf starts, in order: 256 positions at a time, by warp and lane
        u32 starts = 0, boundaries = 0;  // bit per item
#pragma unroll
        for (int it = 0; it < kItems; ++it) {
            const u32 o = it * kThreads + tid, j = t0 + o, q = o + halo;
            bool on = false, boundary = false;
            if (plain) {
                on = third(s_max[q]) > third(shared_bits(s_key[q - 1], s_key[q]));
            } else if (j >= p0 && j <= p1) {
                boundary = j == p0 || j == p1;
                if (BATCH && !boundary)
                    boundary = static_cast<u32>(__ldg(v.offsets + set_of(v, s_sets[0], s_sets[1], j))) == j;
                on = boundary || third(s_max[q]) > third(shared_bits(s_key[q - 1], s_key[q]));
            }
            starts |= on ? 1u << it : 0u;
            boundaries |= boundary ? 1u << it : 0u;
            const u32 bal = __ballot_sync(0xffffffffu, on);
            if (lane == 0) s_count[it * kWarps + warp] = __popc(bal);
        }
        __syncthreads();
        if (warp == 0) {  // 64 counts to starts
            const u32 c0 = s_count[2 * lane], c1 = s_count[2 * lane + 1];
            u32 incl = c0 + c1;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const u32 x = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += x;
            }
            s_count[2 * lane] = incl - c0 - c1;
            s_count[2 * lane + 1] = incl - c1;
            if (lane == 31) {
                s_listed = incl;
                s_list = incl ? atomicAdd(t.n_starts, incl) : 0u;
            }
        }
        __syncthreads();
#pragma unroll
        for (int it = 0; it < kItems; ++it) {
            const bool on = (starts >> it) & 1u;
            const u32 bal = __ballot_sync(0xffffffffu, on);
            if (on) {
                const u32 o = it * kThreads + tid, q = o + halo;
                const bool end = t0 + o == p1, begin = t0 + o == p0;
                s_start[s_count[it * kWarps + warp] + __popc(bal & lanemask_lt())] =
                    o | (end ? 0u : static_cast<u32>(third(s_max[q])) << 11) |
                    (begin ? 0u : static_cast<u32>(third(s_max[q - 1])) << 16) | (((boundaries >> it) & 1u) << 21);
            }
        }
        __syncthreads();
        u32 elems = 0;
        for (u32 i = tid; i < s_listed; i += kThreads) {
            const u32 w = s_start[i], o = w & 0x7ffu, j = t0 + o, q = o + halo;
            const int level = static_cast<int>((w >> 11) & 31u), prev_level = static_cast<int>((w >> 16) & 31u);
            const Key key = s_key[q], prev = s_key[q - 1];
            const int d = (w >> 21) ? -1 : shared_digits(prev, key);
            if (d >= 0 && key < prev) raise_error(hdr, CSTONE_ERR_INVALID_ARG, kDisorder);
            elems += d < 0 ? elements_at_boundary(v, j, p0, p1, prev, key, prev_level, level)
                           : elements_between(prev, key, d, prev_level, level);
            if (j < p1 && level > d + 1) {  // internal nodes of levels d + 1 .. level - 1 start here
                atomicAdd(&s_levels[d + 1], 1);
                atomicSub(&s_levels[level], 1);
            }
            if (s_list < t.start_cap && i < t.start_cap - s_list) t.starts[s_list + i] = w;
        }
        for (int o = 16; o > 0; o >>= 1) elems += __shfl_xor_sync(0xffffffffu, elems, o);
        if (lane == 0 && elems) atomicAdd(&s_elems, elems);
        __syncthreads();
        if (tid == 0) {
            t.list[tile] = s_list;
            t.count[tile] = s_listed;
            t.elems[tile] = s_elems;
        }
        __syncthreads();  // the shared arrays are rewritten by the next tile
    }
    if (tid < kLevels + 2 && s_levels[tid] != 0) atomicAdd(&t.levels[tid], s_levels[tid]);
}
static_assert(kItems * kWarps == 64, "two counts per lane");

// Index of every tile's first element, and the outcome as the loop would have it: pass l splits the
// internal nodes of level l, the pass after the last of them changes nothing. One block.
//
// Self-check: keys that are not sorted (or set offsets that do not ascend) can list more starts than the array
// has elements, and so more than the list holds. Of a sorted set every start emits its leaf, and the starts
// together emit the array; anything else is an error, before the list is read.
__global__ void __launch_bounds__(1024) outcome_kernel(Tiles t, int n_sets, u32 ecap, int max_iters,
                                                       WsHeader* hdr) {
    __shared__ u32 s_warp[32];
    const u32 listed = *t.n_starts, err = hdr->err;  // loaded while the tiles are scanned
    u32 run = 0, all;
    constexpr u32 kPer = 4;
    for (u32 k0 = 0; k0 < t.tiles; k0 += 1024 * kPer) {
        u32 c[kPer], sum = 0;
#pragma unroll
        for (u32 q = 0; q < kPer; ++q) {
            const u32 k = k0 + threadIdx.x * kPer + q;
            c[q] = k < t.tiles ? t.elems[k] : 0u;
            sum += c[q];
        }
        u32 at = run + scan_block(sum, s_warp, all);
        run += all;
#pragma unroll
        for (u32 q = 0; q < kPer; ++q) {
            const u32 k = k0 + threadIdx.x * kPer + q;
            if (k < t.tiles) t.elems[k] = at;
            at += c[q];
        }
    }
    if (threadIdx.x != 0) return;
    u64 ne = 2ull * n_sets;
    long long nodes = 0;
    for (int pass = 0; pass < max_iters; ++pass) {
        nodes += pass < kLevels ? t.levels[pass] : -nodes;  // of level `pass`
        if (nodes == 0) {
            if (err) return;
            if (listed > ne || run != static_cast<u32>(ne)) {
                raise_error(hdr, CSTONE_ERR_INVALID_ARG, kDisorder);
                return;
            }
            *outcome_of(hdr) = Outcome{static_cast<u32>(pass + 1), 1u, 0u, static_cast<u32>(ne)};
            return;
        }
        ne += 7ull * static_cast<u64>(nodes);
        if (ne > ecap) {
            outcome_of(hdr)->required = static_cast<u32>(ne > 0xffffffffULL ? 0xffffffffULL : ne);
            raise_error(hdr, CSTONE_ERR_CAPACITY, 0u);
            return;
        }
    }
    outcome_of(hdr)->iters = static_cast<u32>(max_iters);
}

// The leaves (and end keys) that the listed positions emit, with their first particles.
template <bool BATCH>
__global__ void __launch_bounds__(kThreads) emit_kernel(const Key* __restrict__ P, View v, Tiles t, u32 ecap,
                                                        WsHeader* hdr, Key* __restrict__ elements,
                                                        u32* __restrict__ first_particle, long long* element_offsets) {
    __shared__ u32 s_warp[kWarps];
    if (outcome_of(hdr)->converged == 0u) return;
    const u32 p0 = first_of(v), p1 = end_of(v);
    for (u32 tile = blockIdx.x; tile < t.tiles; tile += gridDim.x) {
        const u32 list = t.list[tile], count = t.count[tile];
        u32 base = t.elems[tile];
        for (u32 i0 = 0; i0 < count; i0 += kThreads) {
            const u32 i = i0 + threadIdx.x;
            u32 cnt = 0, j = 0, all;
            int level = 0, prev_level = 0, d = -1;
            bool boundary = false;
            Key key = 0, prev = 0;
            if (i < count) {
                const u32 w = t.starts[list + i];
                j = tile * kTile + (w & 0x7ffu);
                level = static_cast<int>((w >> 11) & 31u);
                prev_level = static_cast<int>((w >> 16) & 31u);
                boundary = (w >> 21) != 0u;
                if (j < p1) key = __ldg(P + j);
                if (j > p0) prev = __ldg(P + j - 1);
                if (!boundary) d = shared_digits(prev, key);
                cnt = boundary ? elements_at_boundary(v, j, p0, p1, prev, key, prev_level, level)
                               : elements_between(prev, key, d, prev_level, level);
            }
            u32 at = base + scan_block(cnt, s_warp, all);
            base += all;
            if (i < count) {
                auto put = [&](Key k) {
                    if (at < ecap) {
                        elements[at] = k;
                        first_particle[at] = j;
                    }
                    ++at;
                };
                // siblings after the branch of the previous particle, from its leaf up
                const int up_to = boundary ? 1 : d + 2;
                if (j > p0)
                    for (int l = prev_level; l >= up_to; --l)
                        for (u32 q = digit_at(prev, l) + 1u; q < 8u; ++q)
                            put(prefix(prev, l - 1) + (static_cast<Key>(q) << (3 * (kLevels - l))));
                if (boundary) {
                    const int2 sets = sets_at(v, j, p0, p1);
                    if (j > p0) put(kKeyEnd);
                    for (int s = sets.y + 1; s < sets.x; ++s) {
                        if (BATCH) element_offsets[s] = at;
                        put(0);
                        put(kKeyEnd);
                    }
                    if (BATCH) element_offsets[sets.x] = at;  // of the set of j, or the total
                } else {
                    for (u32 q = digit_at(prev, d + 1) + 1u; q < digit_at(key, d + 1); ++q)
                        put(prefix(key, d) + (static_cast<Key>(q) << (3 * (kLevels - d - 1))));
                }
                if (j < p1) {
                    for (int l = boundary ? 1 : d + 2; l <= level; ++l)  // siblings before the branch of j
                        for (u32 q = 0; q < digit_at(key, l); ++q)
                            put(prefix(key, l - 1) + (static_cast<Key>(q) << (3 * (kLevels - l))));
                    put(prefix(key, level));
                }
            }
        }
    }
}

// Leaf counts from the first particles; with BATCH, zero at the end keys. After a failed build without
// a host to report to, every set's root array instead (as the loop leaves it).
template <bool BATCH>
__global__ void __launch_bounds__(kThreads) counts_kernel(const Key* __restrict__ P, View v, int fallback,
                                                          WsHeader* hdr, Key* elements, u32* __restrict__ counts,
                                                          const u32* first_particle, u32* out_offsets,
                                                          long long* element_offsets) {
    const u32 gtid = blockIdx.x * kThreads + threadIdx.x, gthreads = gridDim.x * kThreads;
    if (outcome_of(hdr)->converged == 0u) {
        if (fallback)
            write_root_arrays<BATCH>(P, v.n, SetView{v.offsets, element_offsets, v.n_sets}, gtid, gthreads, elements, counts,
                                     out_offsets);
        return;
    }
    const u32 ne = outcome_of(hdr)->ne;
    for (u32 e = gtid; e + 1u < ne; e += gthreads) {
        const u32 c = first_particle[e + 1] - first_particle[e];
        counts[e] = BATCH && elements[e] == kKeyEnd ? 0u : c;
    }
    if (BATCH && gtid == 0) counts[ne - 1u] = 0u;
}

}  // namespace cold
}  // namespace
}  // namespace CST_NS
