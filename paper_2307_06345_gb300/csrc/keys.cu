// Bounding cube and space-filling-curve keys (Sec. 3).
//
// Keys are streaming work: 24 bytes of coordinates in, 8 bytes of key out per particle. The
// kernel reads the three coordinate arrays with 16-byte vector loads (two particles per thread
// per step), computes the grid cell with the result of IEEE double precision with explicitly
// rounded operations (an integer fixed-point evaluation where its error bound proves the same
// cell; no FMA contraction, so the cell matches any IEEE host bit for bit) and encodes it. With
// masses, a second kernel also writes each particle's multipole record from the same read.
//
// Hilbert encoding uses a finite-state machine equivalent to J. Skilling's transpose formulation
// of the Hilbert curve: walking the bit levels from the top, Skilling's per-level inversions and
// exchanges act on all lower bits as a signed permutation of the axes, and the final Gray-code
// flip of a level is the parity of the Gray-coded third axis above it. Tracking (permutation,
// flips, parity) as a state gives 48 reachable states. The host builds the one-level table
// (state, octant) -> (digit, next state) once and passes it to the kernels as a by-value
// parameter (no device memory or symbol upload); each block composes it into a table of several levels
// in shared memory: three from 2^22 particles on, so that a 21-level key takes 7 lookups, and two below
// (11 lookups), where composing the larger table would take longer than the keys.
#include <mutex>

#include <cooperative_groups.h>

#include "common.cuh"
#include "records.cuh"

namespace cg = cooperative_groups;

namespace CST_NS {

// ---------------------------------------------------------------------------------- bounding cube
namespace {

// A double as a signed 64-bit integer of the same order: the magnitude bits of a negative value
// are flipped, so that a more negative double is a smaller integer (the sign bit is kept, which
// makes the map its own inverse). Minima and maxima then take integer min / max: on this part the
// FP64 min / max and the unsigned 64-bit compare-and-select both cost more than the HBM stream.
__device__ __forceinline__ long long ordered_bits(double v) {
    const long long b = __double_as_longlong(v);
    return b ^ static_cast<long long>(static_cast<u64>(b >> 63) >> 1);
}

__device__ __forceinline__ double from_ordered(long long o) {
    return __longlong_as_double(o ^ static_cast<long long>(static_cast<u64>(o >> 63) >> 1));
}

constexpr long long kOrderedMax = 0x7fffffffffffffffLL;
constexpr long long kOrderedMin = -kOrderedMax - 1;

struct BoxAcc {
    long long lo[3];  // ordered bits of the per-axis minimum
    long long hi[3];  // ordered bits of the per-axis maximum
};

__global__ void bbox_init_kernel(BoxAcc* acc) {
    int t = threadIdx.x;
    if (t < 3) {
        acc->lo[t] = kOrderedMax;
        acc->hi[t] = kOrderedMin;
    }
}

__global__ void __launch_bounds__(256) bbox_reduce_kernel(const double* __restrict__ x, const double* __restrict__ y,
                                                          const double* __restrict__ z, long long n, BoxAcc* acc) {
    long long lo[3] = {kOrderedMax, kOrderedMax, kOrderedMax}, hi[3] = {kOrderedMin, kOrderedMin, kOrderedMin};
    const double* c[3] = {x, y, z};
    auto take = [&](int d, double v) {
        const long long o = ordered_bits(v);
        lo[d] = min(lo[d], o);
        hi[d] = max(hi[d], o);
    };
    const bool vec = ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(y) | reinterpret_cast<uintptr_t>(z)) &
                      15u) == 0;
    const long long stride = (long long)gridDim.x * blockDim.x;
    long long done = 0;
    if (vec) {  // two 16-byte loads per array and thread per step: 6 loads in flight
        const long long quads = n >> 2;
        for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < quads; q += stride) {
            double2 v[3][2];
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const double2* p = reinterpret_cast<const double2*>(c[d]) + 2 * q;
                v[d][0] = __ldcg(p);
                v[d][1] = __ldcg(p + 1);
            }
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                take(d, v[d][0].x);
                take(d, v[d][0].y);
                take(d, v[d][1].x);
                take(d, v[d][1].y);
            }
        }
        done = quads << 2;
    }
    for (long long i = done + blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += stride) {
#pragma unroll
        for (int d = 0; d < 3; ++d) take(d, __ldg(c[d] + i));
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        for (int s = 16; s > 0; s >>= 1) {
            lo[d] = min(lo[d], __shfl_xor_sync(0xffffffffu, lo[d], s));
            hi[d] = max(hi[d], __shfl_xor_sync(0xffffffffu, hi[d], s));
        }
    }
    // the block's warps through shared memory, then one update of the global bounds per block
    // (all blocks update the same six words)
    __shared__ long long s_lo[8][3], s_hi[8][3];
    const int warp = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0)
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            s_lo[warp][d] = lo[d];
            s_hi[warp][d] = hi[d];
        }
    __syncthreads();
    if (threadIdx.x < 3) {
        const int d = threadIdx.x;
        long long l = s_lo[0][d], h = s_hi[0][d];
        for (int w = 1; w < static_cast<int>(blockDim.x >> 5); ++w) {
            l = min(l, s_lo[w][d]);
            h = max(h, s_hi[w][d]);
        }
        atomicMin(&acc->lo[d], l);
        atomicMax(&acc->hi[d], h);
    }
}

// Per-axis minima and maxima {min x, min y, min z, max x, max y, max z}; with no points the
// minima are +inf and the maxima -inf, so that a reduction over several sets ignores an empty one.
__global__ void bounds_finalize_kernel(const BoxAcc* acc, long long n, double* bounds) {
    if (threadIdx.x >= 3) return;
    const int d = threadIdx.x;
    bounds[d] = n > 0 ? from_ordered(acc->lo[d]) : __longlong_as_double(0x7ff0000000000000LL);
    bounds[3 + d] = n > 0 ? from_ordered(acc->hi[d]) : __longlong_as_double(static_cast<long long>(0xfff0000000000000ULL));
}

__global__ void bbox_finalize_kernel(const BoxAcc* acc, long long n, double* box) {
    if (threadIdx.x != 0) return;
    if (n == 0) {
        box[0] = box[1] = box[2] = 0.0;
        box[3] = 1.0;
        return;
    }
    double side = 0.0;
    for (int d = 0; d < 3; ++d) {
        double lo = from_ordered(acc->lo[d]);
        double hi = from_ordered(acc->hi[d]);
        box[d] = lo;
        double ext = __dsub_rn(hi, lo);
        side = ext > side ? ext : side;
    }
    box[3] = side > 0.0 ? side : 1.0;
}

// ---------------------------------------------------------------------------------- grid + keys
struct HilbertTable {
    unsigned short one[kHilbertStates * 8];  // (state, 1 octant) -> 3 digit bits | next << 3
};

// Cell index of one coordinate: floor((x - lo) * scale) clamped to [0, 2^21 - 1], with the
// subtraction and the product rounded once each (explicit round-to-nearest intrinsics keep the
// compiler from fusing them into an FMA).
__device__ __forceinline__ u32 grid_cell(double x, double lo, double scale) {
    double u = __dmul_rn(__dsub_rn(x, lo), scale);
    if (!(u > 0.0)) return 0u;
    if (u >= 2097152.0) return 2097151u;
    return __double2uint_rz(u);
}

// Integer evaluation of grid_cell. Double-precision throughput is a small fraction of the integer
// throughput on this GPU, so the cell is first computed in 64-bit fixed point:
//   X = trunc(x * 2^F), LO = trunc(lo * 2^F), u * 2^R ~= ((X - LO) * S) >> 64, S = scale * 2^G,
// with F chosen so |X| < 2^61 on [lo, lo + 2 side) and S holding scale's 53-bit mantissa at the
// top of 64 bits. The truncations, the product and the two IEEE roundings of the reference
// together move u by far less than 2^-24 cells, so whenever the fixed-point u is at least 2^-20
// away from an integer its floor is the floor of the IEEE result. The remaining ~2^-19 of
// coordinates, and boxes where the error bound does not hold, take the IEEE path.
struct FixedGrid {  // one axis
    long long lo_fixed;   // LO
    u64 scale_fixed;      // S
    u64 lo_ord, hi_ord;   // order-preserving bits of lo and of lo + 2 side
    double lo, scale;
    int F, R;
    int ok;               // the values allow a bound (whether it holds depends on F)
    int fast;             // the bound holds at this F
};

__device__ __forceinline__ u64 order_bits(double v) {
    const u64 b = static_cast<u64>(__double_as_longlong(v));
    return (b >> 63) ? ~b : (b | (1ULL << 63));
}

__device__ __forceinline__ int exponent_of(double v) {  // unbiased exponent field (0 for zero/subnormal)
    return static_cast<int>((static_cast<u64>(__double_as_longlong(v)) >> 52) & 0x7ffu);
}

// trunc(x * 2^F) for |x| * 2^F < 2^62
__device__ __forceinline__ long long to_fixed(double x, int F) {
    u64 b = static_cast<u64>(__double_as_longlong(x));
    int e = static_cast<int>((b >> 52) & 0x7ffu);
    u64 mant = b & ((1ULL << 52) - 1);
    if (e != 0) mant |= (1ULL << 52);
    int sh = (e == 0 ? 1 : e) - 1075 + F;
    u64 mag = sh >= 0 ? (mant << sh) : (sh > -64 ? (mant >> (-sh)) : 0ULL);
    return (b >> 63) ? -static_cast<long long>(mag) : static_cast<long long>(mag);
}

__device__ __forceinline__ bool bound_holds(int F, int R) {
    const int es = F - R - 53;  // scale = mantissa * 2^es
    return R >= 26 && R <= 62 && es + 78 <= F && F <= 1074;
}

// The axis in the widest frame that holds it.
__device__ FixedGrid make_fixed_grid(double lo, double side) {
    FixedGrid f;
    f.lo = lo;
    f.scale = __ddiv_rn(2097152.0, side);
    const double hi = __dadd_rn(lo, __dmul_rn(2.0, side));
    f.lo_ord = order_bits(lo);
    f.hi_ord = order_bits(hi);
    // 2^E > max(|lo|, |hi|)
    const int e_max = max(exponent_of(lo), exponent_of(hi)) - 1023 + 1;
    f.F = 61 - e_max;
    const int es = exponent_of(f.scale) - 1023 - 52;
    const int G = 11 - es;
    f.R = f.F + G - 64;
    u64 sb = static_cast<u64>(__double_as_longlong(f.scale));
    f.scale_fixed = ((sb & ((1ULL << 52) - 1)) | (1ULL << 52)) << 11;
    f.ok = exponent_of(f.scale) != 0 && exponent_of(f.scale) != 0x7ff && e_max < 1024 && !(hi <= lo);
    f.fast = f.ok && bound_holds(f.F, f.R);
    f.lo_fixed = f.fast ? to_fixed(lo, f.F) : 0;
    return f;
}

// The same evaluation in the form the kernels run. The kernels are bound by the integer pipe, which
// takes two cycles for a warp's instruction, so: the three axes share one frame (the box's), so that
// scale, shift and limits are the same; a coordinate is brought to fixed point by one right shift of
// its mantissa; the product's high word is the cell and its low word the fraction; and whatever is not
// plainly inside the box and away from cell borders, on any axis, takes one rare path. 2^25 Plummer
// particles, Hilbert keys: 421 us with a frame, limits and selections per axis, 291 now (the integer
// pipe 77 % busy); 7.7e7 Morton keys of 512 sets 1610 -> 731 us.
struct FastGrid {
    u64 neg_lo[3];  // -trunc(lo * 2^F)
    u64 scale;      // S such that (((X - LO) << d_shift) * S) >> 64 has 32 fraction bits
    u32 e_end;      // exponents below this are in the frame: |X| is the mantissa at bit 61 shifted right by e_end - e
    u32 d_end;      // distances from the corner whose high word is below this are inside the box
    int d_shift;
    int fast;       // the error bound holds
    FixedGrid axis[3];  // for the rare path
};

// The frame that holds all axes, which is the records' frame (make_frame). Called by whole warps: lane d of a
// group of four takes axis d (the fourth repeats the last), and the group writes *g where `write` is set. One
// thread with the axes one after the other took 2 us longer, of the 8 that the keys of 1000 particles take.
__device__ __forceinline__ void make_fast_grid(const double* box, FastGrid* g, bool write) {
    const u32 d = min(threadIdx.x & 3u, 2u);
    const double side = box[3];
    const FixedGrid f = make_fixed_grid(box[d], side);
    int F = f.F, ok = f.ok;
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) {
        F = min(F, __shfl_xor_sync(0xffffffffu, F, o));
        ok &= __shfl_xor_sync(0xffffffffu, ok, o);
    }
    const int R = F + f.R - f.F;
    const int fast = ok && bound_holds(F, R) && F <= 900;  // so that subnormal coordinates are zero in fixed point
    if (!write || (threadIdx.x & 3u) == 3u) return;
    g->axis[d] = f;
    g->neg_lo[d] = fast ? 0ULL - static_cast<u64>(to_fixed(f.lo, F)) : 0ULL;
    if (d != 0) return;
    g->scale = R >= 32 ? f.scale_fixed >> (R - 32) : f.scale_fixed;
    g->d_shift = R >= 32 ? 0 : 32 - R;
    g->e_end = static_cast<u32>(9 + 1075 - F);
    g->d_end = fast ? static_cast<u32>(static_cast<u64>(to_fixed(side, F)) >> 32) : 0u;
    g->fast = fast;
}

// X = trunc(x * 2^F) and its distance d from the box's corner; returns the exponent field.
__device__ __forceinline__ u32 to_frame(double x, u64 neg_lo, u32 e_end, u64& X, u64& d) {
    const u32 hi = static_cast<u32>(__double2hiint(x)), lo = static_cast<u32>(__double2loint(x));
    const u32 e = (hi >> 20) & 0x7ffu;
    const u64 m = ((static_cast<u64>((hi & 0xfffffu) | 0x100000u) << 32) | lo) << 9;
    const u64 mag = m >> min(e_end - e, 63u);
    const u32 neg = hi >> 31;
    const u64 flip = static_cast<u64>(static_cast<long long>(static_cast<int>(hi) >> 31));
    X = (mag ^ flip) + neg;
    d = (mag ^ flip) + neg_lo + neg;
    return e;
}

// (a * b) >> 64 without the product of the low words: at most 2 too small.
__device__ __forceinline__ u64 mul_high(u64 a, u64 b) {
    const u32 al = static_cast<u32>(a), ah = static_cast<u32>(a >> 32), bl = static_cast<u32>(b), bh = static_cast<u32>(b >> 32);
    return static_cast<u64>(ah) * bh + ((static_cast<u64>(al) * bh) >> 32) + __umulhi(ah, bl);
}

// Cell of one coordinate on the rare path, d its axis: in the shared frame once more, since mostly another axis of
// the particle led here; beyond the box by the order of the bits; where another axis of the box lies too far out
// for the shared frame (10^6 sides from the origin), in the axis' own; at the borders of cells and where no bound
// holds by IEEE arithmetic (inside the box without grid_cell's comparisons, which run at the FP64 rate too).
// 2^25 Morton keys with IEEE arithmetic on all three axes, and so: one axis of the box far out 957 -> 479 us, every
// tenth particle outside the box 939 -> 463, all on the borders of cells 960 -> 784.
__device__ __forceinline__ u32 cell_exact(double x, const FastGrid& g, int d) {
    const FixedGrid& f = g.axis[d];
    if (g.fast) {
        u64 X, dist;
        const u32 e = to_frame(x, g.neg_lo[d], g.e_end, X, dist);
        const u64 u = mul_high(dist << g.d_shift, g.scale);
        if (e < g.e_end && static_cast<u32>(dist >> 32) < g.d_end && static_cast<u32>(u) + 0x1000u >= 0x2000u)
            return static_cast<u32>(u >> 32);
    }
    if (!f.fast) return grid_cell(x, f.lo, f.scale);
    const u64 o = order_bits(x);
    if (o <= f.lo_ord) return 0u;
    if (o >= f.hi_ord) return 2097151u;
    if (!g.fast) {
        const u64 u = __umul64hi(static_cast<u64>(to_fixed(x, f.F) - f.lo_fixed), f.scale_fixed);
        const u32 frac20 = static_cast<u32>(u >> (f.R - 20)) & 0xfffffu;
        const u64 c = u >> f.R;
        if (frac20 != 0u && frac20 != 0xfffffu) return c > 2097151ULL ? 2097151u : static_cast<u32>(c);
    }
    return min(__double2uint_rz(__dmul_rn(__dsub_rn(x, f.lo), f.scale)), 2097151u);
}

// The three cells of a particle on the rare path, 21 bits each.
__device__ __noinline__ u64 cells_exact(double px, double py, double pz, const FastGrid& g) {
    return cell_exact(px, g, 0) | (static_cast<u64>(cell_exact(py, g, 1)) << 21) |
           (static_cast<u64>(cell_exact(pz, g, 2)) << 42);
}

// Cells of a particle; X gets its fixed-point coordinates where the grid is fast. Returns whether all
// coordinates are in the frame (always true where the grid is not fast).
__device__ __forceinline__ bool cells_of(const FastGrid& g, double px, double py, double pz, u32 c[3], u64 X[3]) {
    bool in = true, sure = false;
    if (g.fast) {
        u64 d[3];
        const u32 e = max(to_frame(px, g.neg_lo[0], g.e_end, X[0], d[0]),
                          max(to_frame(py, g.neg_lo[1], g.e_end, X[1], d[1]),
                              to_frame(pz, g.neg_lo[2], g.e_end, X[2], d[2])));
        u32 dh = 0, frac = 0xffffffffu;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            dh = max(dh, static_cast<u32>(d[k] >> 32));
            const u64 u = mul_high(d[k] << g.d_shift, g.scale);
            c[k] = static_cast<u32>(u >> 32);
            frac = min(frac, static_cast<u32>(u) + 0x1000u);
        }
        in = e < g.e_end;
        sure = in && dh < g.d_end && frac >= 0x2000u;  // 2^-20 cells or more from every border
    }
    if (!sure) {
        const u64 cells = cells_exact(px, py, pz, g);
        c[0] = static_cast<u32>(cells) & 0x1fffffu;
        c[1] = static_cast<u32>(cells >> 21) & 0x1fffffu;
        c[2] = static_cast<u32>(cells >> 42);
    }
    return in;
}

// Every third bit of a word: bit b of the low 10 bits to bit 3b, by the multiply-and-mask steps of T. Karras
// ("Thinking Parallel, Part III", 2012). The multiplications run beside the integer pipe.
__device__ __forceinline__ u32 spread10(u32 v) {
    v = (v * 0x00010001u) & 0xff0000ffu;
    v = (v * 0x00000101u) & 0x0f00f00fu;
    v = (v * 0x00000011u) & 0xc30c30c3u;
    return (v * 0x00000005u) & 0x49249249u;
}

__device__ __forceinline__ u64 morton_of(u32 gx, u32 gy, u32 gz) {
    const u32 low = spread10(gx & 0x3ffu) * 4u + spread10(gy & 0x3ffu) * 2u + spread10(gz & 0x3ffu);
    const u32 mid = spread10((gx >> 10) & 0x3ffu) * 4u + spread10((gy >> 10) & 0x3ffu) * 2u + spread10((gz >> 10) & 0x3ffu);
    const u32 top = ((gx >> 20) << 2) | ((gy >> 20) << 1) | (gz >> 20);
    return (static_cast<u64>(top) << 60) | (static_cast<u64>(mid) << 30) | low;
}

// Key of this build's length from a 63-bit key: the cell of a coarser grid is the top 3L bits of
// the 21-level key (octree prefix of both curves, and floor(cell_21 / 2^(21-L)) = cell_L exactly
// because the grid scales differ by a power of two).
__device__ __forceinline__ Key to_key(u64 k63) { return static_cast<Key>(k63 >> (63 - kKeyBits)); }

// The box's grid and the one-level Hilbert table in shared memory. Hilbert keys
// take several levels per lookup from a table that each block composes of the one-level table, indexed
// by the state and TL bits of each coordinate's cell (x bits above y bits above z bits): three levels
// (48 KB of dynamic shared memory, 7 lookups per key) where a block has many particles, two levels
// (6 KB, 11 lookups) for sets of fewer than kTwoLevelMax particles, where composing the large table took
// most of the time (2^20 particles: 56 -> 21 us).
struct KeySmem {
    unsigned short t1[kHilbertStates * 8];
    FastGrid grid;
};
constexpr long long kTwoLevelMax = 1ll << 22;
constexpr int kKeyThreads = 512, kKeyBlocks = 6;  // blocks per SM in the grid: two waves
template <int TL>
constexpr int kTableEntries = kHilbertStates << (3 * TL);
template <int TL>
constexpr size_t kTableBytes = kTableEntries<TL> * sizeof(unsigned short);

// Entry (state, bits): the digits of TL levels | next state << 3 TL.
template <int TL>
__device__ __forceinline__ void compose_table(KeySmem& sm, unsigned short* table, const HilbertTable& one) {
    for (int i = threadIdx.x; i < kHilbertStates * 8; i += blockDim.x) sm.t1[i] = one.one[i];
    __syncthreads();
    for (int e = threadIdx.x; e < kTableEntries<TL>; e += blockDim.x) {
        u32 state = static_cast<u32>(e >> (3 * TL)), digits = 0;
#pragma unroll
        for (int lv = TL - 1; lv >= 0; --lv) {
            const u32 o = (((e >> (2 * TL + lv)) & 1u) << 2) | (((e >> (TL + lv)) & 1u) << 1) | ((e >> lv) & 1u);
            const u32 v = sm.t1[state * 8u + o];
            digits = (digits << 3) | (v & 7u);
            state = v >> 3;
        }
        table[e] = static_cast<unsigned short>(digits | (state << (3 * TL)));
    }
}

// Key of a cell from the table: TL levels per step, as far as this build's keys reach.
template <int TL>
__device__ __forceinline__ Key hilbert_of_cell(u32 gx, u32 gy, u32 gz, const unsigned short* table,
                                               const unsigned short* t1) {
    constexpr u32 kMask = (1u << TL) - 1u, kDigits = (1u << (3 * TL)) - 1u;
    constexpr int kSteps = kLevels == 21 ? 21 / TL : (10 + TL - 1) / TL;
    constexpr int kLeft = kLevels - kSteps * TL;  // 1: one more level; 0; or levels too many (negative)
    u64 key = 0;
    u32 state = 0, acc = 0;  // state: as stored in an entry's high bits; acc: up to 27 bits of digits
#pragma unroll
    for (int q = 0; q < kSteps; ++q) {
        const int sh = 21 - TL * (q + 1);
        const u32 idx = (((gx >> sh) & kMask) << (2 * TL)) | (((gy >> sh) & kMask) << TL) | ((gz >> sh) & kMask);
        const u32 v = table[state | idx];
        acc = (acc << (3 * TL)) | (v & kDigits);
        state = v & ~kDigits;
        constexpr int kPer = 27 / (3 * TL);  // steps whose digits fit acc
        if (q % kPer == kPer - 1 || q == kSteps - 1) {
            key = (key << (3 * TL * (q % kPer + 1))) | acc;
            acc = 0;
        }
    }
    if (kLeft > 0) {
        static_assert(kLeft <= 1, "one single level at most");
        const u32 v = t1[(state >> (3 * TL)) * 8u + (((gx & 1u) << 2) | ((gy & 1u) << 1) | (gz & 1u))];
        key = (key << 3) | (v & 7u);
    }
    return static_cast<Key>(kLeft < 0 ? key >> (3 * (kLeft < 0 ? -kLeft : 0)) : key);
}

template <int CURVE, int TL>
__device__ __forceinline__ Key key_of_cell(u32 gx, u32 gy, u32 gz, const KeySmem& sm, const unsigned short* table) {
    if (CURVE == CSTONE_HILBERT) return hilbert_of_cell<TL>(gx, gy, gz, table, sm.t1);
    return to_key(morton_of(gx, gy, gz));
}

template <int CURVE, int TL, bool VEC>
__global__ void __launch_bounds__(kKeyThreads, 3) keys_kernel(const double* __restrict__ x, const double* __restrict__ y,
                                                             const double* __restrict__ z, long long n,
                                                             const double* __restrict__ box, Key* __restrict__ keys,
                                                             const __grid_constant__ HilbertTable one) {
    __shared__ KeySmem sm;
    extern __shared__ unsigned short table[];  // kTableBytes<TL> for Hilbert keys
    if (CURVE == CSTONE_HILBERT) compose_table<TL>(sm, table, one);
    if (threadIdx.x < 32) make_fast_grid(box, &sm.grid, threadIdx.x < 4);
    __syncthreads();
    auto encode = [&](double px, double py, double pz) -> Key {
        u32 c[3];
        u64 X[3];
        cells_of(sm.grid, px, py, pz, c, X);
        return key_of_cell<CURVE, TL>(c[0], c[1], c[2], sm, table);
    };

    if (!VEC) {
        for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
            keys[i] = encode(__ldcg(x + i), __ldcg(y + i), __ldcg(z + i));
        return;
    }
    const long long pairs = n >> 1;
    const double2* x2 = reinterpret_cast<const double2*>(x);
    const double2* y2 = reinterpret_cast<const double2*>(y);
    const double2* z2 = reinterpret_cast<const double2*>(z);
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < pairs; i += (long long)gridDim.x * blockDim.x) {
        double2 a = __ldcg(x2 + i), b = __ldcg(y2 + i), c = __ldcg(z2 + i);
        const Key k0 = encode(a.x, b.x, c.x), k1 = encode(a.y, b.y, c.y);
        if constexpr (sizeof(Key) == 8)
            __stcs(reinterpret_cast<ulonglong2*>(keys) + i, make_ulonglong2(k0, k1));
        else
            __stcs(reinterpret_cast<uint2*>(keys) + i, make_uint2(k0, k1));
    }
    if ((n & 1) && blockIdx.x == 0 && threadIdx.x == 0) {
        long long i = n - 1;
        keys[i] = encode(x[i], y[i], z[i]);
    }
}

// Keys and each particle's multipole record (fixed-point position and mass, records.cuh) from
// the same read of the coordinates. A warp takes 64 consecutive particles, lane l the particles
// l and l + 32: both halves keep the warp's loads and stores contiguous (a warp's two 16-byte
// record stores cover 1 KB), and the two encodings interleave.
template <int CURVE, int TL>
__global__ void __launch_bounds__(kKeyThreads, 2)
    keys_records_kernel(const double* __restrict__ x, const double* __restrict__ y, const double* __restrict__ z,
                        const float* __restrict__ m, long long n, const double* __restrict__ box,
                        Key* __restrict__ keys, Record* __restrict__ rec, WsHeader* hdr,
                        const __grid_constant__ HilbertTable one) {
    __shared__ KeySmem sm;
    __shared__ FixedFrame s_frame;
    extern __shared__ unsigned short table[];  // kTableBytes<TL> for Hilbert keys
    if (CURVE == CSTONE_HILBERT) compose_table<TL>(sm, table, one);
    if (threadIdx.x < 32) make_fast_grid(box, &sm.grid, threadIdx.x < 4);
    if (threadIdx.x == 32) s_frame = make_frame(box);
    __syncthreads();
    const FixedFrame fr = s_frame;
    const long long lane = threadIdx.x & 31;
    const long long warps = (long long)gridDim.x * (blockDim.x >> 5);
    auto encode = [&](long long i, double px, double py, double pz, float pm) -> Key {
        u32 c[3];
        u64 X[3];  // the grid's frame is the records'
        bool in = cells_of(sm.grid, px, py, pz, c, X);
        if (!sm.grid.fast) {
            const double p[3] = {px, py, pz};
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const bool ok = exponent_of(p[d]) < fr.e_lim;
                X[d] = ok ? static_cast<u64>(fixed_of(p[d], fr.F)) : 0ULL;
                in = in && ok;
            }
        }
        longlong2* dst = reinterpret_cast<longlong2*>(rec + i);
        __stcs(dst, make_longlong2(in ? static_cast<long long>(X[0]) : 0, in ? static_cast<long long>(X[1]) : 0));
        __stcs(dst + 1, make_longlong2(in ? static_cast<long long>(X[2]) : 0, static_cast<long long>(__float_as_uint(pm))));
        if (!in) raise_error(hdr, CSTONE_ERR_INVALID_ARG, static_cast<u32>(i));
        return key_of_cell<CURVE, TL>(c[0], c[1], c[2], sm, table);
    };
    for (long long base = ((long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * 64; base < n;
         base += warps * 64) {
        const long long i0 = base + lane, i1 = base + 32 + lane;
        if (i0 >= n) break;
        const bool ok1 = i1 < n;
        const double ax = __ldcg(x + i0), ay = __ldcg(y + i0), az = __ldcg(z + i0);
        const float am = __ldcg(m + i0);
        double bx = 0.0, by = 0.0, bz = 0.0;
        float bm = 0.f;
        if (ok1) {
            bx = __ldcg(x + i1);
            by = __ldcg(y + i1);
            bz = __ldcg(z + i1);
            bm = __ldcg(m + i1);
        }
        keys[i0] = encode(i0, ax, ay, az, am);
        if (ok1) keys[i1] = encode(i1, bx, by, bz, bm);
    }
}

// ------------------------------------------------------------------ host: Hilbert state machine
// State of Skilling's walk seen from one bit level: perm[i] = input axis currently feeding
// transposed axis i, flip[i] = inversion of that axis, gray = parity of the Gray-coded third
// axis over the levels above (the final per-level flip of Skilling's algorithm).
struct WalkState {
    int perm[3];
    int flip[3];
    int gray;
    bool operator==(const WalkState& o) const {
        for (int i = 0; i < 3; ++i)
            if (perm[i] != o.perm[i] || flip[i] != o.flip[i]) return false;
        return gray == o.gray;
    }
};

// One bit level: input octant bits (x high) -> output digit, state updated for the next level.
int walk_level(WalkState& s, int octant) {
    int in[3] = {(octant >> 2) & 1, (octant >> 1) & 1, octant & 1};
    int e[3];
    for (int i = 0; i < 3; ++i) e[i] = in[s.perm[i]] ^ s.flip[i];
    for (int i = 0; i < 3; ++i) {
        if (e[i]) {
            s.flip[0] ^= 1;  // inversion of the first axis' lower bits
        } else {             // exchange of the lower bits of the first axis and axis i
            int tp = s.perm[0], tf = s.flip[0];
            s.perm[0] = s.perm[i];
            s.flip[0] = s.flip[i];
            s.perm[i] = tp;
            s.flip[i] = tf;
        }
    }
    int g0 = e[0], g1 = e[1] ^ e[0], g2 = e[2] ^ g1;
    int digit = ((g0 ^ s.gray) << 2) | ((g1 ^ s.gray) << 1) | (g2 ^ s.gray);
    s.gray ^= g2;
    return digit;
}

const HilbertTable& hilbert_table() {
    static HilbertTable table;
    static std::once_flag once;
    std::call_once(once, [] {
        WalkState states[kHilbertStates];
        int count = 1;
        states[0] = WalkState{{0, 1, 2}, {0, 0, 0}, 0};
        int next1[kHilbertStates][8], digit1[kHilbertStates][8];
        for (int s = 0; s < count; ++s) {
            for (int o = 0; o < 8; ++o) {
                WalkState w = states[s];
                digit1[s][o] = walk_level(w, o);
                int id = -1;
                for (int k = 0; k < count; ++k)
                    if (states[k] == w) id = k;
                if (id < 0) {
                    id = count;
                    if (count < kHilbertStates) states[count++] = w;
                }
                next1[s][o] = id;
            }
        }
        for (int s = 0; s < kHilbertStates; ++s) {
            for (int o = 0; o < 8; ++o)
                table.one[s * 8 + o] = static_cast<unsigned short>(digit1[s][o] | (next1[s][o] << 3));
        }
    });
    return table;
}

// ------------------------------------------------------------------ batched sets
// Set of particle p: the last set whose first particle is <= p (sets are stored back to back).
__device__ __forceinline__ int set_of(const long long* __restrict__ set_offsets, int n_sets, long long p) {
    int lo = 0, hi = n_sets;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(set_offsets + mid) <= p)
            lo = mid;
        else
            hi = mid;
    }
    while (lo + 1 < n_sets && __ldg(set_offsets + lo + 1) <= p) ++lo;  // skip empty sets
    return lo;
}

// Bounding cube of every set: one cluster of kBoxCluster blocks per set (a large set is read by
// kBoxCluster SMs, not one); each block reduces its share of the set, and the cluster's first block
// combines the blocks' results from their shared memory (distributed shared memory of the cluster).
// Bound by loads in flight and by clusters, which start only where 16 blocks are free: six blocks per SM (with 44
// registers and five, 500 sets of 2 or 2,000 particles took 68 and 76 us; so 60 and 66). Large sets are read in
// pairs of particles by 16-byte loads (512 sets of 1,024 to 1,048,576: 457 -> 406 us; 4 of 4 million 474 -> 328); more
// in flight per thread, 512 threads or clusters of 8 gained nothing more. Sets of at most two particles per thread
// are read one by one, since the pairs' odd ends would be a second round of loads.
constexpr int kBoxCluster = 16;  // a non-portable cluster size, allowed per kernel at launch
constexpr int kBoxThreads = 256;

__global__ void __cluster_dims__(kBoxCluster, 1, 1) __launch_bounds__(kBoxThreads, 6)
    bbox_batched_kernel(const double* __restrict__ x, const double* __restrict__ y, const double* __restrict__ z,
                        const long long* __restrict__ set_offsets, double* __restrict__ boxes) {
    __shared__ long long s_lo[kBoxThreads / 32][3], s_hi[kBoxThreads / 32][3];
    __shared__ long long s_blo[3], s_bhi[3];  // this block's result, read by the cluster's first block
    cg::cluster_group cluster = cg::this_cluster();
    const unsigned rank = cluster.block_rank();
    const int set = static_cast<int>(blockIdx.x / kBoxCluster);
    const long long a = set_offsets[set], b = set_offsets[set + 1];
    long long lo[3] = {kOrderedMax, kOrderedMax, kOrderedMax}, hi[3] = {kOrderedMin, kOrderedMin, kOrderedMin};
    const double* c[3] = {x, y, z};
    auto take = [&](int d, double v) {
        const long long o = ordered_bits(v);
        lo[d] = min(lo[d], o);
        hi[d] = max(hi[d], o);
    };
    const long long first = static_cast<long long>(rank) * kBoxThreads + threadIdx.x;
    constexpr long long kStep = static_cast<long long>(kBoxCluster) * kBoxThreads;
    constexpr long long kPairsFrom = 2 * kStep;
    const uintptr_t bases = reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(y) |
                            reinterpret_cast<uintptr_t>(z);
    if ((bases & 15u) == 0 && b - a > kPairsFrom) {  // pairs of particles of even index, and the odd ones at the set's ends
        const long long q1 = b >> 1;
        for (long long q = ((a + 1) >> 1) + first; q < q1; q += kStep) {
            double2 v[3];
#pragma unroll
            for (int d = 0; d < 3; ++d) v[d] = __ldg(reinterpret_cast<const double2*>(c[d]) + q);
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                take(d, v[d].x);
                take(d, v[d].y);
            }
        }
        const long long odd = first == 0 ? a : b - 1;  // a when it is odd, b - 1 when it is even
        if (a < b && ((first == 0 && (a & 1)) || (first == 1 && (b & 1)))) {
#pragma unroll
            for (int d = 0; d < 3; ++d) take(d, __ldg(c[d] + odd));
        }
    } else {
        for (long long i = a + first; i < b; i += kStep) {
#pragma unroll
            for (int d = 0; d < 3; ++d) take(d, __ldg(c[d] + i));
        }
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        for (int sft = 16; sft > 0; sft >>= 1) {
            lo[d] = min(lo[d], __shfl_xor_sync(0xffffffffu, lo[d], sft));
            hi[d] = max(hi[d], __shfl_xor_sync(0xffffffffu, hi[d], sft));
        }
    }
    const int warp = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0)
        for (int d = 0; d < 3; ++d) {
            s_lo[warp][d] = lo[d];
            s_hi[warp][d] = hi[d];
        }
    __syncthreads();
    if (threadIdx.x < 3) {
        const int d = threadIdx.x;
        long long l = s_lo[0][d], h = s_hi[0][d];
        for (int w = 1; w < kBoxThreads / 32; ++w) {
            l = min(l, s_lo[w][d]);
            h = max(h, s_hi[w][d]);
        }
        s_blo[d] = l;
        s_bhi[d] = h;
    }
    cluster.sync();  // every block's result is in its shared memory
    if (rank == 0 && threadIdx.x == 0) {
        double* box = boxes + 4 * set;
        if (b <= a) {
            box[0] = box[1] = box[2] = 0.0;
            box[3] = 1.0;
        } else {
            double side = 0.0;
            for (int d = 0; d < 3; ++d) {
                long long l = s_blo[d], h = s_bhi[d];
                for (unsigned r = 1; r < kBoxCluster; ++r) {
                    l = min(l, cluster.map_shared_rank(s_blo, r)[d]);
                    h = max(h, cluster.map_shared_rank(s_bhi, r)[d]);
                }
                const double lod = from_ordered(l), hid = from_ordered(h);
                box[d] = lod;
                const double ext = __dsub_rn(hid, lod);
                side = ext > side ? ext : side;
            }
            box[3] = side > 0.0 ? side : 1.0;
        }
    }
    cluster.sync();  // the other blocks keep their shared memory until it has been read
}

__global__ void keys_batched_setup_kernel(const double* __restrict__ boxes, int n_sets, FastGrid* grids) {
    const int set = static_cast<int>((blockIdx.x * blockDim.x + threadIdx.x) >> 2);  // four lanes per set
    const int at = min(set, n_sets - 1);
    make_fast_grid(boxes + 4 * at, grids + at, set < n_sets);
}

// A block takes a stretch of consecutive tiles of particles. Where a tile lies in one set, which one load
// shows, its grid is read from shared memory, else every particle looks its set up; so does every particle
// of sets that are smaller than a tile on average (by_tile is 0), instead of a search before its own.
constexpr int kBatchItems = 2;
constexpr int kBatchTile = kKeyThreads * kBatchItems;

template <int CURVE, int TL>
__global__ void __launch_bounds__(kKeyThreads, 3) keys_batched_kernel(const double* __restrict__ x,
                                                                     const double* __restrict__ y,
                                                                     const double* __restrict__ z,
                                                                     const long long* __restrict__ set_offsets, int n_sets,
                                                                     long long n, int by_tile, const FastGrid* __restrict__ grids,
                                                                     Key* __restrict__ keys,
                                                                     const __grid_constant__ HilbertTable one) {
    __shared__ KeySmem sm;
    extern __shared__ unsigned short table[];  // kTableBytes<TL> for Hilbert keys
    if (CURVE == CSTONE_HILBERT) compose_table<TL>(sm, table, one);
    const u32 tiles = static_cast<u32>((n + kBatchTile - 1) / kBatchTile);
    const u32 b0 = static_cast<u32>(static_cast<u64>(tiles) * blockIdx.x / gridDim.x);
    const u32 b1 = static_cast<u32>(static_cast<u64>(tiles) * (blockIdx.x + 1) / gridDim.x);
    int set = 0;              // set of the tile's first particle
    u32 first = 0, end = 0;   // its particles
    if (!by_tile) __syncthreads();  // the table
    for (u32 tile = b0; tile < b1; ++tile) {
        const u32 t0 = tile * kBatchTile, t1 = min(t0 + kBatchTile, static_cast<u32>(n));
        double p[kBatchItems][3];
#pragma unroll
        for (int k = 0; k < kBatchItems; ++k) {
            const u32 i = t0 + k * kKeyThreads + threadIdx.x;
            const bool on = i < t1;
            p[k][0] = on ? __ldcg(x + i) : 0.0;
            p[k][1] = on ? __ldcg(y + i) : 0.0;
            p[k][2] = on ? __ldcg(z + i) : 0.0;
        }
        if (by_tile && t0 >= end) {  // the same in every thread
            set = set_of(set_offsets, n_sets, t0);
            first = static_cast<u32>(__ldg(set_offsets + set));
            end = static_cast<u32>(__ldg(set_offsets + set + 1));
            __syncthreads();  // the table, and the previous set's grids
            if (threadIdx.x < sizeof(FastGrid) / 8)
                reinterpret_cast<u64*>(&sm.grid)[threadIdx.x] = __ldg(reinterpret_cast<const u64*>(grids + set) + threadIdx.x);
            __syncthreads();
        }
        const bool whole = t0 >= first && t1 <= end;
#pragma unroll
        for (int k = 0; k < kBatchItems; ++k) {
            const u32 i = t0 + k * kKeyThreads + threadIdx.x;
            u32 c[3];
            u64 X[3];
            if (whole || (i >= first && i < end))
                cells_of(sm.grid, p[k][0], p[k][1], p[k][2], c, X);
            else
                cells_of(grids[set + set_of(set_offsets + set, n_sets - set, i < t1 ? i : t0)], p[k][0], p[k][1], p[k][2],
                         c, X);
            if (i < t1) keys[i] = key_of_cell<CURVE, TL>(c[0], c[1], c[2], sm, table);
        }
    }
}

}  // namespace

const HilbertDecodeTable& hilbert_decode_table() {
    static HilbertDecodeTable dec;
    static std::once_flag once;
    std::call_once(once, [] {
        const HilbertTable& t = hilbert_table();
        for (int s = 0; s < kHilbertStates; ++s)
            for (int o = 0; o < 8; ++o) {
                const int e = t.one[s * 8 + o];
                dec.one[s * 8 + (e & 7)] = static_cast<unsigned short>(o | ((e >> 3) << 3));
            }
    });
    return dec;
}

// Dynamic shared memory beyond the default limit (48 KB with the static part) for the three-level table.
template <class Kernel>
int allow_table(Kernel kernel, size_t smem) {
    if (smem > kTableBytes<2>)
        CST_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem)));
    return CSTONE_OK;
}

size_t keys_batched_ws_bytes(int n_sets) {
    Carver c(nullptr);
    c.take<FastGrid>((size_t)n_sets);
    return c.size();
}

int launch_bbox_batched(const double* x, const double* y, const double* z, const long long* set_offsets, int n_sets,
                        double* boxes, cudaStream_t st) {
    CST_CUDA(cudaFuncSetAttribute(bbox_batched_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    bbox_batched_kernel<<<n_sets * kBoxCluster, kBoxThreads, 0, st>>>(x, y, z, set_offsets, boxes);
    CST_LAUNCHED("bbox_batched_kernel");
    return CSTONE_OK;
}

int launch_keys_batched(const double* x, const double* y, const double* z, const long long* set_offsets, int n_sets,
                        long long n, const double* boxes, int curve, Key* keys, void* ws, cudaStream_t st) {
    Carver c(ws);
    FastGrid* grids = c.take<FastGrid>((size_t)n_sets);
    keys_batched_setup_kernel<<<(n_sets + 31) / 32, 128, 0, st>>>(boxes, n_sets, grids);
    CST_LAUNCHED("keys_batched_setup_kernel");
    if (n == 0) return CSTONE_OK;
    const HilbertTable& tab = hilbert_table();
    const int by_tile = n >= static_cast<long long>(n_sets) * kBatchTile ? 1 : 0;
    const long long want = (n + kBatchTile - 1) / kBatchTile, most = (long long)sm_count() * kKeyBlocks;
    const unsigned grid = static_cast<unsigned>(want < most ? want : most);
    auto launch = [&](auto kernel, size_t smem) -> int {
        if (int rc = allow_table(kernel, smem)) return rc;
        kernel<<<grid, kKeyThreads, smem, st>>>(x, y, z, set_offsets, n_sets, n, by_tile, grids, keys, tab);
        CST_LAUNCHED("keys_batched_kernel");
        return CSTONE_OK;
    };
    if (curve != CSTONE_HILBERT) return launch(keys_batched_kernel<CSTONE_MORTON, 2>, 0);
    if (n < kTwoLevelMax) return launch(keys_batched_kernel<CSTONE_HILBERT, 2>, kTableBytes<2>);
    return launch(keys_batched_kernel<CSTONE_HILBERT, 3>, kTableBytes<3>);
}

int launch_keys(const double* x, const double* y, const double* z, long long n, const double* box, int curve,
                Key* keys, cudaStream_t st) {
    if (n == 0) return CSTONE_OK;
    const HilbertTable& tab = hilbert_table();
    const long long want = ((n + 1) / 2 + kKeyThreads - 1) / kKeyThreads, most = (long long)sm_count() * kKeyBlocks;
    const unsigned grid = static_cast<unsigned>(want < most ? want : most);
    const bool vec = ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(y) | reinterpret_cast<uintptr_t>(z) |
                       reinterpret_cast<uintptr_t>(keys)) & 15u) == 0;
    auto launch = [&](auto kernel, size_t smem) -> int {
        if (int rc = allow_table(kernel, smem)) return rc;
        kernel<<<grid, kKeyThreads, smem, st>>>(x, y, z, n, box, keys, tab);
        CST_LAUNCHED("keys_kernel");
        return CSTONE_OK;
    };
    if (curve != CSTONE_HILBERT)
        return vec ? launch(keys_kernel<CSTONE_MORTON, 2, true>, 0) : launch(keys_kernel<CSTONE_MORTON, 2, false>, 0);
    if (n < kTwoLevelMax)
        return vec ? launch(keys_kernel<CSTONE_HILBERT, 2, true>, kTableBytes<2>)
                   : launch(keys_kernel<CSTONE_HILBERT, 2, false>, kTableBytes<2>);
    return vec ? launch(keys_kernel<CSTONE_HILBERT, 3, true>, kTableBytes<3>)
               : launch(keys_kernel<CSTONE_HILBERT, 3, false>, kTableBytes<3>);
}

// Keys and multipole records in one pass; ws holds only the header (error word).
int launch_keys_records(const double* x, const double* y, const double* z, const float* m, long long n,
                        const double* box, int curve, Key* keys, Record* rec, void* ws, cudaStream_t st) {
    WsHeader* hdr = reinterpret_cast<WsHeader*>(ws);
    CST_CUDA(cudaMemsetAsync(hdr, 0, sizeof(WsHeader), st));
    if (n == 0) return CSTONE_OK;
    const HilbertTable& tab = hilbert_table();
    const long long per = 2 * kKeyThreads;  // 64 particles per warp and step
    const long long want = (n + per - 1) / per, most = (long long)sm_count() * kKeyBlocks;
    const unsigned grid = static_cast<unsigned>(want < most ? want : most);
    auto launch = [&](auto kernel, size_t smem) -> int {
        if (int rc = allow_table(kernel, smem)) return rc;
        kernel<<<grid, kKeyThreads, smem, st>>>(x, y, z, m, n, box, keys, rec, hdr, tab);
        CST_LAUNCHED("keys_records_kernel");
        return CSTONE_OK;
    };
    if (curve != CSTONE_HILBERT) return launch(keys_records_kernel<CSTONE_MORTON, 2>, 0);
    if (n < kTwoLevelMax) return launch(keys_records_kernel<CSTONE_HILBERT, 2>, kTableBytes<2>);
    return launch(keys_records_kernel<CSTONE_HILBERT, 3>, kTableBytes<3>);
}

// bounding cube (bounds == false: box = {lo, side}) or per-axis bounds (bounds == true)
int launch_bbox(const double* x, const double* y, const double* z, long long n, double* box, void* ws,
                cudaStream_t st, bool bounds = false) {
    Carver c(ws);
    BoxAcc* acc = c.take<BoxAcc>(1);
    bbox_init_kernel<<<1, 32, 0, st>>>(acc);
    CST_LAUNCHED("bbox_init_kernel");
    if (n > 0) {
        long long want = (n + 1023) / 1024;  // 16 blocks per SM measured best (two waves of 8)
        int grid = static_cast<int>(want < (long long)sm_count() * 16 ? want : (long long)sm_count() * 16);
        bbox_reduce_kernel<<<grid, 256, 0, st>>>(x, y, z, n, acc);
        CST_LAUNCHED("bbox_reduce_kernel");
    }
    if (bounds) {
        bounds_finalize_kernel<<<1, 32, 0, st>>>(acc, n, box);
        CST_LAUNCHED("bounds_finalize_kernel");
    } else {
        bbox_finalize_kernel<<<1, 32, 0, st>>>(acc, n, box);
        CST_LAUNCHED("bbox_finalize_kernel");
    }
    return CSTONE_OK;
}

size_t bbox_ws_bytes() {
    Carver c(nullptr);
    c.take<BoxAcc>(1);
    return c.size();
}

}  // namespace CST_NS

extern "C" {

int CSTONE_FN(keys)(const double* x, const double* y, const double* z, int64_t n, const double* box, int curve,
                    CST_KEY_C* keys, void* stream) {
    if (n < 0 || n >= CSTONE_MAX_PARTICLES || !box || (n > 0 && (!x || !y || !z || !keys)))
        return cst::fail(CSTONE_ERR_INVALID_ARG, CST_STR(CSTONE_FN(keys)) ": bad argument (n=%lld)", (long long)n);
    if (curve != CSTONE_MORTON && curve != CSTONE_HILBERT)
        return cst::fail(CSTONE_ERR_INVALID_ARG, CST_STR(CSTONE_FN(keys)) ": unknown curve %d", curve);
    if (((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(y) | reinterpret_cast<uintptr_t>(z)) & 7u) != 0 ||
        (reinterpret_cast<uintptr_t>(keys) & (sizeof(CST_KEY_C) - 1)) != 0)
        return cst::fail(CSTONE_ERR_INVALID_ARG, CST_STR(CSTONE_FN(keys)) ": arrays must be aligned to their element size");
    return CST_NS::launch_keys(x, y, z, n, box, curve, reinterpret_cast<CST_NS::Key*>(keys), cst::as_stream(stream));
}

int CSTONE_FN(keys_records)(const double* x, const double* y, const double* z, const float* m, int64_t n,
                            const double* box, int curve, CST_KEY_C* keys, void* records, void* ws, size_t ws_bytes,
                            void* stream) {
    if (n < 0 || n >= CSTONE_MAX_PARTICLES || !box || (n > 0 && (!x || !y || !z || !m || !keys || !records)))
        return cst::fail(CSTONE_ERR_INVALID_ARG, CST_STR(CSTONE_FN(keys_records)) ": bad argument (n=%lld)",
                         (long long)n);
    if (curve != CSTONE_MORTON && curve != CSTONE_HILBERT)
        return cst::fail(CSTONE_ERR_INVALID_ARG, CST_STR(CSTONE_FN(keys_records)) ": unknown curve %d", curve);
    if (((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(y) | reinterpret_cast<uintptr_t>(z)) & 7u) != 0 ||
        (reinterpret_cast<uintptr_t>(m) & 3u) != 0 || (reinterpret_cast<uintptr_t>(records) & 15u) != 0 ||
        (reinterpret_cast<uintptr_t>(keys) & (sizeof(CST_KEY_C) - 1)) != 0)
        return cst::fail(CSTONE_ERR_INVALID_ARG,
                         CST_STR(CSTONE_FN(keys_records)) ": arrays must be aligned (records to 16 bytes)");
    if (int rc = cst::check_ws(ws, ws_bytes, sizeof(cst::WsHeader), CST_STR(CSTONE_FN(keys_records)))) return rc;
    return CST_NS::launch_keys_records(x, y, z, m, n, box, curve, reinterpret_cast<CST_NS::Key*>(keys),
                                       static_cast<cst::Record*>(records), ws, cst::as_stream(stream));
}

#ifndef CSTONE_KEY32  // the bounding cube and the batched entry points exist once, for 63-bit keys
int cstone_records_size(int64_t n, size_t* bytes) {
    if (!bytes || n < 0 || n >= CSTONE_MAX_PARTICLES)
        return cst::fail(CSTONE_ERR_INVALID_ARG, "cstone_records_size: bad argument");
    *bytes = static_cast<size_t>(n > 0 ? n : 1) * sizeof(cst::Record);
    return CSTONE_OK;
}

int cstone_keys_records_workspace_size(size_t* bytes) {
    if (!bytes) return cst::fail(CSTONE_ERR_INVALID_ARG, "cstone_keys_records_workspace_size: bad argument");
    *bytes = sizeof(cst::WsHeader);
    return CSTONE_OK;
}

int cstone_bbox_workspace_size(int64_t n, size_t* bytes) {
    if (!bytes || n < 0) return cst::fail(CSTONE_ERR_INVALID_ARG, "cstone_bbox_workspace_size: bad argument");
    *bytes = cst::bbox_ws_bytes();
    return CSTONE_OK;
}

int cstone_bbox(const double* x, const double* y, const double* z, int64_t n, double* box, void* ws, size_t ws_bytes,
                void* stream) {
    if (n < 0 || n >= CSTONE_MAX_PARTICLES || !box || (n > 0 && (!x || !y || !z)))
        return cst::fail(CSTONE_ERR_INVALID_ARG, "cstone_bbox: bad argument (n=%lld)", (long long)n);
    if (int rc = cst::check_ws(ws, ws_bytes, cst::bbox_ws_bytes(), "cstone_bbox")) return rc;
    return cst::launch_bbox(x, y, z, n, box, ws, cst::as_stream(stream));
}

int cstone_bounds(const double* x, const double* y, const double* z, int64_t n, double* bounds, void* ws,
                  size_t ws_bytes, void* stream) {
    if (n < 0 || n >= CSTONE_MAX_PARTICLES || !bounds || (n > 0 && (!x || !y || !z)))
        return cst::fail(CSTONE_ERR_INVALID_ARG, "cstone_bounds: bad argument (n=%lld)", (long long)n);
    if (int rc = cst::check_ws(ws, ws_bytes, cst::bbox_ws_bytes(), "cstone_bounds")) return rc;
    return cst::launch_bbox(x, y, z, n, bounds, ws, cst::as_stream(stream), true);
}

int cstone_bbox_batched(const double* x, const double* y, const double* z, const int64_t* set_offsets, int32_t n_sets,
                        double* boxes, void* stream) {
    if (n_sets < 1 || n_sets > (1 << 20) || !set_offsets || !boxes || !x || !y || !z)
        return cst::fail(CSTONE_ERR_INVALID_ARG, "cstone_bbox_batched: bad argument");
    return cst::launch_bbox_batched(x, y, z, reinterpret_cast<const long long*>(set_offsets), n_sets, boxes,
                                    cst::as_stream(stream));
}

int cstone_keys_batched_workspace_size(int32_t n_sets, size_t* bytes) {
    if (!bytes || n_sets < 1 || n_sets > (1 << 20))
        return cst::fail(CSTONE_ERR_INVALID_ARG, "cstone_keys_batched_workspace_size: bad argument");
    *bytes = cst::keys_batched_ws_bytes(n_sets);
    return CSTONE_OK;
}

int cstone_keys_batched(const double* x, const double* y, const double* z, int64_t n, const int64_t* set_offsets,
                        int32_t n_sets, const double* boxes, int curve, uint64_t* keys, void* ws, size_t ws_bytes,
                        void* stream) {
    if (n < 0 || n >= CSTONE_MAX_PARTICLES || n_sets < 1 || n_sets > (1 << 20) || !set_offsets || !boxes ||
        (n > 0 && (!x || !y || !z || !keys)))
        return cst::fail(CSTONE_ERR_INVALID_ARG, "cstone_keys_batched: bad argument");
    if (curve != CSTONE_MORTON && curve != CSTONE_HILBERT)
        return cst::fail(CSTONE_ERR_INVALID_ARG, "cstone_keys_batched: unknown curve %d", curve);
    if (int rc = cst::check_ws(ws, ws_bytes, cst::keys_batched_ws_bytes(n_sets), "cstone_keys_batched")) return rc;
    return cst::launch_keys_batched(x, y, z, reinterpret_cast<const long long*>(set_offsets), n_sets, n, boxes, curve,
                                    reinterpret_cast<cst::u64*>(keys), ws, cst::as_stream(stream));
}
#endif

}  // extern "C"
