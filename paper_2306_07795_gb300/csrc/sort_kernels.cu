// sort_kernels.cu -- fused passes of the sorting network of Sec. 6.1.
//
// A fused pass is the tiled BMMC pass of Sec. 4.1 (16-byte asynchronous copies
// into swizzled shared memory, barrier, 16-byte gathers and stores) with
// comparator stages run on the tile in between.  The stages come in groups
// (sort_desc.h): for one group, every thread loads 2^R keys of the tile into
// registers, and each stage of the group orders pairs of those registers, the
// pair's low position (index with g_s . x = 0) receiving the smaller key
// (Sec. 6.1: a pair is kept when first <= second and swapped otherwise).  The
// keys go back to the same slots, and a barrier separates the groups.
//
// Arrays of at most 2^12 keys are one block of that kernel; those of at most
// 2^7 run in bmmc_sort_small: keys at their positions in shared memory, one
// stage at a time.
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <atomic>

#include "pass_desc.h"
#include "sort_desc.h"
#include "tile_body.cuh"

namespace bmmc {

namespace {

template <int E_LOG> struct KeyWord;
template <> struct KeyWord<2> { using type = uint32_t; };
template <> struct KeyWord<3> { using type = unsigned long long; };

// Sec. 6.1's comparator: the pair (a at the low position, b at the high one)
// is kept when a <= b.
template <int KEY, typename V>
__device__ __forceinline__ bool keep(V a, V b)
{
    if constexpr (KEY <= dev::kKeyF32) return dev::keep_pair<KEY>((uint32_t)a, (uint32_t)b);
    else return dev::keep_pair64<KEY>((uint64_t)a, (uint64_t)b);
}

// Float keys without NaN and -0.0 are totally ordered, and the pair may be
// ordered by other means than IEEE <=: 4-byte ones by minimum and maximum, and
// 8-byte ones, whose compare runs on the FP64 pipe at about two lanes a clock
// per SM, as integers of the same order.  A block looks at its keys as its
// first group loads them and keeps the exact comparator if any is special.
//
// ordered(): the integer of a double's order, and back (its own inverse); the
// order of signed integers is that of <= outside special keys, NaN beyond the
// infinities and -0.0 just below +0.0.
__device__ __forceinline__ unsigned long long ordered(unsigned long long x)
{
    const uint32_t hi = (uint32_t)(x >> 32), m = (uint32_t)((int32_t)hi >> 31);
    return ((unsigned long long)(hi ^ (m & 0x7fffffffu)) << 32) | ((uint32_t)x ^ m);
}

// Whether any of 2^R keys is special: NaN or -0.0 (8-byte keys as ordered() gives
// them; there also the infinities and negative numbers too small for the high
// word).  By the extremes of the keys' bits (8-byte keys: of the high words) as
// signed and unsigned integers, two keys an instruction (n = 24: float32 692 -> 684 us
// against two compares a key, float64 1658 -> 1647 against three operations).
template <int E, typename V>
__device__ __forceinline__ bool any_special(const V (&v)[E])
{
    constexpr int kShift = sizeof(V) == 8 ? 32 : 0;
    int32_t top = (int32_t)(v[0] >> kShift), low = top;
    uint32_t utop = (uint32_t)top;
#pragma unroll
    for (int j = 1; j < E; j += 2) {
        const uint32_t x = (uint32_t)(v[j] >> kShift);
        const uint32_t y = j + 1 < E ? (uint32_t)(v[j + 1] >> kShift) : x;
        top = __vimax3_s32(top, (int32_t)x, (int32_t)y);
        low = __vimin3_s32(low, (int32_t)x, (int32_t)y);
        utop = __vimax3_u32(utop, x, y);
    }
    if constexpr (sizeof(V) == 4)  // NaN: above the infinities; -0.0: the lowest
        return top > 0x7f800000 || utop > 0xff800000u || low == (int32_t)0x80000000;
    else  // -0.0 has the greatest high word of all, unsigned
        return top >= 0x7ff00000 || low < (int32_t)0x80100000 || utop == ~0u;
}

// How a stage orders pairs: as the key type, or one of these.
constexpr int kF32MinMax = 7;   // 4-byte float keys, none special
constexpr int kF64Ordered = 8;  // ordered() 8-byte float keys, compared as the doubles they are

// a <= b of the doubles whose ordered() integers are a and b: not beyond the
// infinities (NaN), and +0.0 <= -0.0.  n = 24 with a -0.0 among
// every 500 keys: 2006 us; decoding the keys for a compare on the FP64 pipe took
// 2795, and that compare on the keys as they come, in every pass, 5450.
__device__ __forceinline__ bool keep_ordered(unsigned long long a, unsigned long long b)
{
    constexpr long long kMinusInf = (long long)0x800fffffffffffffull;
    constexpr long long kPlusInf = 0x7ff0000000000000ll;
    return ((long long)a <= (long long)b && (long long)a >= kMinusInf &&
            (long long)b <= kPlusInf) ||
           (a | ~b) == 0;
}

// Runtime 1 and -1 (from a kernel parameter, so that the compiler keeps the
// products): x * one + y and y - x as 32-bit multiply-adds.
struct Units {
    uint32_t one, minus_one;
};

__device__ __forceinline__ uint32_t mad32(uint32_t x, uint32_t m, uint32_t y)
{
    uint32_t r;
    asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(r) : "r"(x), "r"(m), "r"(y));
    return r;
}

// The other one of the pair {a, b}, given one of them: a + b - x.
__device__ __forceinline__ uint32_t other(uint32_t a, uint32_t b, uint32_t x, Units u)
{
    return mad32(x, u.minus_one, mad32(a, u.one, b));
}
__device__ __forceinline__ unsigned long long other(unsigned long long a, unsigned long long b,
                                                    unsigned long long x, Units u)
{
    // word by word: both words of x come from the same key
    const uint32_t lo = other((uint32_t)a, (uint32_t)b, (uint32_t)x, u);
    const uint32_t hi =
        other((uint32_t)(a >> 32), (uint32_t)(b >> 32), (uint32_t)(x >> 32), u);
    return ((unsigned long long)hi << 32) | lo;
}

// How many pairs of four take their other key from multiply-adds: the compares,
// minima and selects of a pair run on the ALU pipe at half the issue rate, and
// sharing the work with the multiply-add pipe is faster.  n = 24, none / one /
// two / three / all of four, us: int32 702 / 696 / 685 / 675 / 695, float32
// 768 / 738 / 717 / 731 / 755 (the smaller sorts are fastest with two); int64
// 1916 / 1840 / - / 1656 / 1577, float64 2120 / 2042 / - / 1833 / 1762.
template <typename V> constexpr int kMadPairs = sizeof(V) == 4 ? 2 : 4;

// Order the pair: a becomes the low one, b the high one.
template <int HOW, bool MAD>
__device__ __forceinline__ void order(uint32_t &a, uint32_t &b, Units u)
{
    uint32_t lo, hi;
    if constexpr (HOW == kF32MinMax) {
        lo = __float_as_uint(fminf(__uint_as_float(a), __uint_as_float(b)));
        hi = __float_as_uint(fmaxf(__uint_as_float(a), __uint_as_float(b)));
    } else {
        const bool k = keep<HOW>(a, b);
        lo = k ? a : b;
        hi = k ? b : a;
    }
    if constexpr (MAD) hi = other(a, b, lo, u);
    a = lo;
    b = hi;
}
template <int HOW, bool MAD>
__device__ __forceinline__ void order(unsigned long long &a, unsigned long long &b, Units u)
{
    bool k;
    if constexpr (HOW == kF64Ordered) k = keep_ordered(a, b);
    else k = keep<HOW>(a, b);
    const unsigned long long lo = k ? a : b;
    b = MAD ? other(a, b, lo, u) : k ? b : a;
    a = lo;
}

// One stage on the registers: the pairs (j, j ^ ones at bits I..L-1), bit I of j
// clear at the low position.
template <int I, int L, int HOW, int R, int J = 0, typename V>
__device__ __forceinline__ void ce_run(V (&v)[1 << R], Units u)
{
    if constexpr (L <= R && J < (1 << R)) {
        constexpr int nth = (J & ((1 << I) - 1)) | ((J >> (I + 1)) << I);
        if constexpr (!(J & (1 << I)))
            order<HOW, ((nth & 3) < kMadPairs<V>)>(v[J], v[J ^ ((1 << L) - (1 << I))], u);
        ce_run<I, L, HOW, R, J + 1>(v, u);
    }
}

// The stage of a sort_stage_code (the same for the whole block).
template <int HOW, int R, typename V>
__device__ __forceinline__ void ce_stage(uint32_t code, V (&v)[1 << R], Units u)
{
    static_assert(kSortMaxRegBits == 5, "one case per stage code");
    switch (code) {
    case sort_stage_code(0, 1): ce_run<0, 1, HOW, R>(v, u); break;
    case sort_stage_code(0, 2): ce_run<0, 2, HOW, R>(v, u); break;
    case sort_stage_code(1, 2): ce_run<1, 2, HOW, R>(v, u); break;
    case sort_stage_code(0, 3): ce_run<0, 3, HOW, R>(v, u); break;
    case sort_stage_code(1, 3): ce_run<1, 3, HOW, R>(v, u); break;
    case sort_stage_code(2, 3): ce_run<2, 3, HOW, R>(v, u); break;
    case sort_stage_code(0, 4): ce_run<0, 4, HOW, R>(v, u); break;
    case sort_stage_code(1, 4): ce_run<1, 4, HOW, R>(v, u); break;
    case sort_stage_code(2, 4): ce_run<2, 4, HOW, R>(v, u); break;
    case sort_stage_code(3, 4): ce_run<3, 4, HOW, R>(v, u); break;
    case sort_stage_code(0, 5): ce_run<0, 5, HOW, R>(v, u); break;
    case sort_stage_code(1, 5): ce_run<1, 5, HOW, R>(v, u); break;
    case sort_stage_code(2, 5): ce_run<2, 5, HOW, R>(v, u); break;
    case sort_stage_code(3, 5): ce_run<3, 5, HOW, R>(v, u); break;
    case sort_stage_code(4, 5): ce_run<4, 5, HOW, R>(v, u); break;
    }
}

// The stages of a group of kind sort_cycle_kind(F, FIRST).
template <int HOW, int R, int F, int FIRST, int S = 0, typename V>
__device__ __forceinline__ void run_cycle(V (&v)[1 << R], Units u)
{
    if constexpr (F <= R && S < F) {
        ce_run<(FIRST + S) % F, F, HOW, R>(v, u);
        run_cycle<HOW, R, F, FIRST, S + 1>(v, u);
    }
}

// The first R merges, from stage I of merge L.
template <int HOW, int R, int L = 1, int I = 0, typename V>
__device__ __forceinline__ void run_levels(V (&v)[1 << R], Units u)
{
    if constexpr (L <= R) {
        ce_run<I, L, HOW, R>(v, u);
        if constexpr (I + 1 < L) run_levels<HOW, R, L, I + 1>(v, u);
        else run_levels<HOW, R, L + 1, 0>(v, u);
    }
}

// The stages of a group whose kind is not 0: no choice between stages, which for
// a few warps costs more than the exchanges do (against run_stages alone, int32:
// n = 11 9.8 -> 7.2 us, n = 16 28.2 -> 22.6, n = 24 739 -> 685).
template <int HOW, int R, typename V>
__device__ __forceinline__ void run_kind(uint32_t kind, V (&v)[1 << R], Units u)
{
    switch (kind) {
    case sort_cycle_kind(1, 0): run_cycle<HOW, R, 1, 0>(v, u); break;
    case sort_cycle_kind(2, 0): run_cycle<HOW, R, 2, 0>(v, u); break;
    case sort_cycle_kind(2, 1): run_cycle<HOW, R, 2, 1>(v, u); break;
    case sort_cycle_kind(3, 0): run_cycle<HOW, R, 3, 0>(v, u); break;
    case sort_cycle_kind(3, 1): run_cycle<HOW, R, 3, 1>(v, u); break;
    case sort_cycle_kind(3, 2): run_cycle<HOW, R, 3, 2>(v, u); break;
    case sort_cycle_kind(4, 0): run_cycle<HOW, R, 4, 0>(v, u); break;
    case sort_cycle_kind(4, 1): run_cycle<HOW, R, 4, 1>(v, u); break;
    case sort_cycle_kind(4, 2): run_cycle<HOW, R, 4, 2>(v, u); break;
    case sort_cycle_kind(4, 3): run_cycle<HOW, R, 4, 3>(v, u); break;
    case sort_cycle_kind(5, 0): run_cycle<HOW, R, 5, 0>(v, u); break;
    case sort_cycle_kind(5, 1): run_cycle<HOW, R, 5, 1>(v, u); break;
    case sort_cycle_kind(5, 2): run_cycle<HOW, R, 5, 2>(v, u); break;
    case sort_cycle_kind(5, 3): run_cycle<HOW, R, 5, 3>(v, u); break;
    case sort_cycle_kind(5, 4): run_cycle<HOW, R, 5, 4>(v, u); break;
    case kSortLevelsKind: run_levels<HOW, R>(v, u); break;
    }
}

// The stages of a group, one by one.
template <int HOW, int R, typename V>
__device__ __forceinline__ void run_stages(uint32_t n_stage, uint64_t codes, V (&v)[1 << R], Units u)
{
    for (uint32_t s = n_stage; s > 0; --s, codes >>= 4)
        ce_stage<HOW, R>((uint32_t)codes & 15u, v, u);
}

// XOR of tab[b] over the set bits b of v, b < N.
template <int N>
__device__ __forceinline__ uint32_t xor_table(const uint16_t *tab, uint32_t v)
{
    uint32_t acc = 0;
#pragma unroll
    for (int b = 0; b < N; ++b)
        if ((v >> b) & 1u) acc ^= tab[b];
    return acc;
}

// What a block keeps in shared memory behind its tile: the pass's tables, and
// for each group, in bytes, what its threads read: codes and register offsets in
// a few words, offsets of its lanes (the block's own part included) and warps.
struct GroupTab {
    uint4 head;      // codes; register offsets 0 | 1 << 16, 2 | 3 << 16
    uint32_t reg4;   // register offset 4 | stages << 16 | kind << 24
    uint32_t round;
    uint16_t lane[32];
    uint16_t warp[1 << (kSortMaxThreadBits - 5)];
    uint32_t pad[2];
};
struct SortTab {
    GroupTab grp[kSortMaxGroups];
    SortDesc d;
};

// Fill tab.grp, a warp per group.
template <int E_LOG>
__device__ __forceinline__ void expand_groups(SortTab &tab, uint32_t cta, uint32_t n_cta)
{
    const uint32_t lane = threadIdx.x & 31u;
    const bool cta_bit = lane < n_cta && ((cta >> lane) & 1u);
    for (uint32_t gi = threadIdx.x >> 5; gi < tab.d.n_group; gi += blockDim.x >> 5) {
        const SortGroup &G = tab.d.grp[gi];
        GroupTab &g = tab.grp[gi];
        const uint32_t base = __reduce_xor_sync(0xffffffffu, cta_bit ? (uint32_t)G.cta[lane] : 0u);
        g.lane[lane] = (uint16_t)((base ^ xor_table<5>(G.lane, lane)) << E_LOG);
        if (lane < (1u << (kSortMaxThreadBits - 5)))
            g.warp[lane] = (uint16_t)(xor_table<kSortMaxThreadBits - 5>(G.warp, lane) << E_LOG);
        if (lane == 31u) {
            g.head = make_uint4(G.code[0], G.code[1],
                                ((uint32_t)G.reg[0] | (uint32_t)G.reg[1] << 16) << E_LOG,
                                ((uint32_t)G.reg[2] | (uint32_t)G.reg[3] << 16) << E_LOG);
            g.reg4 = (uint32_t)G.reg[4] << E_LOG | (uint32_t)G.n_stage << 16 |
                     (uint32_t)G.kind << 24;
            g.round = (uint32_t)G.round << E_LOG;
        }
    }
}

// Byte offset of register j of a group: off[j % 8] ^ top[j / 8].
template <int R>
struct RegOffsets {
    static constexpr int LO = 8, HI = (1 << R) / LO;
    uint32_t off[LO], top[HI];

    // reg: byte offsets of the register bits, two in a word
    __device__ __forceinline__ RegOffsets(const uint32_t (&reg)[3], uint32_t base)
    {
        off[0] = base;
        top[0] = 0;
#pragma unroll
        for (int t = 0; t < R; ++t) {
            const uint32_t v = t & 1 ? reg[t / 2] >> 16 : reg[t / 2] & 0xffffu;
            if (t < 3) {
#pragma unroll
                for (int j = 0; j < (1 << t); ++j) off[j + (1 << t)] = off[j] ^ v;
            } else {
#pragma unroll
                for (int j = 0; j < (1 << (t - 3)); ++j) top[j + (1 << (t - 3))] = top[j] ^ v;
            }
        }
    }
    __device__ __forceinline__ uint32_t operator[](int j) const { return off[j % LO] ^ top[j / LO]; }
};

// The groups on the tile.  A group's table entries are loaded together at its
// start and kept: a chain of shared-memory loads in front of the keys and
// again in front of their stores costs a one-block sort more than its stages.
template <int E_LOG, int KEY, int R, int NR>
__device__ __forceinline__ void run_groups(const SortTab &tab, uint8_t *tile, Units u)
{
    using V = typename KeyWord<E_LOG>::type;
    constexpr int E = 1 << R;
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const uint32_t n_group = tab.d.n_group;
    constexpr bool kFloat = KEY == dev::kKeyF32 || KEY == dev::kKeyF64;
    // Whether a key of the block is special is known after the first group's
    // barrier; until then a warp goes by its own keys, since a pair's two are in
    // one thread.  Asking the block before the first group's stages, or looking
    // through the tile beforehand, costs a barrier (n = 24, the latter: float32
    // 718 us against 692, float64 1763 against 1668); only where a thread has one
    // set of 4-byte keys is the extra barrier cheaper than the warp's vote
    // (n = 18 float32 32.3 against 33.3).
    constexpr bool kAskBlock = KEY == dev::kKeyF32 && NR == 1;
    bool exact = false, seen = false;
    for (uint32_t gi = 0; gi < n_group; ++gi) {
        const GroupTab &g = tab.grp[gi];
        const uint4 head = g.head;
        const uint32_t reg[3] = {head.z, head.w, g.reg4 & 0xffffu};
        const uint32_t n_stage = (g.reg4 >> 16) & 0xffu, kind = g.reg4 >> 24, round = g.round;
        const uint32_t base = (uint32_t)g.lane[lane] ^ g.warp[warp];
#pragma unroll 1
        for (int rd = 0; rd < NR; ++rd) {
            const uint32_t at0 = rd ? base ^ round : base;
            V v[E];
            {
                const RegOffsets<R> at(reg, at0);
#pragma unroll
                for (int j = 0; j < E; ++j) v[j] = *reinterpret_cast<const V *>(tile + at[j]);
            }
            uint64_t codes = ((uint64_t)head.y << 32) | head.x;
            if constexpr (kFloat) {
                if (gi == 0) {
                    if constexpr (KEY == dev::kKeyF64)
                        if (tab.d.first_pass)
#pragma unroll
                            for (int j = 0; j < E; ++j) v[j] = ordered(v[j]);
                    const bool any = any_special(v);
                    exact = kAskBlock ? __syncthreads_or(any) : __any_sync(0xffffffffu, any);
                    seen |= exact;
                }
            }
            if constexpr (kFloat) {
                if (exact) {
                    constexpr int how = KEY == dev::kKeyF32 ? KEY : kF64Ordered;
                    // (the sequences for 8-byte keys would cost those without
                    // special ones 1.5 % by their size alone)
                    constexpr bool straight = E_LOG == 2 || R == 3;
                    if (straight && kind) run_kind<how, R>(kind, v, u);
                    else run_stages<how, R>(n_stage, codes, v, u);
                } else {
                    constexpr int how = KEY == dev::kKeyF32 ? kF32MinMax : dev::kKeyI64;
                    if (kind) run_kind<how, R>(kind, v, u);
                    else run_stages<how, R>(n_stage, codes, v, u);
                }
                if constexpr (KEY == dev::kKeyF64)
                    if (tab.d.last_pass && gi + 1 == n_group)
#pragma unroll
                        for (int j = 0; j < E; ++j) v[j] = ordered(v[j]);
            } else if (kind) {
                run_kind<KEY, R>(kind, v, u);
            } else {
                run_stages<KEY, R>(n_stage, codes, v, u);
            }
            {
                // computed again: kept across the stages they would not fit
                // the registers
                uint32_t again = at0;
                asm volatile("" : "+r"(again));
                const RegOffsets<R> at(reg, again);
#pragma unroll
                for (int j = 0; j < E; ++j) *reinterpret_cast<V *>(tile + at[j]) = v[j];
            }
        }
        if (kFloat && !kAskBlock && gi == 0) exact = __syncthreads_or(seen);
        else __syncthreads();
    }
}

// Copy a launch table into shared memory, 4 bytes per thread and step: the
// group loop indexes it by a runtime group and lane.
__device__ __forceinline__ void stage_words(const void *from, void *to, uint32_t bytes)
{
    const uint32_t *src = reinterpret_cast<const uint32_t *>(from);
    uint32_t *dst = reinterpret_cast<uint32_t *>(to);
    for (uint32_t i = threadIdx.x; i < bytes / 4; i += blockDim.x) dst[i] = src[i];
}

constexpr int kMaxSortThreads = 1 << kSortMaxThreadBits;

// Field f of this thread's chunk 0: the block's and warp's part from one
// warp-wide XOR (bits of `outer`: thread block, then warp), the lane's from its
// five bits.
template <int F>
__device__ __forceinline__ uint32_t chunk_field(const SortTile &t, uint32_t outer)
{
    constexpr uint32_t kOuterBits = kSortMaxCtaBits + kSortMaxThreadBits - 5;
    const uint32_t lane = threadIdx.x & 31u;
    uint32_t x = __reduce_xor_sync(
        0xffffffffu, lane < kOuterBits && ((outer >> lane) & 1u) ? t.block[F][lane] : 0u);
#pragma unroll
    for (int b = 0; b < 5; ++b)
        if ((lane >> b) & 1u) x ^= t.lane[F][b];
    return x;
}

// Field f of chunk c relative to chunk 0.
template <int F, int C>
__device__ __forceinline__ uint32_t chunk_step(const SortTile &t)
{
    uint32_t x = 0;
    if constexpr ((C & 1) != 0) x ^= t.chunk[F][0];
    if constexpr ((C & 2) != 0) x ^= t.chunk[F][1];
    if constexpr ((C & 4) != 0) x ^= t.chunk[F][2];
    if constexpr ((C & 8) != 0) x ^= t.chunk[F][3];
    return x;
}

template <int E_LOG, int C, int N>
__device__ __forceinline__ void load_chunks(const SortTile &t, uint32_t from, uint32_t to,
                                            const uint8_t *__restrict__ in, uint32_t sbase)
{
    if constexpr (C < N) {
        const uint32_t g = from ^ chunk_step<kSortIn, C>(t);
        dev::cp_async_16(sbase + (to ^ chunk_step<kSortDst, C>(t)),
                         in + ((uint64_t)g << E_LOG));
        load_chunks<E_LOG, C + 1, N>(t, from, to, in, sbase);
    }
}

// Output chunks C..N-1: the elements from the tile (load j gives element
// j ^ rot), one 16-byte store each.  e: tile offset of element j of chunk 0.
template <int E_LOG, bool ROT, int C, int N>
__device__ __forceinline__ void store_chunks(const SortTile &t, const uint32_t (&e)[16 >> E_LOG],
                                             uint32_t to, uint32_t rot,
                                             uint8_t *__restrict__ out, const uint8_t *tile)
{
    if constexpr (C < N) {
        const uint32_t s = chunk_step<kSortSrc, C>(t);
        const uint32_t o = to ^ chunk_step<kSortOut, C>(t);
        uint4 v;
        if constexpr (E_LOG == 2) {
            uint32_t a0 = *reinterpret_cast<const uint32_t *>(tile + (s ^ e[0]));
            uint32_t a1 = *reinterpret_cast<const uint32_t *>(tile + (s ^ e[1]));
            uint32_t a2 = *reinterpret_cast<const uint32_t *>(tile + (s ^ e[2]));
            uint32_t a3 = *reinterpret_cast<const uint32_t *>(tile + (s ^ e[3]));
            if constexpr (ROT) {
                dev::swap_if((rot & 1u) != 0u, a0, a1);
                dev::swap_if((rot & 1u) != 0u, a2, a3);
                dev::swap_if((rot & 2u) != 0u, a0, a2);
                dev::swap_if((rot & 2u) != 0u, a1, a3);
            }
            v = make_uint4(a0, a1, a2, a3);
        } else {
            uint2 a0 = *reinterpret_cast<const uint2 *>(tile + (s ^ e[0]));
            uint2 a1 = *reinterpret_cast<const uint2 *>(tile + (s ^ e[1]));
            if constexpr (ROT) dev::swap_if((rot & 1u) != 0u, a0, a1);
            v = make_uint4(a0.x, a0.y, a1.x, a1.y);
        }
        dev::stg128(out + ((uint64_t)o << E_LOG), v);
        store_chunks<E_LOG, ROT, C + 1, N>(t, e, to, rot, out, tile);
    }
}

// One block of at most 256 threads per tile of 2^P keys; a thread runs NR sets of
// 2^R keys in turn in each group and moves as many in and out, in 16-byte
// chunks.  64 KiB tiles run as two sets per thread, three blocks per SM, rather
// than 512 threads, two per SM (n = 24 float32, before the stages were straight
// sequences: 804 against 940 us).
//
// What bounds it: in the exchanges the ALU pipe, which takes 1.5 of the 2.5
// instructions of a float pair at half rate; between them loads, shared memory
// and the group barriers, with 24 to 32 warps per SM to hide them (a 14-stage
// pass of 2^24 floats: issue and ALU about half busy, DRAM at 22 % of its peak).
// The 17 passes of that sort take 684 us, 3.3 TB/s in and out and 3.7 T
// comparators a second (1510 us as 29 passes of four-stage groups with a variant
// per orientation); 16 rows of 2^16 doubles 60 us (299); 2^11 integers 7.2 (20).
//
// Four blocks per SM of one set: with 32 4-byte float keys a thread that is 64
// registers and a 24-byte spill, three without it (float32, 4 / 3 blocks, us:
// n = 20 63.5 / 61.6, n = 21 100 / 121, n = 22 184 / 203, n = 23 357 / 375).
template <int E_LOG, int KEY, int R, int NR>
__global__ void __launch_bounds__(kMaxSortThreads, NR == 1 ? 4 : 3)
    bmmc_sort_pass(const __grid_constant__ SortDesc sd, const uint8_t *__restrict__ in,
                   uint8_t *__restrict__ out, Units u)
{
    extern __shared__ __align__(128) uint8_t smem[];
    constexpr int kChunks = NR << R >> (4 - E_LOG);
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(smem);
    SortTab &tab = *reinterpret_cast<SortTab *>(smem + sd.tile_bytes);
    stage_words(&sd, &tab.d,
                (uint32_t)(offsetof(SortDesc, grp) + sd.n_group * sizeof(SortGroup)));
    const uint32_t outer = blockIdx.x | (threadIdx.x >> 5) << kSortMaxCtaBits;
    __syncthreads();
    const SortTile &t = tab.d.tile;
    expand_groups<E_LOG>(tab, blockIdx.x, sd.n_cta);
    {
        const uint32_t from = chunk_field<kSortIn>(t, outer);
        const uint32_t to = chunk_field<kSortDst>(t, outer);
        dev::grid_dependency_wait();
        dev::allow_dependent_launch();
        load_chunks<E_LOG, 0, kChunks>(t, from, to, in, sbase);
    }
    dev::cp_async_wait_all();
    __syncthreads();
    run_groups<E_LOG, KEY, R, NR>(tab, smem, u);
    uint32_t rot = 0;
#pragma unroll
    for (int b = 0; b < 5; ++b)
        if ((threadIdx.x >> b) & 1u) rot ^= t.rot[b];
    const uint32_t src = chunk_field<kSortSrc>(t, outer) ^ t.elem[rot];
    const uint32_t to = chunk_field<kSortOut>(t, outer);
    uint32_t e[16 >> E_LOG];
#pragma unroll
    for (int j = 0; j < (16 >> E_LOG); ++j) e[j] = src ^ t.elem[j];
    if (t.any_rot) store_chunks<E_LOG, true, 0, kChunks>(t, e, to, rot, out, smem);
    else store_chunks<E_LOG, false, 0, kChunks>(t, e, to, rot, out, smem);
}

template <int E_LOG, int KEY>
__global__ void __launch_bounds__(256)
    bmmc_sort_small(const __grid_constant__ SortSmallDesc dp, const uint8_t *__restrict__ in,
                    uint8_t *__restrict__ out)
{
    using V = typename KeyWord<E_LOG>::type;
    extern __shared__ __align__(128) uint8_t smem[];
    V *sm = reinterpret_cast<V *>(smem);
    const V *src = reinterpret_cast<const V *>(in);
    V *dst = reinterpret_cast<V *>(out);
    const uint32_t count = 1u << dp.N;
    // the tables follow the keys
    SortSmallDesc *tab = reinterpret_cast<SortSmallDesc *>(smem + ((size_t)count << E_LOG));
    stage_words(&dp, tab, sizeof(dp));
    const SortSmallDesc &d = *tab;
    dev::grid_dependency_wait();
    dev::allow_dependent_launch();
    for (uint32_t x = threadIdx.x; x < count; x += blockDim.x) sm[x] = src[x];
    __syncthreads();
    for (uint32_t s = 0; s < d.n_stage; ++s) {
        const uint32_t u = d.u[s], g = d.g[s];
        const uint32_t piv = (uint32_t)__ffs((int)u) - 1u;
        const uint32_t below = (1u << piv) - 1u;
        for (uint32_t t = threadIdx.x; t < count / 2; t += blockDim.x) {
            const uint32_t x = ((t & ~below) << 1) | (t & below);  // bit piv of x is 0
            const uint32_t y = x ^ u;
            const bool x_low = (__popc(g & x) & 1) == 0;
            const uint32_t lo = x_low ? x : y, hi = x_low ? y : x;
            const V a = sm[lo], b = sm[hi];
            const bool k = keep<KEY>(a, b);
            sm[lo] = k ? a : b;
            sm[hi] = k ? b : a;
        }
        __syncthreads();
    }
    for (uint32_t x = threadIdx.x; x < count; x += blockDim.x)
        dst[x] = sm[x];
}

template <typename... Args>
cudaError_t launch_pdl(void (*kernel)(Args...), dim3 grid, dim3 block, size_t smem,
                       cudaStream_t s, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

constexpr int kMaxDevices = 64;
constexpr int kSortTile = 64 * 1024;  // largest tile buffer of a fused pass
constexpr int kSortSmem = kSortTile + (int)((sizeof(SortTab) + 127) & ~(size_t)127);
std::atomic<bool> g_sort_attr[kMaxDevices][7][3][2];

template <int E_LOG, int KEY, int R, int NR>
cudaError_t launch_variant(const SortDesc &sd, const void *in, void *out, cudaStream_t s)
{
    const size_t smem = sd.tile_bytes + sizeof(SortTab);
    if (smem > 48 * 1024) {
        int dev = 0;
        cudaError_t err = cudaGetDevice(&dev);
        if (err != cudaSuccess) return err;
        if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
        std::atomic<bool> &flag = g_sort_attr[dev][KEY][R - 3][NR - 1];
        if (!flag.load(std::memory_order_acquire)) {
            err = cudaFuncSetAttribute(bmmc_sort_pass<E_LOG, KEY, R, NR>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, kSortSmem);
            if (err != cudaSuccess) return err;
            flag.store(true, std::memory_order_release);
        }
    }
    const uint32_t threads = sd.tile_bytes / (NR << (E_LOG + R));
    if (threads < 32 || threads > kMaxSortThreads) return cudaErrorInvalidValue;
    return launch_pdl(bmmc_sort_pass<E_LOG, KEY, R, NR>, dim3(1u << sd.n_cta), dim3(threads), smem, s,
                      sd, static_cast<const uint8_t *>(in), static_cast<uint8_t *>(out),
                      Units{1u, ~0u});
}

template <int E_LOG, int KEY>
cudaError_t launch_typed(const SortDesc &sd, const void *in, void *out, cudaStream_t s)
{
    if constexpr (E_LOG == 2) {
        if (sd.reg_bits == 5 && sd.rounds == 1) return launch_variant<E_LOG, KEY, 5, 1>(sd, in, out, s);
        if (sd.reg_bits == 5 && sd.rounds == 2) return launch_variant<E_LOG, KEY, 5, 2>(sd, in, out, s);
    } else if (sd.reg_bits == 4 && sd.rounds == 2) {
        return launch_variant<E_LOG, KEY, 4, 2>(sd, in, out, s);
    }
    if (sd.reg_bits == 3 && sd.rounds == 1) return launch_variant<E_LOG, KEY, 3, 1>(sd, in, out, s);
    if (sd.reg_bits == 4 && sd.rounds == 1) return launch_variant<E_LOG, KEY, 4, 1>(sd, in, out, s);
    return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_sort_pass(const SortDesc &sd, const void *in, void *out, cudaStream_t s)
{
    using namespace dev;
    if (sd.tile_bytes > (uint32_t)kSortTile) return cudaErrorInvalidValue;
    switch (sd.key) {
    case kKeyI32: return launch_typed<2, kKeyI32>(sd, in, out, s);
    case kKeyU32: return launch_typed<2, kKeyU32>(sd, in, out, s);
    case kKeyF32: return launch_typed<2, kKeyF32>(sd, in, out, s);
    case kKeyI64: return launch_typed<3, kKeyI64>(sd, in, out, s);
    case kKeyU64: return launch_typed<3, kKeyU64>(sd, in, out, s);
    case kKeyF64: return launch_typed<3, kKeyF64>(sd, in, out, s);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_sort_small(const SortSmallDesc &d, int e_log, const void *in, void *out,
                              cudaStream_t s)
{
    using namespace dev;
    const size_t smem = (((size_t)1 << d.N) << e_log) + sizeof(SortSmallDesc);
    const uint8_t *src = static_cast<const uint8_t *>(in);
    uint8_t *dst = static_cast<uint8_t *>(out);
    switch (d.key) {
    case kKeyI32: return launch_pdl(bmmc_sort_small<2, kKeyI32>, dim3(1), dim3(256), smem, s, d, src, dst);
    case kKeyU32: return launch_pdl(bmmc_sort_small<2, kKeyU32>, dim3(1), dim3(256), smem, s, d, src, dst);
    case kKeyF32: return launch_pdl(bmmc_sort_small<2, kKeyF32>, dim3(1), dim3(256), smem, s, d, src, dst);
    case kKeyI64: return launch_pdl(bmmc_sort_small<3, kKeyI64>, dim3(1), dim3(256), smem, s, d, src, dst);
    case kKeyU64: return launch_pdl(bmmc_sort_small<3, kKeyU64>, dim3(1), dim3(256), smem, s, d, src, dst);
    case kKeyF64: return launch_pdl(bmmc_sort_small<3, kKeyF64>, dim3(1), dim3(256), smem, s, d, src, dst);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace bmmc
