// sort_desc.h -- launch tables of the fused sorting-network passes, shared by
// the host planner (sortnet.cpp), its host emulation and the CUDA kernels
// (sort_kernels.cu).
//
// The sorting network of Sec. 6.1 is a list of comparator stages.  Written in
// the coordinates of the unsorted array ("virtual" indices), stage s orders
// every pair {x, x + u_s}: the element whose index has g_s . x = 0 receives
// the smaller key (u_s and g_s come from the parm permutations between the
// comparator columns, Sec. 6.2, composed by the fusion rule of Sec. 3).  A
// fused pass is a tiled BMMC pass (Sec. 4.1) whose thread blocks hold tiles
// closed under the partner vectors of a run of stages: after loading a tile
// into shared memory, a block runs those stages on it and only then writes
// it out, in the layout the next pass reads.
//
// Inside a pass the stages are cut into groups.  The f <= R distinct low tests
// of a group's stages, in the order of the network's index bits, are the first
// coordinates of the 2^R keys that a thread holds in registers for the group:
// register j holds the key whose index has test t equal to bit t of j, for
// every t < f, in every thread and block.  The planner finds the slot vectors
// reg[t] dual to the tests in the span of the partner vectors, takes lanes,
// warps and the unused register bits from the common kernel of the tests, and
// moves the block's own part of the tests into its slot base (cta).  So a
// stage is the same exchange between registers everywhere: it pairs j with
// j ^ m, where m, the partner vector in the tests' coordinates, turns out to
// be a run of ones from bit i (the stage's own test) to bit l - 1, and the
// register with bit i clear takes the smaller key.  There are R (R + 1) / 2
// such stages, compiled as that many variants, against 2 R 2^(R-1) with
// registers in the order of the partner vectors, where the test is a parity of
// several register bits and of the block.  A group may hold more than R
// stages: the network's first R levels are one group of R (R + 1) / 2.
// Between groups the registers go back to shared memory.
#pragma once
#include <stdint.h>

#include "pass_desc.h"

namespace bmmc {

constexpr int kSortMaxRegBits = 5;     // R: at most 32 keys per thread
constexpr int kSortMaxThreadBits = 8;  // 256 threads
constexpr int kSortMaxGroups = 26;     // register groups in one pass
constexpr int kSortMaxGroupStages = 16;
constexpr int kSortMaxCtaBits = 20;    // thread-block bits: 32 - 12
constexpr int kSortSmallMaxBits = 7;   // bmmc_sort_small: at most 2^7 keys
constexpr int kSortSmallMaxStages = 28;  // 7 * 8 / 2

// The stage pairing register j with j ^ (ones at bits i..l-1), bit i low.
constexpr BMMC_HD int sort_stage_code(int i, int l) { return l * (l - 1) / 2 + i; }

// A group of f stages that are the f exchanges (i, f) of its tests in cyclic order
// from i = r, as whole groups of a merge are (r = 0, or r > 0 where the group
// runs over the end of a merge into the next).
constexpr BMMC_HD int sort_cycle_kind(int f, int r) { return f * (f - 1) / 2 + r + 1; }
// The group that is the first R merges of the network.
constexpr int kSortLevelsKind = sort_cycle_kind(kSortMaxRegBits, kSortMaxRegBits - 1) + 1;

struct SortGroup {
    uint8_t n_stage;                 // stages of the group
    uint8_t kind;                    // sort_cycle_kind, kSortLevelsKind, or 0 for any other
    uint16_t reg[kSortMaxRegBits];   // slot vector of register bit t
    uint32_t code[2];                // sort_stage_code of stage s: 4 bits at 4 s
    uint16_t lane[5];                // slot vector of lane bit t
    uint16_t warp[kSortMaxThreadBits - 5];  // slot vector of warp bit t
    uint16_t round;                  // slot vector of the second round
    uint16_t cta[kSortMaxCtaBits];   // slot part of thread-block bit b
    uint16_t pad;
};

// How the 16-byte chunks of a tile come in and go out (the tables of pass_desc.h
// by chunk bits of this kernel's blocks): chunk c of a thread, for the input
// its place in the array and in the tile, for the output the tile offset of its
// first element and its place in the array, each the XOR of the entries of the
// set bits of (thread block, warp, lane, c).
enum SortField { kSortIn = 0, kSortDst = 1, kSortSrc = 2, kSortOut = 3 };

struct SortTile {
    // thread-block bits, then warp bits; in and out in elements, tile in bytes
    uint32_t block[4][kSortMaxCtaBits + kSortMaxThreadBits - 5];
    uint32_t lane[4][5];
    uint32_t chunk[4][4];
    uint32_t elem[4];  // tile offset of element j of an output chunk
    uint32_t rot[5];   // element rotation of a lane bit: load j gives element j ^ rot
    uint32_t any_rot;
};

struct SortDesc {
    uint32_t key;          // bmmc_key_type of the keys
    uint32_t reg_bits;     // R
    uint32_t rounds;       // 1 or 2: sets of 2^R keys that a thread runs in turn
    uint32_t n_stage;
    uint32_t n_cta;        // 2^n_cta thread blocks
    uint32_t tile_bytes;   // bytes of a tile, 2^(P + e_log)
    uint32_t first_pass;   // 1: reads the caller's keys; between passes 8-byte
    uint32_t last_pass;    //    float keys are kept as ordered integers
    uint32_t n_group;
    SortTile tile;
    SortGroup grp[kSortMaxGroups];
};

// The whole network on one thread block, for arrays of at most 2^7 keys: the
// keys stay in shared memory at their virtual positions, which are also where
// the network leaves them.
struct SortSmallDesc {
    uint32_t N;        // 2^N keys
    uint32_t key;
    uint32_t n_stage;
    uint32_t pad;
    uint32_t u[kSortSmallMaxStages];
    uint32_t g[kSortSmallMaxStages];
};

}  // namespace bmmc
