// sortnet.cpp -- the sorting network of Sec. 6.1 as a straight program of
// permutations and comparator columns (host only).
//
// The paper writes an even/odd merge sort with a balanced periodic merger in
// terms of parm (Sec. 6.1):
//
//     sort n    = merge n  o  parm 1 (sort (n - 1))
//     merge n   = parm 2^(n-1) (merge (n - 1))  o  vcolumn n
//     vcolumn n = parm 3 (vcolumn (n - 1)),   vcolumn 1 orders a pair
//
// and parm mask f = bmmc(A^{-1}) o parm 2^(n-1) f o bmmc(A) with A the matrix
// of bmmc_parm_matrix (Sec. 6.2), the inner f acting on the low n - 1 index
// bits (the two halves; the top bit is kept).  Unrolling the recursion gives
// a list of permutations and comparator columns; every column orders the
// pairs (2j, 2j + 1), because the innermost f is vcolumn 1 on two elements.
// The fusion rule (Sec. 3) collapses each run of permutations between two
// columns into one matrix, which gives n (n + 1) / 2 stages "permute by M_s,
// then order adjacent pairs" and a final permutation.
#include <cuda_runtime.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <functional>
#include <string>
#include <utility>
#include <vector>

#include "bmmc.h"
#include "bmmc_sort.h"
#include "debug_hooks.hpp"
#include "f2.hpp"
#include "guard.hpp"
#include "sortnet.hpp"
#include "sortnet_plan.hpp"

namespace bmmc {
namespace sortnet {

namespace {

struct Op {
    bool ce;     // true: order the pairs (2j, 2j + 1)
    f2::Mat m;   // the permutation matrix when !ce
};
using Prog = std::vector<Op>;

f2::Mat parm_matrix(int n, uint64_t mask)
{
    f2::Mat a;
    a.n = n;
    const int low = __builtin_ctzll(mask);
    for (int i = 0; i < n; ++i) {
        if (i == n - 1) a.r[i] = mask;
        else if (i < low) a.r[i] = 1ull << i;
        else a.r[i] = 1ull << (i + 1);
    }
    return a;
}

// A program on the low m bits, acting on m + 1 bits with the top bit kept.
Prog lift(const Prog &p, int m)
{
    Prog out = p;
    for (Op &op : out)
        if (!op.ce) {
            op.m.n = m + 1;
            op.m.r[m] = 1ull << m;
        }
    return out;
}

Prog parm(uint64_t mask, const Prog &inner, int n)
{
    const f2::Mat a = parm_matrix(n, mask);
    f2::Mat ainv;
    f2::inverse(a, &ainv);  // parm matrices are permutations of bits: invertible
    Prog out;
    out.push_back({false, a});
    const Prog l = lift(inner, n - 1);
    out.insert(out.end(), l.begin(), l.end());
    out.push_back({false, ainv});
    return out;
}

Prog vcolumn(int n)
{
    if (n == 1) return Prog{{true, f2::Mat()}};
    return parm(3, vcolumn(n - 1), n);
}

Prog merge(int n)
{
    if (n == 0) return {};
    Prog out = vcolumn(n);
    const Prog rest = parm(1ull << (n - 1), merge(n - 1), n);
    out.insert(out.end(), rest.begin(), rest.end());
    return out;
}

Prog sort(int n)
{
    if (n == 0) return {};
    Prog out = parm(1, sort(n - 1), n);
    const Prog m = merge(n);
    out.insert(out.end(), m.begin(), m.end());
    return out;
}

}  // namespace

void schedule(int n, std::vector<f2::Mat> *stages, f2::Mat *final_perm)
{
    stages->clear();
    f2::Mat acc = f2::Mat::identity(n);
    for (const Op &op : sort(n)) {
        if (op.ce) {
            stages->push_back(acc);
            acc = f2::Mat::identity(n);
        } else {
            acc = f2::mul(op.m, acc);  // apply acc first, then op.m
        }
    }
    *final_perm = acc;
}

}  // namespace sortnet
}  // namespace bmmc

extern "C" int bmmc_sort_schedule(int n, uint64_t *stage_rows, int max_stages,
                                  uint64_t *final_rows, int *final_is_identity)
{
    using namespace bmmc;
    if (n < 1 || n > 30) return BMMC_ERR_INVALID;
    const int count = n * (n + 1) / 2;
    if (!stage_rows && !final_rows && !final_is_identity) return count;
    if (stage_rows && max_stages < count) return BMMC_ERR_INVALID;
    return guarded([&] {
        std::vector<f2::Mat> stages;
        f2::Mat fin;
        sortnet::schedule(n, &stages, &fin);
        if ((int)stages.size() != count) return (int)BMMC_ERR_INVALID;
        if (stage_rows)
            for (int s = 0; s < count; ++s)
                memcpy(stage_rows + (size_t)s * n, stages[s].r, sizeof(uint64_t) * n);
        if (final_rows) memcpy(final_rows, fin.r, sizeof(uint64_t) * n);
        if (final_is_identity) *final_is_identity = fin == f2::Mat::identity(n) ? 1 : 0;
        return count;
    });
}

// ---------------------------------------------------------------------------
// Fused passes: several comparator stages per tiled pass
// ---------------------------------------------------------------------------
//
// Virtual coordinates.  Let Q_s = M_s ... M_1 be the permutation applied to
// the array before stage s's comparator column.  That column orders the pairs
// of physical positions (2j, 2j + 1); in the positions of the unsorted array
// (x = Q_s^{-1} y) it orders the pairs {x, x + u_s} with u_s = Q_s^{-1} e_0,
// and the element with g_s . x = 0 (g_s = row 0 of Q_s) takes the smaller key.
// So the network is the stage list (u_s, g_s) followed by one permutation,
// Q_final = F Q_S, and a fused executor may store the array in any layout
// between stages.
//
// Passes.  Pass p reads the array in layout L_{p-1} (virtual x at physical
// L_{p-1} x) and writes it in layout L_p, i.e. it is the BMMC
// T_p = L_p L_{p-1}^{-1} (Sec. 3).  Its thread blocks hold cosets of a
// subspace S_p (virtual) that contains
//   * the partner vectors u_s of the pass's stages (pairs stay in a block),
//   * L_{p-1}^{-1} Lo (whole input segments, Sec. 4.1), and
//   * L_p^{-1} Lo (whole output segments),
// of dimension at most D (a block holds 2^D keys).  L_0 = I and the last
// layout is Q_final.  The planner fills each pass with as many consecutive
// stages as fit, and chooses L_p^{-1} Lo in the span of the next pass's
// partner vectors, and in its own where it can, so that the segments cost
// neither pass a dimension.

namespace bmmc {
namespace sortnet {

namespace {

// Coordinates in a list of independent vectors (bit i: vector i is used), by
// elimination on (vector, combination) pairs.
struct Coords {
    uint32_t vec[32] = {}, comb[32] = {};  // by leading bit

    bool add(uint32_t v, int index)
    {
        uint32_t c = 1u << index;
        reduce(&v, &c);
        if (!v) return false;
        vec[31 - __builtin_clz(v)] = v;
        comb[31 - __builtin_clz(v)] = c;
        return true;
    }
    // False if x is not in the span.
    bool of(uint32_t x, uint32_t *coords) const
    {
        uint32_t c = 0;
        reduce(&x, &c);
        *coords = c;
        return !x;
    }

  private:
    void reduce(uint32_t *v, uint32_t *c) const
    {
        while (*v) {
            const int b = 31 - __builtin_clz(*v);
            if (!vec[b]) return;
            *v ^= vec[b];
            *c ^= comb[b];
        }
    }
};

uint64_t xor_bits64(const uint64_t *tab, uint64_t bits)
{
    uint64_t acc = 0;
    for (int i = 0; bits; ++i, bits >>= 1)
        if (bits & 1ull) acc ^= tab[i];
    return acc;
}

f2::Mat from_columns(const std::vector<uint64_t> &cols, int n)
{
    f2::Mat m;
    m.n = n;
    for (int j = 0; j < n; ++j)
        for (int i = 0; i < n; ++i)
            if ((cols[j] >> i) & 1ull) m.r[i] |= 1ull << j;
    return m;
}

struct PassPlan {
    int first = 0, end = 0;     // stages [first, end)
    std::vector<uint64_t> span;  // S_p (virtual)
    std::vector<uint64_t> out;   // basis of L_p^{-1} Lo
};

// A subspace of F2^32 as a basis with distinct leading bits.
struct Span {
    uint32_t lead[32] = {};  // the basis vector whose leading bit is i, or 0
    int dim = 0;

    uint32_t reduce(uint32_t v) const
    {
        while (v) {
            const uint32_t b = lead[31 - __builtin_clz(v)];
            if (!b) break;
            v ^= b;
        }
        return v;
    }
    bool add(uint32_t v)
    {
        v = reduce(v);
        if (!v) return false;
        lead[31 - __builtin_clz(v)] = v;
        ++dim;
        return true;
    }
};

// k vectors for the segments that a pass with span S writes and the next pass
// reads: combinations of the next pass's stages U[e], U[e + 1], ... that lie in
// S, the earliest first, so that they cost neither pass a dimension; `extra`
// stage vectors that do not lie in S are taken as they come (they cost this
// pass a dimension each).  What the stages do not give is filled from S.
// Returns false if k vectors were not found.
bool next_segments(const std::vector<uint64_t> &U, int e, int walk, int k, int extra,
                   const Span &S, std::vector<uint32_t> *out)
{
    Span W = S;                     // S and the extra vectors taken
    Span got;
    uint32_t rest[32] = {}, comb[32] = {};  // stages outside W: reduced modulo W
                                            // by leading bit, and the combination
    out->clear();
    for (int t = e; t < (int)U.size() && t < e + walk && (int)out->size() < k; ++t) {
        const uint32_t u = (uint32_t)U[t];
        uint32_t r = W.reduce(u), c = u;
        while (r) {
            const int b = 31 - __builtin_clz(r);
            if (!rest[b]) break;
            r = W.reduce(r ^ rest[b]);
            c ^= comb[b];
        }
        if (!r) {
            if (got.add(c)) out->push_back(c);
        } else if (extra > 0) {
            --extra;
            W.add(u);
            if (got.add(u)) out->push_back(u);
            // the kept remainders modulo the larger W
            uint32_t r0[32], c0[32];
            memcpy(r0, rest, sizeof(r0));
            memcpy(c0, comb, sizeof(c0));
            memset(rest, 0, sizeof(rest));
            for (int i = 0; i < 32; ++i) {
                uint32_t r2 = W.reduce(r0[i]), c2 = c0[i];
                while (r2) {
                    const int b = 31 - __builtin_clz(r2);
                    if (!rest[b]) {
                        rest[b] = r2;
                        comb[b] = c2;
                        break;
                    }
                    r2 = W.reduce(r2 ^ rest[b]);
                    c2 ^= comb[b];
                }
            }
        } else {
            rest[31 - __builtin_clz(r)] = r;
            comb[31 - __builtin_clz(r)] = c;
        }
    }
    for (int i = 0; i < 32 && (int)out->size() < k; ++i)
        if (S.lead[i] && got.add(S.lead[i])) out->push_back(S.lead[i]);
    return (int)out->size() == k;
}

// Stages from e on that fit a pass reading the segments in `in`.
int stages_that_fit(const std::vector<uint64_t> &U, int e, const std::vector<uint32_t> &in, int D)
{
    Span sp;
    for (uint32_t v : in) sp.add(v);
    while (e < (int)U.size() && (sp.dim < D || !sp.reduce((uint32_t)U[e]))) {
        sp.add((uint32_t)U[e]);
        ++e;
    }
    return e;
}

// Cut the stages into passes (see above): a beam search over the cuts and the
// segments between passes for the fewest passes.  A cut is (stages done,
// segments); of the cuts reached with one pass more, those from which the next
// pass gets furthest are kept.  Taking the most stages at every pass instead
// leaves no dimension for the next pass's segments, which then cost that pass
// k of its D: 29 passes at n = 24 (D = 14) where this finds 17, and 26 at
// n = 20 (D = 12) where this finds 14.
int group_stages(const std::vector<uint64_t> &U, int k, int D,
                 const std::vector<uint64_t> &o_final, std::vector<PassPlan> *passes)
{
    constexpr int kBeam = 8;      // cuts kept per pass
    constexpr int kShorter = 8;   // ends tried per cut: the furthest and earlier ones
    const int S = (int)U.size();
    struct Cut {
        int from;                  // index of the cut before
        int done;                  // stages run so far
        int reach;                 // stages after one more pass
        std::vector<uint32_t> in;  // segments the next pass reads
    };
    std::vector<Cut> cuts;  // every cut kept, in order of the passes
    Cut first;
    first.from = -1;
    first.done = 0;
    for (int j = 0; j < k; ++j) first.in.push_back(1u << j);
    first.reach = stages_that_fit(U, 0, first.in, D);
    cuts.push_back(first);
    size_t begin = 0;
    int last = -1;
    while (last < 0) {
        const size_t end = cuts.size();
        std::vector<Cut> next;
        for (size_t ci = begin; ci < end && last < 0; ++ci) {
            const Cut &c = cuts[ci];
            Span sp;
            for (uint32_t v : c.in) sp.add(v);
            std::vector<Span> spans;  // spans[i]: after stage c.done + i
            int e = c.done;
            while (e < S && (sp.dim < D || !sp.reduce((uint32_t)U[e]))) {
                sp.add((uint32_t)U[e]);
                spans.push_back(sp);
                ++e;
            }
            if (e == S && !spans.empty()) {
                // the last pass also writes the final layout's segments
                Span all = sp;
                for (uint64_t v : o_final) all.add((uint32_t)v);
                if (all.dim <= D) {
                    last = (int)ci;
                    break;
                }
            }
            const int low = e - kShorter > c.done ? e - kShorter : c.done;
            for (int q = e; q > low; --q) {
                if (q == S) continue;
                const Span &s0 = spans[q - c.done - 1];
                for (int extra = 0; extra <= D - s0.dim && extra <= k; ++extra) {
                    Cut n;
                    if (!next_segments(U, q, 4 * D, k, extra, s0, &n.in)) continue;
                    n.from = (int)ci;
                    n.done = q;
                    n.reach = stages_that_fit(U, q, n.in, D);
                    bool seen = false;
                    for (const Cut &o : next) seen |= o.done == n.done && o.in == n.in;
                    if (!seen) next.push_back(n);
                }
            }
        }
        if (last >= 0) break;
        if (next.empty()) return -3;  // D too small to make progress
        std::stable_sort(next.begin(), next.end(), [](const Cut &a, const Cut &b) {
            return a.reach != b.reach ? a.reach > b.reach : a.done > b.done;
        });
        if ((int)next.size() > kBeam) next.resize(kBeam);
        begin = end;
        cuts.insert(cuts.end(), next.begin(), next.end());
    }
    // walk back from the last pass
    std::vector<int> chain;
    for (int ci = last; ci >= 0; ci = cuts[ci].from) chain.push_back(ci);
    for (size_t i = chain.size(); i-- > 0;) {
        const Cut &c = cuts[chain[i]];
        PassPlan pp;
        pp.first = c.done;
        pp.end = i ? cuts[chain[i - 1]].done : S;
        if (i)
            pp.out.assign(cuts[chain[i - 1]].in.begin(), cuts[chain[i - 1]].in.end());
        else
            pp.out = o_final;
        Span sp;
        auto take = [&](uint64_t v) {
            if (sp.add((uint32_t)v)) pp.span.push_back(v);
        };
        for (uint32_t v : c.in) take(v);
        for (int q = pp.first; q < pp.end; ++q) take(U[q]);
        for (uint64_t v : pp.out) take(v);
        if (sp.dim > D) return -3;
        passes->push_back(pp);
    }
    return 0;
}

// Basis of the vectors v of F2^P with parity(f & v) = 0 for every f in fs.
std::vector<uint64_t> nullspace(const std::vector<uint64_t> &fs, int P)
{
    std::vector<uint64_t> rows = fs;
    std::vector<int> pivcol;
    size_t r = 0;
    for (int col = 0; col < P && r < rows.size(); ++col) {
        size_t sel = rows.size();
        for (size_t i = r; i < rows.size(); ++i)
            if ((rows[i] >> col) & 1ull) {
                sel = i;
                break;
            }
        if (sel == rows.size()) continue;
        std::swap(rows[r], rows[sel]);
        for (size_t i = 0; i < rows.size(); ++i)
            if (i != r && ((rows[i] >> col) & 1ull)) rows[i] ^= rows[r];
        pivcol.push_back(col);
        ++r;
    }
    std::vector<uint64_t> basis;
    for (int col = 0; col < P; ++col) {
        bool piv = false;
        for (int pc : pivcol) piv |= pc == col;
        if (piv) continue;
        uint64_t v = 1ull << col;
        for (size_t i = 0; i < r; ++i)
            if ((rows[i] >> col) & 1ull) v |= 1ull << pivcol[i];
        basis.push_back(v);
    }
    return basis;
}

// Lanes for a group: 5 vectors of the pool (a basis of K0) whose low bank bits
// (the 5 low slot bits for 4-byte keys, the 4 low ones of lanes 0-3 for 8-byte
// keys) are as independent as the pool allows: elimination on the bank bits, the
// vectors that keep one first.  With fewer, lanes share banks (results still
// exact).  K0 meets the group's register vectors in 0, so any choice is
// independent of those.
// Returns the bank bits lost (0: conflict-free), or -1 for a pool too small.
int pick_lanes(const std::vector<uint64_t> &pool, int e_log, std::vector<uint64_t> *lanes)
{
    if (pool.size() < 5) return -1;
    const int bank_bits = e_log == 2 ? 5 : 4;
    std::vector<uint64_t> v = pool;
    size_t r = 0;
    for (int b = 0; b < bank_bits; ++b) {
        size_t sel = r;
        while (sel < v.size() && !((v[sel] >> b) & 1ull)) ++sel;
        if (sel == v.size()) continue;
        std::swap(v[r], v[sel]);
        for (size_t i = 0; i < v.size(); ++i)
            if (i != r && ((v[i] >> b) & 1ull)) v[i] ^= v[r];
        ++r;
    }
    lanes->assign(v.begin(), v.begin() + 5);
    return bank_bits - (int)r;
}

// Where a pass's tables put virtual indices: a vector's slot part and a
// functional's parts on input positions and on slots.
struct SlotView {
    Coords lam;                 // in the tile's span
    uint32_t slot_pos[32] = {}; // input position of slot bit i, swizzle included
    const SlotMap *map;
    const f2::Mat *L, *L_inv;   // layout the pass reads

    SlotView(const SlotMap &m, const f2::Mat &l, const f2::Mat &l_inv)
        : map(&m), L(&l), L_inv(&l_inv)
    {
        for (int i = 0; i < m.P; ++i) {
            lam.add(m.lam[i], i);
            for (uint32_t s = m.swz(1u << i); s; s &= s - 1) slot_pos[i] ^= m.lam[__builtin_ctz(s)];
        }
    }
    bool slot(uint64_t v, uint32_t *out) const
    {
        uint32_t coords = 0;
        if (!lam.of((uint32_t)L->apply(v), &coords)) return false;
        *out = map->swz(coords);
        return true;
    }
    // g . x_virtual = g . (L^{-1} x_physical)
    uint64_t on_input(uint64_t g) const
    {
        uint64_t hin = 0;
        for (; g; g &= g - 1) hin ^= L_inv->r[__builtin_ctzll(g)];
        return hin;
    }
    uint64_t on_slots(uint64_t hin) const
    {
        uint64_t hs = 0;
        for (int i = 0; i < map->P; ++i)
            hs |= (uint64_t)__builtin_parityll(hin & slot_pos[i]) << i;
        return hs;
    }
};

// The coordinates of a group's stages [first, end): its distinct tests in the
// order of the network's index bits (test of bit i is the functional of virtual
// bit n - 1 - i), and each stage's code.  False if the stages do not make a
// group: more than R tests, tests that do not separate the span of the partner
// vectors, or a stage that is no run.
bool group_coords(const std::vector<uint64_t> &U, const std::vector<uint64_t> &G, int first,
                  int end, int R, std::vector<uint64_t> *tests, std::vector<uint8_t> *codes)
{
    tests->clear();
    codes->clear();
    if (end - first > kSortMaxGroupStages) return false;
    for (int s = first; s < end; ++s)
        if (std::find(tests->begin(), tests->end(), G[s]) == tests->end()) tests->push_back(G[s]);
    std::sort(tests->begin(), tests->end(), std::greater<uint64_t>());
    const int f = (int)tests->size();
    if (f > R) return false;
    Span W, C;  // partner vectors; the same in the tests' coordinates
    for (int s = first; s < end; ++s) {
        uint32_t m = 0;
        int own = -1;
        for (int t = 0; t < f; ++t) {
            m |= (uint32_t)__builtin_parityll((*tests)[t] & U[s]) << t;
            if ((*tests)[t] == G[s]) own = t;
        }
        if (!m || __builtin_ctz(m) != own) return false;
        const int l = 32 - __builtin_clz(m);
        if (m != ((1u << l) - (1u << own))) return false;
        codes->push_back((uint8_t)sort_stage_code(own, l));
        W.add((uint32_t)U[s]);
        C.add(m);
    }
    return W.dim == f && C.dim == f;
}

// Register groups of one pass and their thread mappings in physical slots (see
// sort_desc.h).  *conflicts receives the extra shared-memory wavefronts of a
// key's round trips, over the groups.
int build_groups(SortDesc *sd, const std::vector<uint64_t> &U, const std::vector<uint64_t> &G,
                 int first, int end, const SlotView &view, const PassDesc &desc, int e_log,
                 int *conflicts)
{
    const int P = view.map->P, R = (int)sd->reg_bits;
    const int round_bits = (int)sd->rounds - 1;
    const int warp_bits = P - R - 5 - round_bits;
    if (warp_bits < 0 || warp_bits > kSortMaxThreadBits - 5 || desc.n_cta > kSortMaxCtaBits)
        return -3;
    *conflicts = 0;
    int g = 0, s = first;
    std::vector<uint64_t> tests;
    std::vector<uint8_t> codes;
    while (s < end) {
        if (g >= kSortMaxGroups) return -3;
        SortGroup &Gr = sd->grp[g++];
        memset(&Gr, 0, sizeof(Gr));
        int e = s;
        for (int q = s + 1; q <= end && q - s <= kSortMaxGroupStages; ++q)
            if (group_coords(U, G, s, q, R, &tests, &codes)) e = q;
        if (e == s || !group_coords(U, G, s, e, R, &tests, &codes)) return -3;
        const int f = (int)tests.size();
        Gr.n_stage = (uint8_t)(e - s);
        for (int r = 0; r < f && e - s == f; ++r) {
            bool cycle = true;
            for (int q = 0; q < f; ++q) cycle &= codes[q] == sort_stage_code((r + q) % f, f);
            if (cycle) Gr.kind = (uint8_t)sort_cycle_kind(f, r);
        }
        if (f == R && e - s == R * (R + 1) / 2) {
            bool levels = true;
            for (int q = 0; q < e - s; ++q) levels &= codes[q] == q;
            if (levels) Gr.kind = (uint8_t)kSortLevelsKind;
        }
        for (int q = 0; q < e - s; ++q) Gr.code[q / 8] |= (uint32_t)codes[q] << (4 * (q % 8));
        // vectors dual to the tests in the span of the partner vectors: the
        // stages' vectors, eliminated on the tests
        std::vector<uint64_t> dual(f, 0);
        std::vector<std::pair<uint32_t, uint64_t>> rows;  // (coordinates, vector)
        for (int q = s; q < e; ++q) {
            uint32_t m = 0;
            for (int t = 0; t < f; ++t) m |= (uint32_t)__builtin_parityll(tests[t] & U[q]) << t;
            rows.push_back({m, U[q]});
        }
        for (int t = 0; t < f; ++t) {
            size_t sel = t;
            while (sel < rows.size() && !((rows[sel].first >> t) & 1u)) ++sel;
            if (sel == rows.size()) return -3;
            std::swap(rows[t], rows[sel]);
            for (size_t i = 0; i < rows.size(); ++i)
                if (i != (size_t)t && ((rows[i].first >> t) & 1u)) {
                    rows[i].first ^= rows[t].first;
                    rows[i].second ^= rows[t].second;
                }
        }
        std::vector<uint64_t> reg, fs, hin;
        for (int t = 0; t < f; ++t) {
            uint32_t sl = 0;
            if (!view.slot(rows[t].second, &sl)) return BMMC_ERR_INVALID;
            reg.push_back(sl);
            hin.push_back(view.on_input(tests[t]));
            fs.push_back(view.on_slots(hin.back()));
        }
        const std::vector<uint64_t> k0 = nullspace(fs, P);
        // lanes from K0, then unused register bits and warps from K0
        std::vector<uint64_t> lanes;
        const int lost = pick_lanes(k0, e_log, &lanes);
        if (lost < 0) return -3;
        *conflicts += (1 << lost) - 1;
        Span all;
        for (uint64_t v : reg) all.add((uint32_t)v);
        for (uint64_t v : lanes) all.add((uint32_t)v);
        std::vector<uint64_t> fill;
        for (uint64_t v : k0)
            if (all.add((uint32_t)v)) fill.push_back(v);
        if (all.dim != P || (int)fill.size() != R - f + warp_bits + round_bits)
            return -3;
        size_t fi = 0;
        while ((int)reg.size() < R) reg.push_back(fill[fi++]);
        for (int t = 0; t < R; ++t) Gr.reg[t] = (uint16_t)reg[t];
        for (int t = 0; t < 5; ++t) Gr.lane[t] = (uint16_t)lanes[t];
        for (int t = 0; t < warp_bits; ++t) Gr.warp[t] = (uint16_t)fill[fi++];
        if (round_bits) Gr.round = (uint16_t)fill[fi++];
        // a block whose input base has test t set finds register j's key at
        // the slot of j with bit t flipped
        for (uint32_t bb = 0; bb < desc.n_cta; ++bb)
            for (int t = 0; t < f; ++t)
                if (__builtin_parityll(hin[t] & desc.cta_in[bb])) Gr.cta[bb] ^= (uint16_t)reg[t];
        // the tests are 1 on their own register vector, 0 on everything else
        for (int t = 0; t < f; ++t) {
            for (int q = 0; q < R; ++q)
                if (__builtin_parityll(fs[t] & reg[q]) != (q == t)) return -3;
            for (uint64_t v : lanes)
                if (__builtin_parityll(fs[t] & v)) return -3;
            for (uint64_t v : fill)
                if (__builtin_parityll(fs[t] & v)) return -3;
        }
        s = e;
    }
    sd->n_group = (uint32_t)g;
    sd->n_stage = (uint32_t)(end - first);
    return 0;
}

// Register bits of a thread.  Few keys per thread shorten the chain of a block's
// instructions, many save round trips through shared memory: a whole sort in
// one block of 2^11 keys takes 7.2 us with 8 keys a thread and 7.7 with 16
// (int32; 9.8 and 11.3 int64), 2^18 keys in 2^12-key blocks 29.8 us with 16 and
// 34.4 with 32 (int32), and 2^13-key blocks take 32 for their 13 stages in three
// groups.  32 8-byte keys do not fit the registers.
int reg_bits(int e_log, int D)
{
    if (D <= 11) return 3;
    return e_log == 2 && D >= 13 ? 5 : 4;
}

// The chunk tables of a pass from those of a tiled pass (thread and loop bits of
// that kernel's blocks, in order, are this one's lane, warp and chunk bits).
int build_tile(SortDesc *sd, const PassDesc &d, int e_log)
{
    SortTile &t = sd->tile;
    const int w_log = 4 - e_log, P = (int)d.thread_bits + __builtin_ctz(d.loop) + w_log;
    const int key_bits = (int)(sd->reg_bits + sd->rounds - 1);
    const int T = P - key_bits;  // thread bits of this kernel
    const int chunk_bits = key_bits - w_log;
    if (T < 5 || T > kSortMaxThreadBits || chunk_bits > 4 || d.n_cta > kSortMaxCtaBits ||
        d.out_const || d.src_const)
        return -3;
    sd->n_cta = d.n_cta;
    sd->tile_bytes = d.smem_bytes;
    const uint32_t *thr[4] = {d.thr_in, d.thr_dst, d.thr_src, d.thr_out};
    const uint32_t *loop[4] = {d.loop_in, d.loop_dst, d.loop_src, d.loop_out};
    const uint32_t *cta[4] = {d.cta_in, nullptr, d.cta_src, d.cta_out};
    for (int f = 0; f < 4; ++f) {
        const int sh = f == kSortDst || f == kSortSrc ? e_log : 0;
        for (uint32_t i = 0; i < d.loop; ++i) {  // the loop tables are linear in i
            uint32_t x = 0;
            for (int b = 0; (1u << b) < d.loop; ++b)
                if ((i >> b) & 1u) x ^= loop[f][1u << b];
            if (x != loop[f][i]) return -3;
        }
        for (int b = 0; b < T + chunk_bits; ++b) {
            const uint32_t v = (b < (int)d.thread_bits ? thr[f][b]
                                                       : loop[f][1u << (b - (int)d.thread_bits)])
                               << sh;
            if (b < 5) t.lane[f][b] = v;
            else if (b < T) t.block[f][kSortMaxCtaBits + b - 5] = v;
            else t.chunk[f][b - T] = v;
        }
        for (uint32_t b = 0; cta[f] && b < d.n_cta; ++b) t.block[f][b] = cta[f][b] << sh;
    }
    for (int j = 0; j < 1 << w_log; ++j) t.elem[j] = d.elem_src[j] << e_log;
    for (uint32_t b = 0; b < d.thread_bits; ++b) {
        if (b >= 5 && d.thr_rot[b]) return -3;
        if (b < 5) t.any_rot |= t.rot[b] = d.thr_rot[b];
    }
    return 0;
}

// splitmix64, for the layout search
uint64_t mix64(uint64_t *s)
{
    uint64_t z = (*s += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// Bank bits that a layout L takes from the low tests of the next pass's stages:
// over runs of R stages, the low address bits (rows of L) that are
// combinations of each other and of the run's tests.
int bank_clashes(const PassPlan &next, const std::vector<uint64_t> &G, const f2::Mat &L, int e_log,
                 int R)
{
    const int bank_bits = e_log == 2 ? 5 : 4;
    int clashes = 0;
    for (int s = next.first; s < next.end; s += R) {
        Span sp;
        for (int q = s; q < next.end && q < s + R; ++q) sp.add((uint32_t)G[q]);
        for (int i = 0; i < bank_bits; ++i) clashes += !sp.add((uint32_t)L.r[i]);
    }
    return clashes;
}

// Tables of one pass from layout L_prev to layout L.  *score receives the extra
// shared-memory wavefronts of its register groups and stores, and whether output
// chunks are read rotated.
int derive_sort_pass(const PassPlan &pp, const std::vector<uint64_t> &U,
                     const std::vector<uint64_t> &G, const f2::Mat &L, const f2::Mat &L_prev,
                     const f2::Mat &L_prev_inv, int N, int e_log, int key, int k, int D,
                     SortDesc *sd_out, int *score)
{
    const f2::Mat T = f2::mul(L, L_prev_inv);
    // the block span in physical input positions, padded with unit
    // vectors up to D dimensions
    std::vector<uint64_t> W;
    Span span;
    for (uint64_t v : pp.span) {
        W.push_back(L_prev.apply(v));
        span.add((uint32_t)W.back());
    }
    for (int j = 0; j < N && span.dim < D; ++j)
        if (span.add(1u << j)) W.push_back(1ull << j);
    PassDesc desc;
    PassInfo info;
    SlotMap map;
    PlanOptions opt;
    opt.seg_bits = k;
    int rc = derive_pass_span(T, 0, N, e_log, opt, W.data(), (int)W.size(), &desc, &info, &map);
    if (rc) return rc;
    if (desc.naive || map.P != D) return BMMC_ERR_UNSUPPORTED;
    SortDesc &sd = *sd_out;
    memset(&sd, 0, sizeof(sd));
    sd.key = (uint32_t)key;
    sd.reg_bits = (uint32_t)reg_bits(e_log, D);
    sd.rounds = D - (int)sd.reg_bits > kSortMaxThreadBits ? 2 : 1;
    const SlotView view(map, L_prev, L_prev_inv);
    rc = build_tile(&sd, desc, e_log);
    if (rc) return rc;
    rc = build_groups(&sd, U, G, pp.first, pp.end, view, desc, e_log, score);
    if (rc) return rc;
    *score += info.wavefronts_store - info.ideal_store + (sd.tile.any_rot ? 1 : 0);
    return BMMC_OK;
}

}  // namespace

int plan_sort(bmmc_sort_plan_s *p, int n, int b, int key, int block_log2)
{
    const int e_log = (key >= BMMC_KEY_I32 && key <= BMMC_KEY_F32) ? 2 : 3;
    const int N = n + b;
    p->n = n;
    p->b = b;
    p->N = N;
    p->e_log = e_log;
    p->key = key;

    // The stage list in closed form: merge l = 1..n of the recursion has stages
    // i = 0..l-1, whose pairs differ in virtual bits n-1-i down to n-l and whose
    // low position has bit n-1-i clear; the keys end at their virtual positions.
    // (Composing schedule()'s matrices gives the same and took 10 of the 13 ms
    // that planning n = 20 took.)
    const int S = n * (n + 1) / 2;
    p->stages = S;
    std::vector<uint64_t> U, G;
    for (int l = 1; l <= n; ++l)
        for (int i = 0; i < l; ++i) {
            U.push_back((1ull << (n - i)) - (1ull << (n - l)));
            G.push_back(1ull << (n - 1 - i));
        }

    if (N <= kSortSmallMaxBits) {
        SortSmallDesc &d = p->sdesc;
        memset(&d, 0, sizeof(d));
        d.N = (uint32_t)N;
        d.key = (uint32_t)key;
        d.n_stage = (uint32_t)S;
        for (int s = 0; s < S; ++s) {
            d.u[s] = (uint32_t)U[s];
            d.g[s] = (uint32_t)G[s];
        }
        p->small = true;
        return BMMC_OK;
    }

    constexpr int kMinBlockBits = 12;
    // Segments of one 128-byte line: each of their bits costs a pass that reads
    // or writes them a dimension of its block.
    const int k = 7 - e_log;
    // Default block: more keys per block are fewer passes, fewer keys are more
    // blocks and more threads per key.  The lines are where the larger block
    // starts to win (GB300, us, 2^12 / 2^13 / 2^14 4-byte keys: n = 18 float32
    // 35 / 49 / 72, n = 20 66 / 64 / 95, n = 23 444 / 361 / 381, n = 24
    // 984 / 805 / 721; 2^12 / 2^13 8-byte keys: n = 22 int64 355 / 383,
    // n = 23 810 / 731).  They hold for rows too, also where a larger block would
    // keep whole rows and so be one pass (float32, 2^12 / 2^13 / 2^14 keys a
    // block: 64 rows of 2^13 18.6 / 24.8 / 43.1, 512 rows of 2^13 63.9 / 72.4 /
    // 73.8, 512 rows of 2^14 142 / 115 / 180; int64, 2^12 / 2^13: 512 rows of
    // 2^13 114 / 125, 1024 rows 227 / 215).
    int D = block_log2 ? block_log2 - e_log : kMinBlockBits;
    if (!block_log2)
        D += e_log == 2 ? (N >= 20) + (N >= 24) : (N >= 23);
    if (N <= kMinBlockBits) D = N;  // one block, whatever its size asked for
    else if (D < kMinBlockBits || D + e_log > 16) return BMMC_ERR_UNSUPPORTED;
    if (D > N) D = N;
    p->block_bits = D;

    std::vector<uint64_t> o_final;
    for (int j = 0; j < k; ++j) o_final.push_back(1ull << j);

    std::vector<PassPlan> plans;
    int rc = group_stages(U, k, D, o_final, &plans);
    if (rc) return rc;

    f2::Mat L_prev = f2::Mat::identity(N), L_prev_inv = f2::Mat::identity(N);
    uint64_t seed = 0xB17C0FFEEull;
    for (size_t pi = 0; pi < plans.size(); ++pi) {
        const PassPlan &pp = plans[pi];
        const bool last = pi + 1 == plans.size();
        // A layout between passes is free outside its segments: each other basis
        // vector may have any segment vector added.  That changes which
        // functionals the low address bits are, and so which keys share a
        // shared-memory bank: where a low test g_s of a register group is a
        // combination of the bank bits, no choice of lanes avoids conflicts.
        // The vectors as they come leave half of the tests so in the passes that
        // start at the network's first stages; a few tries of random additions
        // find layouts with none or nearly none (n = 24 float32, the 17 passes
        // before the kernel's present form: 1482 us with the vectors as they come,
        // 1161 us so).
        constexpr int kTries = 6;
        int best = -1;
        for (int attempt = 0; attempt < (last ? 1 : kTries) && best != 0; ++attempt) {
            f2::Mat L, L_inv;
            if (last) {
                L = L_inv = f2::Mat::identity(N);
            } else {
                std::vector<uint64_t> cols = pp.out;
                Span sp;
                for (uint64_t v : cols) sp.add((uint32_t)v);
                for (int j = 0; j < N; ++j)
                    if (sp.add(1u << j)) cols.push_back(1ull << j);
                if (attempt)
                    for (int j = k; j < N; ++j) cols[j] ^= xor_bits64(cols.data(), mix64(&seed) >> (64 - k));
                L_inv = from_columns(cols, N);
                if (!f2::inverse(L_inv, &L)) return BMMC_ERR_INVALID;
            }
            SortDesc sd;
            int score = 0;
            rc = derive_sort_pass(pp, U, G, L, L_prev, L_prev_inv, N, e_log, key, k, D,
                                  &sd, &score);
            if (rc) return rc;
            if (!last) score += bank_clashes(plans[pi + 1], G, L, e_log, reg_bits(e_log, D));
            if (best >= 0 && score >= best) continue;
            if (best >= 0) {
                p->pass.pop_back();
                p->layout.pop_back();
            }
            best = score;
            p->pass.push_back(sd);
            p->layout.push_back(L);
        }
        L_prev = p->layout.back();
        f2::inverse(L_prev, &L_prev_inv);
    }
    p->pass.front().first_pass = 1;
    p->pass.back().last_pass = 1;
    return BMMC_OK;
}

}  // namespace sortnet
}  // namespace bmmc

// ---------------------------------------------------------------------------
// Host emulation of the plan's tables (the index arithmetic of the kernels)
// ---------------------------------------------------------------------------

namespace bmmc {
namespace sortnet {

namespace {

// The comparator of Sec. 6.1 on raw key bits: a <= b under the key type.
bool keep_host(int key, uint64_t a, uint64_t b)
{
    switch (key) {
    case BMMC_KEY_I32: return (int32_t)(uint32_t)a <= (int32_t)(uint32_t)b;
    case BMMC_KEY_U32: return (uint32_t)a <= (uint32_t)b;
    case BMMC_KEY_F32: {
        float fa, fb;
        uint32_t ua = (uint32_t)a, ub = (uint32_t)b;
        memcpy(&fa, &ua, 4);
        memcpy(&fb, &ub, 4);
        return fa <= fb;
    }
    case BMMC_KEY_I64: return (int64_t)a <= (int64_t)b;
    case BMMC_KEY_U64: return a <= b;
    default: {
        double da, db;
        memcpy(&da, &a, 8);
        memcpy(&db, &b, 8);
        return da <= db;
    }
    }
}

uint64_t load_key(const uint8_t *base, uint64_t i, int e_log)
{
    uint64_t v = 0;
    memcpy(&v, base + (i << e_log), (size_t)1 << e_log);
    return v;
}

void store_key(uint8_t *base, uint64_t i, int e_log, uint64_t v)
{
    memcpy(base + (i << e_log), &v, (size_t)1 << e_log);
}

// Order the pair (lo_pos value a, hi_pos value b): a <= b keeps it.
void order_pair(int key, uint64_t *lo_val, uint64_t *hi_val)
{
    if (!keep_host(key, *lo_val, *hi_val)) {
        const uint64_t t = *lo_val;
        *lo_val = *hi_val;
        *hi_val = t;
    }
}

}  // namespace

int emulate(const bmmc_sort_plan_s *p, const void *in_v, void *out_v)
{
    const int e_log = p->e_log;
    const uint64_t count = 1ull << p->N;
    const uint8_t *in = static_cast<const uint8_t *>(in_v);
    uint8_t *out = static_cast<uint8_t *>(out_v);
    if (p->small) {
        const SortSmallDesc &d = p->sdesc;
        std::vector<uint64_t> a(count);
        for (uint64_t x = 0; x < count; ++x) a[x] = load_key(in, x, e_log);
        for (uint32_t s = 0; s < d.n_stage; ++s)
            for (uint64_t x = 0; x < count; ++x) {
                const uint64_t y = x ^ d.u[s];
                if (__builtin_parityll(x & d.g[s]) != 0) continue;  // x is the low one
                order_pair(p->key, &a[x], &a[y]);
            }
        for (uint64_t x = 0; x < count; ++x) store_key(out, x, e_log, a[x]);
        return 0;
    }
    std::vector<uint8_t> bufs[2];
    bufs[0].resize(count << e_log);
    bufs[1].resize(count << e_log);
    const uint8_t *src = in;
    for (size_t pi = 0; pi < p->pass.size(); ++pi) {
        const SortDesc &sd = p->pass[pi];
        const SortTile &t = sd.tile;
        uint8_t *dst = (pi + 1 == p->pass.size()) ? out : bufs[pi & 1].data();
        const uint32_t w = 1u << (4 - e_log);
        const uint32_t slots = sd.tile_bytes >> e_log;
        const uint32_t R = sd.reg_bits, E = 1u << R;
        const uint32_t keys = E * sd.rounds;  // of a thread
        const uint32_t threads = slots / keys;
        std::vector<uint64_t> sm(slots);
        // field f of (block, thread, chunk)
        auto field = [&](int f, uint64_t blk, uint32_t tid, uint32_t c) {
            uint32_t x = 0;
            for (uint32_t b = 0; b < sd.n_cta; ++b)
                if ((blk >> b) & 1ull) x ^= t.block[f][b];
            for (int b = 0; b < kSortMaxThreadBits - 5; ++b)
                if ((tid >> (5 + b)) & 1u) x ^= t.block[f][kSortMaxCtaBits + b];
            for (int b = 0; b < 5; ++b)
                if ((tid >> b) & 1u) x ^= t.lane[f][b];
            for (int b = 0; b < 4; ++b)
                if ((c >> b) & 1u) x ^= t.chunk[f][b];
            return x;
        };
        for (uint64_t blk = 0; blk < (1ull << sd.n_cta); ++blk) {
            // input chunks into their slots
            for (uint32_t tid = 0; tid < threads; ++tid)
                for (uint32_t c = 0; c < keys / w; ++c) {
                    const uint32_t g = field(kSortIn, blk, tid, c);
                    const uint32_t s = field(kSortDst, blk, tid, c) >> e_log;
                    for (uint32_t j = 0; j < w; ++j) sm.at(s + j) = load_key(src, g + j, e_log);
                }
            // comparator stages, group by group, as each thread runs them
            for (uint32_t gi = 0; gi < sd.n_group; ++gi) {
                const SortGroup &G = sd.grp[gi];
                uint32_t cta = 0;
                for (uint32_t bb = 0; bb < sd.n_cta; ++bb)
                    if ((blk >> bb) & 1ull) cta ^= G.cta[bb];
                uint32_t roff[1u << kSortMaxRegBits];
                for (uint32_t j = 0; j < E; ++j) {
                    roff[j] = 0;
                    for (uint32_t t = 0; t < R; ++t)
                        if ((j >> t) & 1u) roff[j] ^= G.reg[t];
                }
                for (uint32_t it = 0; it < threads * sd.rounds; ++it) {
                    const uint32_t tid = it % threads;
                    uint32_t q = cta ^ (it >= threads ? G.round : 0u);
                    for (int t = 0; t < 5; ++t)
                        if ((tid >> t) & 1u) q ^= G.lane[t];
                    for (int t = 0; t < kSortMaxThreadBits - 5; ++t)
                        if ((tid >> (5 + t)) & 1u) q ^= G.warp[t];
                    uint64_t v[1u << kSortMaxRegBits];
                    for (uint32_t j = 0; j < E; ++j) v[j] = sm.at(q ^ roff[j]);
                    for (uint32_t s = 0; s < G.n_stage; ++s) {
                        const uint32_t code = (G.code[s / 8] >> (4 * (s % 8))) & 15u;
                        uint32_t l = 1;
                        while ((uint32_t)sort_stage_code(0, (int)l + 1) <= code) ++l;
                        const uint32_t i = code - (uint32_t)sort_stage_code(0, (int)l);
                        const uint32_t m = (1u << l) - (1u << i);
                        for (uint32_t j = 0; j < E; ++j)
                            if (!((j >> i) & 1u)) order_pair(p->key, &v[j], &v[j ^ m]);
                    }
                    for (uint32_t j = 0; j < E; ++j) sm.at(q ^ roff[j]) = v[j];
                }
            }
            // output chunks from their slots
            for (uint32_t tid = 0; tid < threads; ++tid) {
                uint32_t rot = 0;
                for (int b = 0; b < 5; ++b)
                    if ((tid >> b) & 1u) rot ^= t.rot[b];
                for (uint32_t c = 0; c < keys / w; ++c) {
                    const uint32_t s = field(kSortSrc, blk, tid, c) ^ t.elem[rot];
                    const uint32_t o = field(kSortOut, blk, tid, c);
                    for (uint32_t j = 0; j < w; ++j)
                        store_key(dst, o + (j ^ rot), e_log, sm.at((s ^ t.elem[j]) >> e_log));
                }
            }
        }
        src = dst;
    }
    return 0;
}

}  // namespace sortnet
}  // namespace bmmc

// ---------------------------------------------------------------------------
// C ABI (include/bmmc_sort.h)
// ---------------------------------------------------------------------------

namespace bmmc {
cudaError_t launch_sort_pass(const SortDesc &sd, const void *in, void *out, cudaStream_t s);
cudaError_t launch_sort_small(const SortSmallDesc &d, int e_log, const void *in, void *out,
                              cudaStream_t s);
}  // namespace bmmc

namespace {

// Passes alternate between the output and a workspace; one alone writes the
// output.
bool needs_workspace(const bmmc_sort_plan_s *p) { return p->pass.size() > 1; }

bool overlaps(const void *a, const void *b, uint64_t bytes)
{
    const uintptr_t x = (uintptr_t)a, y = (uintptr_t)b;
    return x < y + bytes && y < x + bytes;
}

}  // namespace

extern "C" {

int bmmc_sort_plan_create(bmmc_sort_plan *out, int n, int b, int key_type,
                          const bmmc_sort_options *opts)
{
    using namespace bmmc;
    if (!out) return BMMC_ERR_INVALID;
    *out = nullptr;
    if (n < 1 || n > 30 || b < 0 || n + b > 32) return BMMC_ERR_INVALID;
    if (key_type < BMMC_KEY_I32 || key_type > BMMC_KEY_F64) return BMMC_ERR_UNSUPPORTED;
    int block_log2 = 0;
    if (opts) {
        for (int r : opts->reserved)
            if (r) return BMMC_ERR_UNSUPPORTED;
        block_log2 = opts->block_log2;
        if (opts->compare_code < 0 || opts->compare_code > 2) return BMMC_ERR_UNSUPPORTED;
        if (block_log2 && (block_log2 < 12 || block_log2 > 16)) return BMMC_ERR_UNSUPPORTED;
    }
    return guarded([&] {
        bmmc_sort_plan_s *p = new bmmc_sort_plan_s();
        const int rc = sortnet::plan_sort(p, n, b, key_type, block_log2);
        if (rc) {
            delete p;
            return rc;
        }
        *out = p;
        return (int)BMMC_OK;
    });
}

void bmmc_sort_plan_destroy(bmmc_sort_plan p) { delete p; }

int bmmc_sort_plan_num_passes(bmmc_sort_plan p)
{
    if (!p) return BMMC_ERR_INVALID;
    return p->small ? 1 : (int)p->pass.size();
}

size_t bmmc_sort_workspace_bytes(bmmc_sort_plan p)
{
    if (!p || !needs_workspace(p)) return 0;
    return ((size_t)1 << p->N) << p->e_log;
}

int bmmc_sort_execute(bmmc_sort_plan p, const void *in, void *out, void *ws,
                      bmmc_stream_t stream)
{
    using namespace bmmc;
    if (!p || !in || !out) return BMMC_ERR_INVALID;
    const uint64_t bytes = (1ull << p->N) << p->e_log;
    if (((uintptr_t)in | (uintptr_t)out | (uintptr_t)ws) & 15u) return BMMC_ERR_ALIGN;
    if (overlaps(in, out, bytes)) return BMMC_ERR_ALIAS;
    cudaStream_t s = (cudaStream_t)stream;
    if (p->small) {
        if (debug_fail_launch()) return BMMC_ERR_CUDA;
        return launch_sort_small(p->sdesc, p->e_log, in, out, s) == cudaSuccess ? BMMC_OK
                                                                                 : BMMC_ERR_CUDA;
    }
    const size_t np = p->pass.size();
    if (needs_workspace(p)) {
        if (!ws) return BMMC_ERR_INVALID;
        if (overlaps(ws, in, bytes) || overlaps(ws, out, bytes)) return BMMC_ERR_ALIAS;
    }
    const void *src = in;
    for (size_t i = 0; i < np; ++i) {
        // the last pass writes out; earlier ones alternate so that they never
        // read and write one buffer
        void *dst = ((np - 1 - i) % 2 == 0) ? out : ws;
        if (debug_fail_launch()) return BMMC_ERR_CUDA;
        if (launch_sort_pass(p->pass[i], src, dst, s) != cudaSuccess)
            return BMMC_ERR_CUDA;
        src = dst;
    }
    return BMMC_OK;
}

int bmmc_sort_plan_emulate(bmmc_sort_plan p, const void *in, void *out)
{
    if (!p || !in || !out) return BMMC_ERR_INVALID;
    return bmmc::guarded([&] { return bmmc::sortnet::emulate(p, in, out); });
}

int bmmc_sort_plan_describe(bmmc_sort_plan p, char *buf, size_t len)
{
    if (!p) return BMMC_ERR_INVALID;
    return bmmc::guarded([&] {
        std::string s = "{\"n\": " + std::to_string(p->n) + ", \"b\": " + std::to_string(p->b) +
                        ", \"key_bytes\": " + std::to_string(1 << p->e_log) +
                        ", \"stages\": " + std::to_string(p->stages) +
                        ", \"one_block\": " + (p->small || p->pass[0].n_cta == 0 ? "true" : "false") +
                        ", \"block_keys_log2\": " + std::to_string(p->block_bits) +
                        ", \"passes\": [";
        for (size_t i = 0; i < p->pass.size(); ++i) {
            char tmp[160];
            snprintf(tmp, sizeof(tmp), "%s{\"stages\": %u, \"groups\": %u, \"blocks\": %llu}",
                     i ? ", " : "", p->pass[i].n_stage, p->pass[i].n_group,
                     (unsigned long long)(1ull << p->pass[i].n_cta));
            s += tmp;
        }
        s += "]}";
        if (buf && len) {
            const size_t cpy = s.size() < len - 1 ? s.size() : len - 1;
            memcpy(buf, s.data(), cpy);
            buf[cpy] = 0;
        }
        return (int)s.size();
    });
}

}  // extern "C"
