// qieo_column.cuh -- the column form of a run (rule R1).
//
// Under rule R1 every qubit of a column (gene) takes the same step, toward the elite's allele
// of that gene, whatever its own allele. A population that starts with equal rows (generation
// 0: every qubit at pi/4) therefore keeps equal rows for ever: one row of angle indices, not
// np of them, is the population's state. A run in this form
//   - keeps one row of angle indices and applies CIP once per gene instead of once per qubit;
//   - holds a gene's observation threshold in a register for all rows of a segment, so that a
//     row's pass is the Philox draws, a compare and an item add per gene, with no state read
//     or written, no table lookup and no rotation;
//   - drops genes that have reached a bound: their allele is the same in every row from then
//     on (T = 0 or 2^32, and the elite carries that allele too, so the angle never leaves the
//     bound). The Philox call is the unit, 4 genes (a "quad"): the list of the quads that still
//     draw is rebuilt when enough have become fixed, and the item sums of the dropped ones are
//     one pair of constants;
//   - stores no alleles while it runs: the elite's alleles, which CIP and the best record need,
//     are drawn again from its counters (two Philox calls per thread and segment), and the allele
//     plane of the last generation is written once at the end of the run (column_plane_kernel).
// The results are those of the row-by-row forms, which the instance keeps for rule R2, for
// states whose rows differ (a checkpoint may hold one) and for the forms that flags ask for.
//
// A run is one cooperative launch, or two (column_run_kernel while the blocks' shares are long,
// column_small_kernel after it), then column_plane_kernel and column_end_kernel; a run of a few
// generations is plain launches of column_observe_kernel and column_step_kernel. What each measured
// against the form it replaces stands at the kernel.
#pragma once

#include "qieo_kernels.cuh"

namespace qieo {

// Counts of a quad list and the item sums of the quads that are not on it.
struct ColSlot {
    unsigned long long fw, fv;    // sums over the dropped quads' genes at theta = pi/2
    unsigned int nv, ns;          // whole vectors (both quads draw), single quads
    unsigned int pad[2];
};

// What the blocks of a generation tell one another: the elite key, the blocks that have arrived, the
// list's quads that were fixed in the generation before. (A post is one 16-byte store, read
// by one 16-byte load.)
struct __align__(16) ColSync {
    unsigned long long key;
    unsigned int arrived, drops;
};

// ctl words (device)
constexpr int kCtlRebuild = 0;    // the run started with quads on its list: it is built again
constexpr int kCtlRan = 1;        // the run executed generations
constexpr int kCtlFirst = 2;      // its first generation
constexpr int kCtlLast = 3;       // its last one
constexpr int kCtlEarly = 4;      // 1: it stopped before the last generation asked for
constexpr int kCtlTicket = 5;     // column_end_kernel: blocks done
constexpr int kCtlRebuilt = 6;    // blocks that have arrived at list rebuilds of the run
constexpr int kCtlPhase = 7;      // what column_run_kernel left: 0 nothing, 1 the rest of the run (the
                                  // words below and ColParams::rest), 2 no generation
constexpr int kCtlGen = 8;        // ... the generations done
constexpr int kCtlCur = 9;        // ... the list
constexpr int kCtlRebuilds = 10;  // ... the rebuilds
constexpr int kCtlElite = 11;     // ... the last elite
constexpr int kCtlImproved = 12;  // ... whether it improved the best

constexpr int kCtlDiffer = 13;    // column_compare_kernel: a row of the full state differs from row 0

constexpr int kColPosted = 64;              // most blocks that meet through posts

struct ColParams {
    uint2 *canon;                 // [2 svec] the state between runs: 4 halfwords (4n) a quad
    uint2 *rows;                  // [2][2 svec] the state generation t observes in parity t & 1 (the
                                  // quads that were on the list of generation t or before)
    int32_t *lists;               // [2][2 svec] vectors at [0, svec), single quads at [svec, 2 svec)
    int2 *best_nib;               // [2 svec] (generation, alleles) of the last best row recorded
    ColSync *sync;                // [4] generation t in t & 3 (arrived: blocks)
    unsigned int *qctr;           // [4][kColQueues] next rows of a tile, generation t in t & 3
    ColSync *post;                // [2][kColPosted] a block's generation t in parity t & 1 (arrived: t + 1)
    ColSlot *slot;                // [3] the counts of a rebuilt list, rebuild r of the run in r % 3
    ColSlot *head;                // the list at the start of a run (in list 0)
    ColSlot *rest;                // the list and the dropped quads' sums at the hand-over
    int32_t *ctl;                 // [16]
    int64_t *run_best;            // [2] runs of column_observe_kernel: best fitness before generation t in t & 1
    uint32_t one;                 // 1 (see mad_add)
    int32_t sum_bits;             // kForm 1: a row's weights, its values and its tiles' count share a word of
                                  // acc, the sums in this many bits each (0: a word each and cnt)
};

__device__ __forceinline__ uint2 *column_parity(const ColParams &c, int32_t svec, int32_t t)
{
    return c.rows + (size_t)(t & 1) * 2u * (size_t)svec;
}

__device__ __forceinline__ int32_t *column_list(const ColParams &c, int32_t svec, int which)
{
    return c.lists + (size_t)which * 2u * (size_t)svec;
}

constexpr int kColRows = 256;               // rows summed in shared memory at once (one a thread)
constexpr int kColLocalPasses = 2;          // at most this many passes: one block that meets nobody
constexpr int kColQueueShare = 32;          // passes per block from which a tile's rows are queued
constexpr int kColQueues = 1024;            // tiles that can have a queue
constexpr int kColSmallShare = 4;           // fewer passes per block: column_small_kernel
constexpr int kColSmallTiles = 128;         // most tiles of a small share (fewer than the blocks)
constexpr int kColSmallRows = 512;          // column_small_kernel: rows summed in shared memory at once

// The two quads of one thread and what its rows share.
template <int kForm>
struct ColItem {
    int32_t qa, qb;               // quad indices, -1: none
    bool whole;                   // qa, qb are the two quads of one vector
    bool none;                    // no lane of the warp has a quad
    uint2 sa, sb;                 // their angle indices (4n)
    uint32_t wv[8];               // kForm 0: items (v << 16 | w); else weights
    int32_t v[kForm == 0 ? 1 : 8];
};

// How a generation's work is cut, from the list's counts (the same in every block).
struct ColGeom {
    int items, ntile, width;      // thread items, tiles, items per tile
    int lanes, warps, rpp;        // a tile's threads; rows per pass (a power of two)
    int nu;                       // passes per tile
    int nb;                       // blocks that take part
    bool small;                   // column_small_kernel's
};

__device__ __forceinline__ ColGeom column_geometry(uint32_t nv, uint32_t ns, int np, int grid)
{
    ColGeom m;
    m.items = (int)(nv + (ns + 1u) / 2u);
    m.ntile = 1;
    m.width = m.items;
    m.lanes = 32;
    m.warps = 8;
    if (m.items > kThreads) {
        m.ntile = (m.items + kThreads - 1) / kThreads;
        m.width = (m.items + m.ntile - 1) / m.ntile;
    } else {
        int tile = 1;
        while (tile < m.items) tile <<= 1;
        m.lanes = min(tile, 32);
        m.warps = max(tile >> 5, 1);
    }
    m.rpp = kThreads / (m.lanes * m.warps);
    m.nu = (np + m.rpp - 1) / m.rpp;
    const uint32_t units = (uint32_t)m.ntile * (uint32_t)m.nu;    // (the population fits memory)
    m.nb = (int)max(min((uint32_t)grid, units), 1u);
    m.small = m.ntile <= kColSmallTiles && units < (uint32_t)kColSmallShare * (uint32_t)grid;
    return m;
}

// The cut of column_run_kernel: every block has a home tile, whose item it keeps in registers
// from generation to generation, and a tile's rows are shared by the same number of blocks
// (`group`); the tiles are made a little narrower so that the blocks divide evenly among them (a
// warp whose lanes all lie past the tile's width does no work). With more tiles than blocks
// every block has `turns` tiles and all their rows.
//
// The blocks that share an SM do not get equal issue slots, so long shares are taken from the
// tile's counter in pieces of decreasing size: round l of one piece a block takes half of what
// is left. (A queue of segments over all tiles, the form before, made a block load and
// rotate an item for every segment: about 400 instructions for 19 rows on average.)
struct ColHome {
    int home, part, group, turns; // first tile, index in the group, blocks per tile, tiles per block
    int stride;                   // distance of a block's tiles
    int share;                    // passes per block
    bool queued;                  // its rows come from the tile's counter
    int round, start, size;       // the round of the last piece, its first pass and its pieces' passes
};

__device__ __forceinline__ ColHome column_home(ColGeom &m, int block, int grid)
{
    ColHome h;
    h.turns = 1;
    if (m.ntile <= grid) {
        h.group = grid / m.ntile;
        if (m.ntile > 1) m.ntile = grid / h.group;
        h.stride = m.ntile;
    } else {
        h.group = 1;
        h.turns = (m.ntile + grid - 1) / grid;
        m.ntile = h.turns * grid;
        h.stride = grid;
    }
    if (m.ntile > 1) m.width = (m.items + m.ntile - 1) / m.ntile;
    h.group = min(h.group, m.nu);
    m.nb = h.stride * h.group;
    h.home = (int)((unsigned int)block % (unsigned int)h.stride);
    h.part = (int)((unsigned int)block / (unsigned int)h.stride);
    h.share = m.nu / h.group;
    h.queued = h.share >= kColQueueShare && h.group > 1;
    return h;
}

// Passes [ua, ub) of piece i of a tile (ua >= nu: none); i grows from call to call of a generation,
// from i < group.
__device__ __forceinline__ void column_piece(const ColGeom &m, ColHome &h, int i, int &ua, int &ub)
{
    if (!h.queued) {
        ua = (int)((int64_t)m.nu * i / h.group);
        ub = (int)((int64_t)m.nu * (i + 1) / h.group);
        return;
    }
    if (i < h.group) {
        h.round = h.start = 0;
        h.size = h.share / 2;
    }
    while (i - h.round >= h.group) {
        h.round += h.group;
        h.start += h.group * h.size;
        h.size = max(h.size / 2, 2);
    }
    ua = h.start + (i - h.round) * h.size;
    ub = min(m.nu, ua + h.size);
}

__device__ __forceinline__ bool quad_fixed(uint2 s, uint32_t off_top)
{
    const uint32_t h[4] = {s.x & 0xffffu, s.x >> 16, s.y & 0xffffu, s.y >> 16};
    bool f = true;
#pragma unroll
    for (int i = 0; i < 4; ++i) f = f && (h[i] == 0u || h[i] == off_top);
    return f;
}

// Alleles (bit i = gene i) of a quad observed with draw d.
__device__ __forceinline__ uint32_t observe_quad(const Draw4 &d, uint2 s, const unsigned char *thr_bytes,
                                                 uint32_t off_top)
{
    const uint32_t h[4] = {s.x & 0xffffu, s.x >> 16, s.y & 0xffffu, s.y >> 16};
    const uint32_t u[4] = {d.a, d.b, d.c, d.d};
    uint32_t x = 0u;
#pragma unroll
    for (int i = 0; i < 4; ++i)
        if (u[i] < *reinterpret_cast<const uint32_t *>(thr_bytes + h[i]) || h[i] == off_top) x |= 1u << i;
    return x;
}

// Alleles of a quad whose genes all sit at a bound.
__device__ __forceinline__ uint32_t quad_sides(uint2 s)
{
    return ((s.x & 0xffffu) ? 1u : 0u) | ((s.x >> 16) ? 2u : 0u) | ((s.y & 0xffffu) ? 4u : 0u) | ((s.y >> 16) ? 8u : 0u);
}

// One CIP step of a quad toward alleles x.
__device__ __forceinline__ uint2 step_quad(uint2 s, uint32_t x, uint32_t k8)
{
    return make_uint2(rotate_pair_signed(s.x, signed_step(delta_pair(x & 3u, 3u)), k8),
                      rotate_pair_signed(s.y, signed_step(delta_pair(x >> 2, 3u)), k8));
}

template <int kForm>
__device__ __forceinline__ void column_load(const GenParams &p, ColItem<kForm> &it, const uint2 *state);

// Item i of a list (i < items): its quads, their items and angle indices from `state`.
template <int kForm>
__device__ __forceinline__ void column_item(const GenParams &p, ColItem<kForm> &it, const int32_t *list, uint32_t nv,
                                            uint32_t ns, int i, bool active, const uint2 *state)
{
    it.qa = it.qb = -1;
    it.whole = false;
    if (active) {
        if ((uint32_t)i < nv) {
            const int32_t vec = __ldcg(list + i);
            it.qa = 2 * vec;
            it.qb = 2 * vec + 1;
            it.whole = true;
        } else {
            const uint32_t j = 2u * ((uint32_t)i - nv);
            it.qa = __ldcg(list + p.svec + j);
            if (j + 1u < ns) it.qb = __ldcg(list + p.svec + j + 1);
        }
    }
    column_load<kForm>(p, it, state);
}

// The items and angle indices of a thread's quads (whole warps).
template <int kForm>
__device__ __forceinline__ void column_load(const GenParams &p, ColItem<kForm> &it, const uint2 *state)
{
    it.none = !__any_sync(0xffffffffu, it.qa >= 0);
    it.sa = it.sb = make_uint2(0u, 0u);
    if (it.qa >= 0) it.sa = __ldcg(state + it.qa);
    if (it.qb >= 0) it.sb = __ldcg(state + it.qb);
    const uint4 z = make_uint4(0u, 0u, 0u, 0u);
    if constexpr (kForm == 0) {
        const uint4 a = it.qa >= 0 ? __ldg(p.items_narrow + it.qa) : z, b = it.qb >= 0 ? __ldg(p.items_narrow + it.qb) : z;
        it.wv[0] = a.x; it.wv[1] = a.y; it.wv[2] = a.z; it.wv[3] = a.w;
        it.wv[4] = b.x; it.wv[5] = b.y; it.wv[6] = b.z; it.wv[7] = b.w;
    } else {
        const int4 zi = make_int4(0, 0, 0, 0);
        const int4 a = it.qa >= 0 ? __ldg(p.w4 + it.qa) : zi, b = it.qb >= 0 ? __ldg(p.w4 + it.qb) : zi;
        const int4 d = it.qa >= 0 ? __ldg(p.v4 + it.qa) : zi, e = it.qb >= 0 ? __ldg(p.v4 + it.qb) : zi;
        it.wv[0] = (uint32_t)a.x; it.wv[1] = (uint32_t)a.y; it.wv[2] = (uint32_t)a.z; it.wv[3] = (uint32_t)a.w;
        it.wv[4] = (uint32_t)b.x; it.wv[5] = (uint32_t)b.y; it.wv[6] = (uint32_t)b.z; it.wv[7] = (uint32_t)b.w;
        it.v[0] = d.x; it.v[1] = d.y; it.v[2] = d.z; it.v[3] = d.w;
        it.v[4] = e.x; it.v[5] = e.y; it.v[6] = e.z; it.v[7] = e.w;
    }
}

// Philox4x32-10 of counter (q, row, t, 0) for a fixed q and t over many rows. Of the first three
// rounds only two products depend on the row: M0 n0 of the second, the same for every q
// (row_product), and M1 c2 of the third; the rest is four words per quad (quad_words), with the
// round keys folded in.
struct QuadWords {
    uint32_t b, d, h, l;          // second round's n2 without the row's part; third round: n0's and n2's xor, c3
};

__device__ __forceinline__ QuadWords quad_words(const GenParams &p, uint32_t q, uint32_t t)
{
    const uint64_t p0 = (uint64_t)kPhiloxM0 * q;
    const uint64_t p1 = (uint64_t)kPhiloxM1 * ((uint32_t)(p0 >> 32) ^ p.rk1[0]);
    const uint32_t lo_t = (uint32_t)((uint64_t)kPhiloxM1 * t);
    const uint64_t p2 = (uint64_t)kPhiloxM0 * ((uint32_t)(p1 >> 32) ^ lo_t ^ p.rk0[1]);
    QuadWords w = {(uint32_t)p0 ^ p.rk1[1], (uint32_t)p1 ^ p.rk0[2], (uint32_t)(p2 >> 32) ^ p.rk1[2], (uint32_t)p2};
    // (kept in registers: the compiler otherwise computes them again for every row)
    asm volatile("" : "+r"(w.b), "+r"(w.d), "+r"(w.h), "+r"(w.l));
    return w;
}

// The round keys of the rest, and of the row's product.
struct RowKeys {
    uint32_t hi;                  // first round: the high word of M1 t, with the key
    uint32_t k0[7], k1[7];        // rounds 3 .. 9
};

__device__ __forceinline__ RowKeys row_keys(const GenParams &p, uint32_t t)
{
    RowKeys k;
    k.hi = (uint32_t)(((uint64_t)kPhiloxM1 * t) >> 32) ^ p.rk0[0];
#pragma unroll
    for (int r = 0; r < 7; ++r) {
        k.k0[r] = p.rk0[r + 3];
        k.k1[r] = p.rk1[r + 3];
    }
    return k;
}

__device__ __forceinline__ uint64_t row_product(const RowKeys &k, uint32_t row) { return (uint64_t)kPhiloxM0 * (k.hi ^ row); }

__device__ __forceinline__ Draw4 quad_draw(const RowKeys &k, const QuadWords &w, uint64_t z)
{
    const uint64_t p1 = (uint64_t)kPhiloxM1 * ((uint32_t)(z >> 32) ^ w.b);
    uint32_t c0 = (uint32_t)(p1 >> 32) ^ w.d, c1 = (uint32_t)p1, c2 = (uint32_t)z ^ w.h, c3 = w.l;
#pragma unroll
    for (int r = 3; r < 10; ++r) {
        const uint64_t a = (uint64_t)kPhiloxM0 * (uint64_t)c0;
        const uint64_t b = (uint64_t)kPhiloxM1 * (uint64_t)c2;
        const uint32_t n0 = (uint32_t)(b >> 32) ^ c1 ^ k.k0[r - 3];
        const uint32_t n2 = (uint32_t)(a >> 32) ^ c3 ^ k.k1[r - 3];
        c1 = (uint32_t)b;
        c3 = (uint32_t)a;
        c0 = n0;
        c2 = n2;
    }
    return {c0, c1, c2, c3};
}

// Sum over the warp of a 64-bit value of magnitude below 2^36, as two 32-bit reductions: 21
// low bits (32 of them stay below 2^26) and the signed rest.
__device__ __forceinline__ int64_t warp_sum64(int64_t s)
{
    const uint32_t lo = __reduce_add_sync(0xffffffffu, (uint32_t)s & 0x1fffffu);
    const int32_t hi = __reduce_add_sync(0xffffffffu, (int32_t)(s >> 21));
    return ((int64_t)hi << 21) + (int64_t)lo;
}

// The sums of one row over a thread's 8 genes: kForm 0 packed (v << 16 | w); 1 and 2 w and v.
template <int kForm>
struct ColSum {
    uint32_t a;                   // kForm 0: packed; 1: w
    uint32_t b;                   // kForm 1: v
    int64_t w, v;                 // kForm 2
};

// The thresholds of a thread's 8 genes, and the mask and the item sums of those at theta = pi/2. A gene at a bound
// gets the threshold 0 (never observed by compare): at theta = 0 that is its allele; at pi/2
// (T = 2^32, which 32 bits do not hold) its items are in the base sums.
template <int kForm>
__device__ __forceinline__ void column_thresholds(const ColItem<kForm> &it, const unsigned char *thr_bytes,
                                                  uint32_t off_top, uint32_t (&T)[8], uint32_t &top, ColSum<kForm> &base)
{
    top = 0u;
    const uint32_t sp[4] = {it.sa.x, it.sa.y, it.sb.x, it.sb.y};
    base.a = base.b = 0u;
    base.w = base.v = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const uint32_t off = (i & 1) ? (sp[i >> 1] >> 16) : (sp[i >> 1] & 0xffffu);
        T[i] = *reinterpret_cast<const uint32_t *>(thr_bytes + off);      // 0 at both bounds
        if (off == off_top) {
            top |= 1u << i;
            if constexpr (kForm == 0) base.a += it.wv[i];
            else if constexpr (kForm == 1) {
                base.a += it.wv[i];
                base.b += (uint32_t)it.v[i];
            } else {
                base.w += (int32_t)it.wv[i];
                base.v += it.v[i];
            }
        }
    }
}

// a + x as a multiply-add by a word that holds 1: the compiler would make a plain add of it, on the
// ALU pipe, which the compares and Philox's xors keep busy; the multiply pipe has room (a pass of
// the loop in column_rows: 188 -> 179 cycles per 256 genes).
__device__ __forceinline__ void mad_add(uint32_t &a, uint32_t x, uint32_t one)
{
    asm("mad.lo.u32 %0, %1, %2, %0;" : "+r"(a) : "r"(x), "r"(one));
}

template <int kForm>
__device__ __forceinline__ ColSum<kForm> column_sum(const ColItem<kForm> &it, const uint32_t (&T)[8],
                                                    const ColSum<kForm> &base, const uint32_t (&u)[8], uint32_t one)
{
    ColSum<kForm> s = base;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        if (u[i] < T[i]) {
            if constexpr (kForm == 0) mad_add(s.a, it.wv[i], one);
            else if constexpr (kForm == 1) {
                s.a += it.wv[i];
                mad_add(s.b, (uint32_t)it.v[i], one);
            } else {
                s.w += (int32_t)it.wv[i];
                s.v += it.v[i];
            }
        }
    }
    return s;
}

template <int kForm>
__device__ __forceinline__ ColSum<kForm> column_row(const RowKeys &k, uint32_t one, const ColItem<kForm> &it, const uint32_t (&T)[8],
                                                    const ColSum<kForm> &base, const QuadWords &wa,
                                                    const QuadWords &wb, uint32_t row)
{
    const uint64_t z = row_product(k, row);
    const Draw4 r0 = quad_draw(k, wa, z), r1 = quad_draw(k, wb, z);
    const uint32_t u[8] = {r0.a, r0.b, r0.c, r0.d, r1.a, r1.b, r1.c, r1.d};
    return column_sum<kForm>(it, T, base, u, one);
}

// Adds lane sums of a row (whole warp) into one lane's keeper; see column_rows.
template <int kForm>
__device__ __forceinline__ ColSum<kForm> column_warp_sum(const ColSum<kForm> &s)
{
    ColSum<kForm> r = s;
    if constexpr (kForm == 0) r.a = __reduce_add_sync(0xffffffffu, s.a);
    else if constexpr (kForm == 1) {
        r.a = __reduce_add_sync(0xffffffffu, s.a);
        r.b = __reduce_add_sync(0xffffffffu, s.b);
    } else {
        r.w = warp_sum64(s.w);
        r.v = warp_sum64(s.v);
    }
    return r;
}

// Adds a row's partial sums to its shared accumulators.
template <int kForm>
__device__ __forceinline__ void column_add(const ColSum<kForm> &s, int row, uint32_t *s_acc32, unsigned long long *s_acc64)
{
    if constexpr (kForm == 0) {
        atomicAdd(s_acc32 + 2 * row, s.a & 0xffffu);
        atomicAdd(s_acc32 + 2 * row + 1, s.a >> 16);
    } else if constexpr (kForm == 1) {
        atomicAdd(s_acc32 + 2 * row, s.a);
        atomicAdd(s_acc32 + 2 * row + 1, s.b);
    } else {
        atomicAdd(s_acc64 + 2 * row, (unsigned long long)s.w);
        atomicAdd(s_acc64 + 2 * row + 1, (unsigned long long)s.v);
    }
}

// Adds the block's sums of row c (its accumulator i, left 0) to the row; the row's elite key if
// that completes it, else 0.
template <int kForm>
__device__ __forceinline__ unsigned long long column_row_done(const GenParams &p, int sum_bits, int ntile, int c, int i,
                                                              const int64_t *s_fix, uint32_t *s_acc32,
                                                              unsigned long long *s_acc64)
{
    int64_t sw, sv;
    if constexpr (kForm == 2) {
        sw = (int64_t)s_acc64[2 * i];
        sv = (int64_t)s_acc64[2 * i + 1];
        s_acc64[2 * i] = s_acc64[2 * i + 1] = 0ull;
    } else {
        sw = (int64_t)s_acc32[2 * i];
        sv = (int64_t)s_acc32[2 * i + 1];
        s_acc32[2 * i] = s_acc32[2 * i + 1] = 0u;
    }
    bool done = true;
    if (ntile > 1) {
        // One word where the sums leave room for the count: its atomic both adds and tells who completed
        // the row. (Two words and a counter are three accesses one after another in every
        // generation: 67 rows of 2,249 genes, 33 generations: 190 us with the reset and the wait, 113 with one word.)
        const int bits = kForm == 0 ? 26 : kForm == 1 ? sum_bits : 0;
        if (bits != 0) {
            const unsigned long long add = (1ull << (2 * bits)) | ((unsigned long long)sv << bits) | (unsigned long long)sw;
            const unsigned long long full = atomicAdd(p.acc + c, add) + add, mask = (1ull << bits) - 1ull;
            done = (int)(full >> (2 * bits)) == ntile;
            if (done) {
                p.acc[c] = 0ull;
                sw = (int64_t)(full & mask);
                sv = (int64_t)((full >> bits) & mask);
            }
        } else {
            atomicAdd(p.acc + 2 * (size_t)c, (unsigned long long)sw);
            atomicAdd(p.acc + 2 * (size_t)c + 1, (unsigned long long)sv);
            done = (int)atom_add_acq_rel(p.cnt + c, 1u) == ntile - 1;
            if (done) {
                sw = (int64_t)ld_relaxed(p.acc + 2 * (size_t)c);
                sv = (int64_t)ld_relaxed(p.acc + 2 * (size_t)c + 1);
                p.acc[2 * (size_t)c] = p.acc[2 * (size_t)c + 1] = 0ull;
                p.cnt[c] = 0u;
            }
        }
    }
    if (!done) return 0ull;
    sw += s_fix[0];
    sv += s_fix[1];
    const int64_t f = sw <= p.capacity ? sv : -p.lambda * (sw - p.capacity);
    p.fitness[c] = f;
    return elite_key(f, c);
}

// The block's sums in accumulators 0 .. n - 1 (n <= kColRows), of rows s_row[i] of one tile: added
// to the rows, and the rows that are complete evaluated (eq. (1)) and offered to the elite key,
// one atomic per warp. Called by the whole block; leaves the accumulators 0.
template <int kForm>
__device__ __forceinline__ void column_flush(const GenParams &p, int sum_bits, int ntile, const int32_t *s_row, int n,
                                             const int64_t *s_fix, unsigned long long *key, uint32_t *s_acc32,
                                             unsigned long long *s_acc64)
{
    __syncthreads();
    const int i = threadIdx.x;
    if (i < ((n + 31) & ~31)) {
        const unsigned long long best =
            i < n ? column_row_done<kForm>(p, sum_bits, ntile, s_row[i], i, s_fix, s_acc32, s_acc64) : 0ull;
        const uint32_t hi = (uint32_t)(best >> 32), mh = __reduce_max_sync(0xffffffffu, hi);
        const uint32_t lo = hi == mh ? (uint32_t)best : 0u, ml = __reduce_max_sync(0xffffffffu, lo);
        if ((i & 31) == 0 && (mh | ml) != 0u) atomicMax(key, ((unsigned long long)mh << 32) | ml);
    }
    __syncthreads();
}

// The sums of rows ra .. ra + n - 1 of one tile into accumulators acc .. acc + n - 1.
template <int kForm>
__device__ __forceinline__ void column_rows(const GenParams &p, uint32_t one, const ColGeom &m, const BlockShare &b,
                                            const ColItem<kForm> &it, const uint32_t (&T)[8], const ColSum<kForm> &base,
                                            int ra, int n, int acc, uint32_t t, uint32_t *s_acc32,
                                            unsigned long long *s_acc64)
{
    const int lane = threadIdx.x & 31;
    const RowKeys k = row_keys(p, t);
    const QuadWords wa = quad_words(p, (uint32_t)it.qa, t), wb = quad_words(p, (uint32_t)it.qb, t);
    if (m.lanes == 32) {
        // Two rows per step (four independent Philox chains). Lane i keeps the warp's sums of
        // row i of each 32 and adds them at once.
        const int sh = __ffs(m.rpp) - 1;
        const int mypass = (n - b.r_sub + m.rpp - 1) >> sh;          // passes with a row of this thread
        const int passes = it.none ? 0 : (n + m.rpp - 1) >> sh;      // (none: past the tile's width)
        uint32_t row = (uint32_t)(ra + b.r_sub);
        const uint32_t step = (uint32_t)m.rpp;
        for (int q0 = 0; q0 < passes; q0 += 32) {
            const int nq = min(32, passes - q0);
            ColSum<kForm> mine = {0u, 0u, 0, 0};
            int q = 0;
#pragma unroll 1
            for (; q + 1 < nq; q += 2) {
                const ColSum<kForm> a = column_row<kForm>(k, one, it, T, base, wa, wb, row);
                const ColSum<kForm> c = column_row<kForm>(k, one, it, T, base, wa, wb, row + step);
                row += 2u * step;
                const ColSum<kForm> as = column_warp_sum<kForm>(a), cs = column_warp_sum<kForm>(c);
                if (lane == q) mine = as;
                if (lane == q + 1) mine = cs;
            }
            if (q < nq) {
                const ColSum<kForm> as = column_warp_sum<kForm>(column_row<kForm>(k, one, it, T, base, wa, wb, row));
                row += step;
                if (lane == q) mine = as;
            }
            if (lane < nq && q0 + lane < mypass)
                column_add<kForm>(mine, acc + (q0 + lane) * m.rpp + b.r_sub, s_acc32, s_acc64);
        }
    } else {
        for (int q = b.r_sub; q < n + b.r_sub; q += m.rpp) {         // the same trips for every thread
            ColSum<kForm> s = column_row<kForm>(k, one, it, T, base, wa, wb, (uint32_t)(ra + q));
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                if (o < m.lanes) {
                    if constexpr (kForm == 2) {
                        s.w += __shfl_xor_sync(0xffffffffu, s.w, o);
                        s.v += __shfl_xor_sync(0xffffffffu, s.v, o);
                    } else {
                        s.a += __shfl_xor_sync(0xffffffffu, s.a, o);
                        if constexpr (kForm == 1) s.b += __shfl_xor_sync(0xffffffffu, s.b, o);
                    }
                }
            }
            if (b.leader && q < n) column_add<kForm>(s, acc + q, s_acc32, s_acc64);
        }
    }
}

// Sums of the items of a quad's genes at theta = pi/2 (a fixed quad's share of every row).
template <int kForm>
__device__ __forceinline__ void quad_items_at_top(const ColItem<kForm> &it, int half, uint2 s, uint32_t off_top,
                                                  int64_t &w, int64_t &v)
{
    const uint32_t h[4] = {s.x & 0xffffu, s.x >> 16, s.y & 0xffffu, s.y >> 16};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if (h[i] == off_top) {
            if constexpr (kForm == 0) {
                w += it.wv[4 * half + i] & 0xffffu;
                v += it.wv[4 * half + i] >> 16;
            } else {
                w += (int32_t)it.wv[4 * half + i];
                v += it.v[4 * half + i];
            }
        }
    }
}

// A warp's quads that still draw appended to a list and the item sums of its fixed ones added
// to the slot. sta, stb: the quad is fixed; mine: this thread's item counts (whole warps call).
__device__ __forceinline__ void column_append(ColSlot *slot, int32_t *list, int32_t svec, bool mine, bool whole,
                                              int32_t qa, int32_t qb, bool sta, bool stb, int64_t fw, int64_t fv)
{
    const uint32_t full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const bool a = mine && qa >= 0 && !sta, b = mine && qb >= 0 && !stb;
    const bool pv = whole && a && b, pa = a && !pv, pb = b && !pv;
    const uint32_t mv = __ballot_sync(full, pv), ma = __ballot_sync(full, pa), mb = __ballot_sync(full, pb);
    uint32_t base_v = 0u, base_s = 0u;
    if (lane == 0) {
        if (mv) base_v = atomicAdd(&slot->nv, (unsigned int)__popc(mv));
        if (ma | mb) base_s = atomicAdd(&slot->ns, (unsigned int)(__popc(ma) + __popc(mb)));
    }
    base_v = __shfl_sync(full, base_v, 0);
    base_s = __shfl_sync(full, base_s, 0);
    const uint32_t below = (1u << lane) - 1u;
    if (pv) list[base_v + __popc(mv & below)] = qa >> 1;
    if (pa) list[svec + base_s + __popc(ma & below)] = qa;
    if (pb) list[svec + base_s + __popc(ma) + __popc(mb & below)] = qb;
    if (!mine) fw = fv = 0;
    if (__any_sync(full, fw != 0 || fv != 0)) {
        fw = warp_sum64(fw);
        fv = warp_sum64(fv);
        if (lane == 0) {
            atomicAdd(&slot->fw, (unsigned long long)fw);
            atomicAdd(&slot->fv, (unsigned long long)fv);
        }
    }
}

// One CIP step of a thread's item toward alleles x (bit i = gene i).
template <int kForm>
__device__ __forceinline__ uint32_t column_apply(ColItem<kForm> &it, uint32_t x, uint32_t k8)
{
    // a pair's steps: halves +4 (allele 1) or -4, picked by bytes from 0x0004fffc
    const auto step = [&](uint32_t s, uint32_t x2) {
        const uint32_t d = __byte_perm(0x0004fffcu, 0u, 0x1010u + (x2 & 1u) * 0x22u + (x2 >> 1 & 1u) * 0x2200u);
        return __viaddmin_s16x2_relu(s, d, k8);
    };
    it.sa = make_uint2(step(it.sa.x, x), step(it.sa.y, x >> 2));
    it.sb = make_uint2(step(it.sb.x, x >> 4), step(it.sb.y, x >> 6));
    return x;
}

// CIP(t - 1) of a thread's item toward the elite's alleles, which are drawn again from row e's
// counters of generation t - 1 with the thresholds that generation had. Returns the alleles.
template <int kForm>
__device__ __forceinline__ uint32_t column_cip(const GenParams &p, ColItem<kForm> &it, int32_t e, int32_t t,
                                               const uint32_t (&T)[8], uint32_t top, uint32_t k8)
{
    const Draw4 d0 = philox4x32_10_rk((uint32_t)it.qa, (uint32_t)e, (uint32_t)(t - 1), 0u, p.rk0, p.rk1);
    const Draw4 d1 = philox4x32_10_rk((uint32_t)it.qb, (uint32_t)e, (uint32_t)(t - 1), 0u, p.rk0, p.rk1);
    const uint32_t u[8] = {d0.a, d0.b, d0.c, d0.d, d1.a, d1.b, d1.c, d1.d};
    uint32_t x = top;
#pragma unroll
    for (int i = 0; i < 8; ++i)
        if (u[i] < T[i]) x |= 1u << i;
    return column_apply<kForm>(it, x, k8);
}

// What the threads that hold row 0 leave of generation t for others: the angle indices it
// observed, the best row's alleles (x: those of the elite of t - 1) if that improved, and the
// number of quads that the list no longer needs. Called by whole warps.
template <int kForm>
__device__ __forceinline__ void column_lead(const GenParams &p, const ColParams &c, const ColItem<kForm> &it, uint32_t x,
                                            int32_t t, bool improved, bool lead, unsigned int *drops)
{
    const uint32_t off_top = (uint32_t)(8 * p.K);
    uint2 *row = column_parity(c, p.svec, t);
    uint32_t n = 0u;
    if (lead && it.qa >= 0) {
        row[it.qa] = it.sa;
        if (improved) c.best_nib[it.qa] = make_int2(t - 1, (int)(x & 15u));
        n += quad_fixed(it.sa, off_top) ? 1u : 0u;
    }
    if (lead && it.qb >= 0) {
        row[it.qb] = it.sb;
        if (improved) c.best_nib[it.qb] = make_int2(t - 1, (int)(x >> 4));
        n += quad_fixed(it.sb, off_top) ? 1u : 0u;
    }
    n = __reduce_add_sync(0xffffffffu, n);
    if ((threadIdx.x & 31) == 0 && n != 0u) atomicAdd(drops, n);
}

__device__ __forceinline__ void load_sync(const ColSync *sy, unsigned long long &lo, unsigned long long &hi)
{
    asm volatile("{ .reg .b128 q; ld.relaxed.gpu.global.b128 q, [%2]; mov.b128 {%0, %1}, q; }"
                 : "=l"(lo), "=l"(hi) : "l"(sy) : "memory");
}

// A full (release, acquire) barrier of the run's nb blocks, bounded; `target` counts arrivals over
// the run. Whole block; false when the wait ran out.
__device__ __forceinline__ bool column_barrier(const GenParams &p, const ColParams &c, int nb, uint32_t &target,
                                               int32_t *s_ok)
{
    __syncthreads();
    target += (uint32_t)nb;
    if (threadIdx.x == 0) {
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" :: "l"(c.ctl + kCtlRebuilt) : "memory");
        const uint64_t deadline = global_ns() + p.wait_ns;
        int ok = 0;
        for (uint32_t n = 0; n < (1u << 30); ++n) {
            if ((uint32_t)ld_acquire(c.ctl + kCtlRebuilt) >= target) {
                ok = 1;
                break;
            }
            if (ld_acquire(p.error) != 0 || global_ns() > deadline) break;
        }
        if (!ok) atomicOr(p.error, kErrBarrierTimeout);
        *s_ok = ok;
    }
    __syncthreads();
    return *s_ok != 0;
}

// The posted form of the wait: every block's word of generation t, read until it holds t + 1;
// s_red[w] receives warp w's part (bounded; false when the wait ran out). Whole block.
__device__ __forceinline__ bool column_wait_posts(const GenParams &p, const ColParams &c, int32_t t, int nb,
                                                  ColSync *s_red, ColSync &out)
{
    const int tid = threadIdx.x;
    const ColSync *post = c.post + (size_t)(t & 1) * kColPosted;
    unsigned long long key = 0ull;
    uint32_t drops = 0u;
    bool ok = true;
    if (tid < nb) {
        const uint64_t deadline = global_ns() + p.wait_ns;
        for (int i = tid; i < nb && ok; i += kThreads) {
            unsigned long long lo, hi;
            uint32_t n = 0u;
            for (;;) {
                load_sync(post + i, lo, hi);
                if ((uint32_t)hi == (uint32_t)t + 1u) break;
                if ((++n & 15u) == 0u && (n >= (1u << 30) || ld_acquire(p.error) != 0 || global_ns() > deadline)) {
                    ok = false;
                    break;
                }
            }
            key = max(key, lo);
            drops += (uint32_t)(hi >> 32);
        }
        if (!ok) atomicOr(p.error, kErrBarrierTimeout);
    }
    const int used = (min(nb, kThreads) + 31) >> 5;       // warps with a word to read
    if ((tid >> 5) < used) {
        __syncwarp();
        const uint32_t hi = (uint32_t)(key >> 32), mh = __reduce_max_sync(0xffffffffu, hi);
        const uint32_t lo = hi == mh ? (uint32_t)key : 0u, ml = __reduce_max_sync(0xffffffffu, lo);
        drops = __reduce_add_sync(0xffffffffu, drops);
        ok = __all_sync(0xffffffffu, ok);
        if ((tid & 31) == 0) {
            ColSync r;
            r.key = ((unsigned long long)mh << 32) | ml;
            r.arrived = ok ? 1u : 0u;
            r.drops = drops;
            s_red[tid >> 5] = r;
        }
    }
    __syncthreads();
    out = s_red[0];
    for (int w = 1; w < used; ++w) {
        const ColSync r = s_red[w];
        out.key = max(out.key, r.key);
        out.arrived &= r.arrived;
        out.drops += r.drops;
    }
    return out.arrived != 0u;
}

// Waits until nb blocks have arrived in *sy (bounded like grid_wait); thread 0 only. An arrival is a
// release add after its block's updates of the key and the drops; the acquire load that sees
// the last one orders the loads of those words, each of the size its atomics have. (One 16-byte load
// of all three would save a trip to L2: 1,000 generations of 1,024 x 10,000 in 1,256 us instead of
// 1,285. But the memory model orders nothing between it and atomics on parts of it.)
__device__ __forceinline__ bool column_wait(const GenParams &p, const ColSync *sy, unsigned int nb, ColSync &out)
{
    const uint64_t deadline = global_ns() + p.wait_ns;
    for (uint32_t n = 0; n < (1u << 30); ++n) {
        if ((unsigned int)ld_acquire(reinterpret_cast<const int32_t *>(&sy->arrived)) >= nb) {
            out.key = ld_relaxed(&sy->key);
            asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(out.drops) : "l"(&sy->drops) : "memory");
            return true;
        }
        if (global_ns() > deadline || ((n & 15u) == 15u && ld_acquire(p.error) != 0)) break;
    }
    atomicOr(p.error, kErrBarrierTimeout);
    return false;
}

// A shorter list of the quads that still draw, built by all nb blocks at the start of generation t
// from the angle indices generation t - 2 observed (every block can read them by now): the quads
// fixed then leave, and both parities hold their state. counts: the list's, in shared memory (and
// the item sums of the quads that left). Whole block; false when a wait ran out.
template <int kForm>
__device__ __forceinline__ bool column_rebuild(const GenParams &p, const ColParams &c, ColItem<kForm> &it, int block,
                                               int nb, int items, uint32_t nv, uint32_t ns, int cur, int32_t t,
                                               uint32_t rebuilds, uint32_t &target, ColSlot *counts, int32_t *s_ok)
{
    const uint32_t off_top = (uint32_t)(8 * p.K);
    const int tid = threadIdx.x;
    ColSlot *slot = nb > 1 ? c.slot + rebuilds % 3u : counts;
    const uint2 *state = column_parity(c, p.svec, t - 2);
    uint2 *other = column_parity(c, p.svec, t - 1);
    for (int i0 = block * kThreads; i0 < items; i0 += nb * kThreads) {
        const int i = i0 + tid;
        const bool mine = i < items;
        column_item<kForm>(p, it, column_list(c, p.svec, cur), nv, ns, i, mine, state);
        const bool sta = quad_fixed(it.sa, off_top), stb = quad_fixed(it.sb, off_top);
        int64_t fw = 0, fv = 0;
        if (it.qa >= 0 && sta) {
            quad_items_at_top<kForm>(it, 0, it.sa, off_top, fw, fv);
            other[it.qa] = it.sa;
        }
        if (it.qb >= 0 && stb) {
            quad_items_at_top<kForm>(it, 1, it.sb, off_top, fw, fv);
            other[it.qb] = it.sb;
        }
        column_append(slot, column_list(c, p.svec, cur ^ 1), p.svec, mine, it.whole, it.qa, it.qb, sta, stb, fw, fv);
    }
    if (nb > 1) {
        if (!column_barrier(p, c, nb, target, s_ok)) return false;
        if (tid == 0) {
            counts->nv = __ldcg(&slot->nv);
            counts->ns = __ldcg(&slot->ns);
            counts->fw = __ldcg(&slot->fw);
            counts->fv = __ldcg(&slot->fv);
            if (block == 0) c.slot[(rebuilds + 1u) % 3u] = ColSlot{};
        }
    }
    __syncthreads();
    return true;
}

// Records of generation t with elite e of fitness f (one thread). drew: vectors that it drew (those on its list).
__device__ __forceinline__ void column_record(const GenParams &p, int32_t t, int32_t e, int64_t f, bool improved,
                                              int32_t run, uint32_t drew)
{
    p.hist_e[t] = e;
    p.hist_f[t] = f;
    *p.elite_idx = e;
    if (improved) {
        p.best[0] = f;
        p.best[1] = t;
        p.best[2] = e;
    }
    if (p.converge) p.conv[t & 1] = run;
    if (p.hist_d) p.hist_d[t] = (unsigned long long)p.np * (unsigned long long)((uint32_t)p.svec - drew);
}

// The end of a run, by block 0: t_last was its last generation if `over`; otherwise every quad is
// fixed from generation t0 + g on, and the remaining generations have equal rows.
__device__ __forceinline__ void column_finish(const GenParams &p, const ColParams &c, int32_t t0, int32_t g, int32_t G,
                                              int32_t t_last, bool over, bool stop, int64_t best_f, int64_t prev_f,
                                              int32_t run, const int64_t *s_fix)
{
    const int tid = threadIdx.x;
    if (!over) {
        const int64_t fw = s_fix[0], fv = s_fix[1];
        const int64_t f = fw <= p.capacity ? fv : -p.lambda * (fw - p.capacity);
        int32_t n = G - g;
        if (p.converge) {
            const int32_t first = (run > 0 && f == prev_f) ? run + 1 : 1;    // at generation t0 + g
            const int32_t need = max(1, kConvergeWindow - first + 1);        // generations until it stops
            stop = need <= n;
            n = min(n, need);
            if (tid == 0) {
                if (n >= 2) p.conv[(t0 + g + n - 2) & 1] = first + n - 2;
                p.conv[(t0 + g + n - 1) & 1] = first + n - 1;
            }
        }
        t_last = t0 + g + n - 1;
        // (a device clock tick each: these generations cost nothing of their own)
        const unsigned long long now = p.gen_ns ? max((unsigned long long)global_ns(), p.gen_ns[g]) : 0ull;
        for (int32_t i = tid; i < n; i += kThreads) {
            p.hist_e[t0 + g + i] = 0;
            p.hist_f[t0 + g + i] = f;
            if (p.hist_d) p.hist_d[t0 + g + i] = (unsigned long long)p.np * (unsigned long long)(uint32_t)p.svec;
            if (p.gen_ns) p.gen_ns[g + 1 + i] = now + 1u + (unsigned long long)i;
        }
        for (int32_t i = tid; i < p.np; i += kThreads) p.fitness[i] = f;
        if (tid == 0) {
            *p.elite_idx = 0;
            if (f > best_f) {
                p.best[0] = f;
                p.best[1] = t0 + g;
                p.best[2] = 0;
            }
        }
    }
    if (tid == 0) {
        c.ctl[kCtlLast] = t_last;
        c.ctl[kCtlEarly] = t_last != t0 + G - 1 ? 1 : 0;
        c.ctl[kCtlRan] = 1;
        if (stop) {
            p.conv[3] = t_last;
            p.conv[2] = kStopped;
        }
    }
}

// Start of a run or of its rest: whether there is anything to do, and the words that say how it
// stands. Whole block; head values are read by every thread.
__device__ __forceinline__ bool column_stopped(const GenParams &p, const ColParams &c, int block)
{
    if (!p.converge || *(volatile const int32_t *)(p.conv + 2) == kRunning) return false;
    if (block == 0 && threadIdx.x == 0) c.ctl[kCtlRan] = 0;
    return true;
}

// Whether an earlier wait of the instance ran out (one thread; its block shares the answer, since
// another block may set the word meanwhile). The words of such a run are not those of any
// generation, so nothing runs on them until a reset: column_begin has left kCtlRan 0, and the
// launches that follow change neither the records nor the generation counter.
__device__ __forceinline__ bool column_failed(const GenParams &p) { return __ldcg(p.error) != 0; }

__device__ __forceinline__ void column_begin(const GenParams &p, const ColParams &c, int32_t t0, bool draws)
{
    c.ctl[kCtlRan] = 0;
    c.ctl[kCtlRebuild] = draws ? 1 : 0;
    c.ctl[kCtlFirst] = t0;
    c.ctl[kCtlEarly] = 0;
    if (p.gen_ns) p.gen_ns[0] = global_ns();
}

template <int kForm>
struct ColRunShared {
    uint32_t thr[kMaxThr];
    unsigned long long acc64[kForm == 2 ? 2 * kColRows : 1];
    uint32_t acc32[kForm == 2 ? 1 : 2 * kColRows];
    ColSync snap;                 // what thread 0 read of the generation before
    int32_t ok;
    ColSlot slot;
    int64_t fix[2];               // item sums of the dropped quads
    uint32_t seg[2];
    float debt;                   // generations' worth of draws of fixed quads
    int32_t shorter;              // build a shorter list
    int32_t row[kColRows];        // rows of the accumulators
};

// The generations of a run whose blocks have several passes each (at least kColSmallShare):
// every block has a home tile (ColHome). Every block follows the same sequence of lists, elites and
// records from the same device words. Once the list is short the rest of the run is handed to
// column_small_kernel.
//
// Bound by the integer pipes: per 8 genes and row two Philox calls (32 wide multiplies, 35 xors),
// 8 compares and 8 adds. Wide multiplies hold the FMA-heavy pipe for four cycles and the ALU's
// issue for two, so a pass costs about 2.13 cycles per ALU instruction plus 2 per wide multiply;
// the row-by-row pass spends 108 ALU instructions where this one spends about 48.
//
// kPerSm blocks per SM: two (up to 128 registers a thread) pass 4-5 % faster than three (up to
// 80), but three cut some populations more evenly; the host takes the cheaper (column_cost).
// Measured, us per generation with every qubit drawn: 4,096 x 100,000 248 with two and 260 with
// three (the row-by-row form 424); 6,001 x 70,001 273 and 260 (441).
template <int kForm, bool kMember>
__device__ __forceinline__ void column_run(const GenParams &p, const ColParams &c, int32_t G, int block, int grid,
                                           ColRunShared<kForm> &sh)
{
    const int tid = threadIdx.x;
    load_thresholds(p, sh.thr);
    for (int i = tid; i < 2 * kColRows; i += kThreads) {
        if constexpr (kForm == 2) sh.acc64[i] = 0ull;
        else sh.acc32[i] = 0u;
    }
    if (!kMember) grid_dependency_wait();
    if (column_stopped(p, c, block)) return;
    const int32_t t0 = *p.gen;
    uint32_t nv = c.head->nv, ns = c.head->ns;
    ColGeom m = column_geometry(nv, ns, p.np, grid);
    if (!kMember && m.small) return;              // the whole run is column_small_kernel's
    ColHome h = column_home(m, block, grid);
    if (block >= m.nb) return;
    if (tid == 0) {
        sh.fix[0] = (int64_t)c.head->fw;
        sh.fix[1] = (int64_t)c.head->fv;
        sh.slot = ColSlot{};
        sh.debt = 0.0f;
        sh.ok = column_failed(p) ? 0 : 1;
    }
    const unsigned char *thr_bytes = reinterpret_cast<const unsigned char *>(sh.thr);
    const uint32_t off_top = (uint32_t)(8 * p.K), k8 = off_top * 0x00010001u;
    // the records' running values, the same in every block
    int64_t best_f = __ldcg(p.best + 1) < 0 ? INT64_MIN : __ldcg(p.best), prev_f = 0;
    int32_t run = 0;                              // equal elite fitness ending at t - 1
    if (p.converge && t0 > 0) {
        run = __ldcg(p.conv + ((t0 - 1) & 1));
        prev_f = __ldcg(p.hist_f + t0 - 1);
    }
    const bool rec = block == 0 && tid == 0;
    if (rec) column_begin(p, c, t0, nv + ns != 0u);
    BlockShare b = tile_geometry(m.lanes, m.warps);
    int cur = 0;
    uint32_t rebuilds = 0u, rb_target = 0u;
    int32_t g_check = 1;                          // the first generation whose count is of this list
    bool loaded = false;                          // the item of a fixed share is in registers
    ColItem<kForm> it;
    uint32_t T[8], top = 0u;
    ColSum<kForm> base;
    int32_t g = 0, e = 0;
    bool improved = false, stop = false;
    __syncthreads();
    if (!sh.ok) return;

    for (; !kMember || m.items != 0; ++g) {
        const int32_t t = t0 + g;
        if (g > 0) {
            // generation t - 1 is complete once every block has arrived
            if (tid == 0) {
                sh.ok = column_wait(p, c.sync + ((t - 1) & 3), (unsigned int)m.nb, sh.snap) ? 1 : 0;
                const uint32_t nq = 2u * nv + ns;
                if (g >= g_check) sh.debt += (float)sh.snap.drops / (float)nq;
                sh.shorter = g >= g_check && (sh.debt * (float)h.share >= 15.0f || sh.snap.drops == nq) ? 1 : 0;
                if (sh.shorter) sh.debt = 0.0f;
            }
            __syncthreads();
            if (!sh.ok) return;
            e = (int32_t)(0xffffffu - (uint32_t)(sh.snap.key & 0xffffffull));
            const int64_t f = (int64_t)(sh.snap.key >> 24) - kKeyBias;
            if (e < 0 || e >= p.np) {             // every row finishes in every generation
                if (rec) atomicOr(p.error, kErrEliteRange);
                e = 0;
            }
            improved = f > best_f;
            if (improved) best_f = f;
            if (p.converge) {
                run = (run > 0 && f == prev_f) ? run + 1 : 1;
                prev_f = f;
                stop = run >= kConvergeWindow;
            }
            if (rec) {
                column_record(p, t - 1, e, f, improved, run, nv + ns);
                if (p.gen_ns) p.gen_ns[g] = global_ns();
            }
            if (g == G || stop) break;
            // A shorter list once the passes spent on fixed quads have cost what building it costs
            // (about 8 us; a pass of a block takes 0.55 us). The count is that of generation
            // t - 2, whose angle indices every block can read by now.
            if (sh.shorter) {
                if (!column_rebuild<kForm>(p, c, it, block, m.nb, m.items, nv, ns, cur, t, rebuilds, rb_target, &sh.slot,
                                           &sh.ok))
                    return;
                g_check = g + 2;
                ++rebuilds;
                cur ^= 1;
                nv = sh.slot.nv;
                ns = sh.slot.ns;
                if (tid == 0) {
                    sh.fix[0] += (int64_t)sh.slot.fw;
                    sh.fix[1] += (int64_t)sh.slot.fv;
                }
                const int before = m.nb;          // (blocks that have left do not come back)
                m = column_geometry(nv, ns, p.np, grid);
                loaded = false;
                if (!kMember && m.small) {
                    if (rec) {
                        c.ctl[kCtlGen] = g;
                        c.ctl[kCtlCur] = cur;
                        c.ctl[kCtlRebuilds] = (int32_t)rebuilds;
                        c.ctl[kCtlElite] = e;
                        c.ctl[kCtlImproved] = improved ? 1 : 0;
                        ColSlot r{};
                        r.nv = nv;
                        r.ns = ns;
                        r.fw = (unsigned long long)sh.fix[0];
                        r.fv = (unsigned long long)sh.fix[1];
                        *c.rest = r;
                        c.ctl[kCtlPhase] = 1;
                    }
                    return;
                }
                h = column_home(m, block, before);
                if (block >= m.nb) return;
                b = tile_geometry(m.lanes, m.warps);
                if (kMember) {
                    __syncthreads();
                    if (tid == 0) sh.slot = ColSlot{};
                    if (m.items == 0) break;
                }
            }
        }
        // Words are cleared two generations ahead: the blocks' parts of t + 1 may be written as
        // soon as their own of t are done.
        ColSync *const sy = c.sync + (t & 3);
        if (rec) c.sync[(t + 2) & 3] = ColSync{};
        const uint2 *state = g == 0 ? c.canon : column_parity(c, p.svec, t + 1);
        for (int turn = 0; turn < h.turns; ++turn) {
            const int tile = h.home + turn * h.stride;
            unsigned int *const queue = c.qctr + (t & 3) * kColQueues + h.home;
            if (h.queued && h.part == 0 && tid == 0) c.qctr[((t + 2) & 3) * kColQueues + h.home] = 0u;
            const int i = tile * m.width + b.v_in;
            const bool active = b.v_in < m.width && i < m.items;
            if (!loaded) {
                column_item<kForm>(p, it, column_list(c, p.svec, cur), nv, ns, i, active, state);
                column_thresholds<kForm>(it, thr_bytes, off_top, T, top, base);
            }
            loaded = h.turns == 1;
            uint32_t x = 0u;
            if (g > 0) {
                x = column_cip<kForm>(p, it, e, t, T, top, k8);
                column_thresholds<kForm>(it, thr_bytes, off_top, T, top, base);
            }
            if (h.part == 0)
                column_lead<kForm>(p, c, it, x, t, improved, b.r_sub == 0 && active, &c.sync[(t + 1) & 3].drops);
            // The sums of several pieces' rows are kept until the accumulators are full.
            int ua, ub, used = 0;
            column_piece(m, h, h.part, ua, ub);
            for (uint32_t piece = 1u; ua < m.nu; ++piece) {
                // the next piece's index arrives while this one is computed
                uint32_t next = 0u;
                if (h.queued && tid == 0) next = atomicAdd(queue, 1u);
                const int rb = min(p.np, ub * m.rpp);
                for (int ra = ua * m.rpp; ra < rb;) {
                    const int n = min(kColRows - used, rb - ra);
                    if (tid < n) sh.row[used + tid] = ra + tid;
                    column_rows<kForm>(p, c.one, m, b, it, T, base, ra, n, used, (uint32_t)t, sh.acc32, sh.acc64);
                    ra += n;
                    used += n;
                    if (used == kColRows) {
                        column_flush<kForm>(p, c.sum_bits, m.ntile, sh.row, used, sh.fix, &sy->key, sh.acc32, sh.acc64);
                        used = 0;
                    }
                }
                if (!h.queued) break;
                if (tid == 0) sh.seg[piece & 1u] = next;
                __syncthreads();
                column_piece(m, h, h.group + (int)sh.seg[piece & 1u], ua, ub);
            }
            if (used) column_flush<kForm>(p, c.sum_bits, m.ntile, sh.row, used, sh.fix, &sy->key, sh.acc32, sh.acc64);
        }
        __syncthreads();
        if (tid == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" :: "l"(&sy->arrived) : "memory");
    }
    if (kMember) __syncthreads();
    if (block == 0) column_finish(p, c, t0, g, G, t0 + g - 1, !kMember || m.items != 0, stop, best_f, prev_f, run, sh.fix);
    if (!kMember && rec) c.ctl[kCtlPhase] = 2;
}

template <int kForm, int kPerSm>
__global__ void __launch_bounds__(kThreads, kPerSm) column_run_kernel(const GenParams p, const ColParams c, int32_t G)
{
    __shared__ ColRunShared<kForm> sh;
    column_run<kForm, false>(p, c, G, (int)blockIdx.x, (int)gridDim.x, sh);
}

// The generations of a run (or of the rest of one) in which a block has at most a few passes: bound
// by the chain from one generation's elite to the next, which the code keeps short. Every block
// has one fixed share of one tile, its item in registers. What does not depend on the elite is
// done before waiting for it: the records and the lead threads' stores of the generation before
// and the draws of the first two passes (Philox is keyed by counters, so generation t's draws
// exist before its angles do). A block left alone also keeps the alleles it observed, so that
// it need not draw the elite's again, and meets nobody.
template <int kForm>
__global__ void __launch_bounds__(kThreads, 2) column_small_kernel(const GenParams p, const ColParams c, int32_t G)
{
    constexpr uint32_t kRedraw = 0x100u;          // the elite's alleles are not in s_x
    __shared__ uint32_t s_thr[kMaxThr];
    __shared__ unsigned long long s_acc64[kForm == 2 ? 2 * kColSmallRows : 1];
    __shared__ uint32_t s_acc32[kForm == 2 ? 1 : 2 * kColSmallRows];
    __shared__ ColSync s_sync[4];                 // this block's part of generation t in t & 3
    __shared__ ColSync s_red[2][kThreads / 32];
    __shared__ ColSync s_snap;
    __shared__ int32_t s_ok;
    __shared__ ColSlot s_slot;
    __shared__ int64_t s_fix[2];
    __shared__ uint8_t s_x[2][kColLocalPasses * kThreads];   // a block alone: alleles by parity, pass, thread
    const int tid = threadIdx.x;
    load_thresholds(p, s_thr);
    for (int i = tid; i < 2 * kColSmallRows; i += kThreads) {
        if constexpr (kForm == 2) s_acc64[i] = 0ull;
        else s_acc32[i] = 0u;
    }
    grid_dependency_wait();
    const int32_t phase = c.ctl[kCtlPhase];
    if (phase == 2 || (phase == 0 && column_stopped(p, c, (int)blockIdx.x))) return;
    const int32_t t0 = phase ? c.ctl[kCtlFirst] : *p.gen;
    const ColSlot *from = phase ? c.rest : c.head;
    uint32_t nv = from->nv, ns = from->ns;
    if (tid == 0) {
        s_fix[0] = (int64_t)from->fw;
        s_fix[1] = (int64_t)from->fv;
        s_slot = ColSlot{};
        for (int i = 0; i < 4; ++i) s_sync[i] = ColSync{};
        s_ok = column_failed(p) ? 0 : 1;          // (column_run_kernel's wait, among others)
    }
    int32_t g = phase ? c.ctl[kCtlGen] : 0, e = phase ? c.ctl[kCtlElite] : 0;
    int cur = phase ? c.ctl[kCtlCur] : 0;
    uint32_t rebuilds = phase ? (uint32_t)c.ctl[kCtlRebuilds] : 0u, rb_target = (uint32_t)c.ctl[kCtlRebuilt];
    bool improved = phase && c.ctl[kCtlImproved], stop = false;
    const unsigned char *thr_bytes = reinterpret_cast<const unsigned char *>(s_thr);
    const uint32_t off_top = (uint32_t)(8 * p.K), k8 = off_top * 0x00010001u;
    int64_t best_f = __ldcg(p.best + 1) < 0 ? INT64_MIN : __ldcg(p.best), prev_f = 0;
    int64_t f = INT64_MIN;                        // fitness of e's record while it is still to be written
    int32_t run = 0;
    if (p.converge && t0 + g > 0) {
        run = __ldcg(p.conv + ((t0 + g - 1) & 1));
        prev_f = __ldcg(p.hist_f + t0 + g - 1);
    }
    const bool rec = blockIdx.x == 0 && tid == 0;
    if (rec && !phase) column_begin(p, c, t0, nv + ns != 0u);

    // geometry of a list: this block's share, at most kColLocalPasses passes
    ColGeom m;
    BlockShare b;
    bool alone, posted, lead_share = false;
    int tile = 0, row0 = 0, rows = 0, passes = 0, nb = 1, most = 1;   // most: passes of the largest share
    auto cut = [&](int grid) {
        m = column_geometry(nv, ns, p.np, grid);
        const uint32_t units = (uint32_t)m.ntile * (uint32_t)m.nu;
        alone = m.items == 0 || (m.ntile == 1 && units <= (uint32_t)kColLocalPasses);
        nb = alone ? 1 : m.nb;
        most = (int)((units + (uint32_t)nb - 1u) / (uint32_t)nb);
        // Rows of a single tile are complete within a block, so nothing but its best row's key
        // need reach the others: each block posts it with its generation number in one 16-byte
        // store and reads everyone's, which saves the key's atomic and the fence before an
        // arrival (about 1,000 cycles). With hundreds of blocks the reads cost more than that.
        posted = !alone && m.ntile == 1 && nb <= kColPosted;
        b = tile_geometry(m.lanes, m.warps);
        if ((int)blockIdx.x >= nb) return;
        tile = (int)blockIdx.x % m.ntile;
        const int part = (int)blockIdx.x / m.ntile, parts = (nb - tile + m.ntile - 1) / m.ntile;
        const int ua = (int)((int64_t)m.nu * part / parts), ub = (int)((int64_t)m.nu * (part + 1) / parts);
        row0 = ua * m.rpp;
        rows = min(p.np, ub * m.rpp) - row0;
        passes = ub - ua;
        lead_share = ua == 0 && ub > 0 && b.r_sub == 0 && b.v_in < m.width && tile * m.width + b.v_in < m.items;
    };
    cut((int)gridDim.x);
    if ((int)blockIdx.x >= nb) return;
    ColItem<kForm> it;
    uint32_t T[8], top = 0u, x = g > 0 ? kRedraw : 0u;
    ColSum<kForm> base;
    auto load = [&](const uint2 *state) {
        const int i = tile * m.width + b.v_in;
        column_item<kForm>(p, it, column_list(c, p.svec, cur), nv, ns, i, b.v_in < m.width && i < m.items, state);
        column_thresholds<kForm>(it, thr_bytes, off_top, T, top, base);
    };
    int32_t g_check = g + 2;
    float debt = 0.0f;                            // generations' worth of draws of fixed quads
    bool have = true;                             // generation t0 + g - 1's elite is known
    int q = 0;                                    // the pass of the pair below
    __syncthreads();
    if (!s_ok) return;
    if (m.items != 0) load(g == 0 ? c.canon : column_parity(c, p.svec, t0 + g + 1));

    while (m.items != 0) {
        const int32_t t = t0 + g;
        // draws of passes q and q + 1
        const uint32_t row = (uint32_t)(row0 + q * m.rpp + b.r_sub);
        const Draw4 a0 = philox4x32_10_rk((uint32_t)it.qa, row, (uint32_t)t, 0u, p.rk0, p.rk1);
        const Draw4 a1 = philox4x32_10_rk((uint32_t)it.qb, row, (uint32_t)t, 0u, p.rk0, p.rk1);
        const Draw4 c0 = philox4x32_10_rk((uint32_t)it.qa, row + (uint32_t)m.rpp, (uint32_t)t, 0u, p.rk0, p.rk1);
        const Draw4 c1 = philox4x32_10_rk((uint32_t)it.qb, row + (uint32_t)m.rpp, (uint32_t)t, 0u, p.rk0, p.rk1);
        if (q == 0) {
            if (!have) {
                ColSync sn;
                if (posted) {
                    if (!column_wait_posts(p, c, t - 1, nb, s_red[t & 1], sn)) return;
                } else if (!alone) {
                    if (tid == 0) s_ok = column_wait(p, c.sync + ((t - 1) & 3), (unsigned int)nb, s_snap) ? 1 : 0;
                    __syncthreads();
                    if (!s_ok) return;
                    sn = s_snap;
                } else {
                    sn = s_sync[(t - 1) & 3];     // (after the last flush's barrier)
                }
                e = (int32_t)(0xffffffu - (uint32_t)(sn.key & 0xffffffull));
                if (e < 0 || e >= p.np) {         // every row finishes in every generation
                    if (rec) atomicOr(p.error, kErrEliteRange);
                    e = 0;
                }
                f = (int64_t)(sn.key >> 24) - kKeyBias;
                improved = f > best_f;
                if (improved) best_f = f;
                if (p.converge) {
                    run = (run > 0 && f == prev_f) ? run + 1 : 1;
                    prev_f = f;
                    stop = run >= kConvergeWindow;
                }
                if (p.gen_ns && rec) p.gen_ns[g] = global_ns();
                if (g == G || stop) break;
                have = true;
                // A shorter list: when it halves (fewer blocks meet sooner), or when its passes have
                // been worth the rebuild (about 5 us; a pass takes 0.3 us).
                const uint32_t nq = 2u * nv + ns;
                if (g >= g_check) debt += (float)sn.drops / (float)nq;
                if (g >= g_check && (2u * sn.drops >= nq || debt * (float)most >= 16.0f)) {
                    debt = 0.0f;
                    if (rec) column_record(p, t - 1, e, f, improved, run, nv + ns);
                    // the posted wait orders nothing but the posts: the angle indices need a barrier
                    __syncthreads();
                    if (posted && !column_barrier(p, c, nb, rb_target, &s_ok)) return;
                    if (!column_rebuild<kForm>(p, c, it, (int)blockIdx.x, nb, m.items, nv, ns, cur, t, rebuilds, rb_target,
                                               &s_slot, &s_ok))
                        return;
                    g_check = g + 2;
                    ++rebuilds;
                    cur ^= 1;
                    nv = s_slot.nv;
                    ns = s_slot.ns;
                    const int before = nb;
                    cut(before);
                    if ((int)blockIdx.x >= nb) return;
                    __syncthreads();
                    if (tid == 0) {
                        s_fix[0] += (int64_t)s_slot.fw;
                        s_fix[1] += (int64_t)s_slot.fv;
                        s_slot = ColSlot{};
                    }
                    __syncthreads();
                    if (m.items != 0) load(column_parity(c, p.svec, t + 1));
                    f = INT64_MIN;
                    x = kRedraw;
                    continue;                     // the draws of the new share
                }
            }
            if (g > 0) {
                if (alone && x != kRedraw) {
                    // the alleles this block observed in row e
                    const uint32_t xe = s_x[(t - 1) & 1][(e / m.rpp) * kThreads + (e % m.rpp) * b.tile_vecs + b.v_in];
                    x = column_apply<kForm>(it, xe | top, k8);
                } else {
                    x = column_cip<kForm>(p, it, e, t, T, top, k8);
                }
                column_thresholds<kForm>(it, thr_bytes, off_top, T, top, base);
            }
        }
        // the sums of the two passes
        const int acc0 = q * m.rpp % kColSmallRows;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint32_t u[8] = {h ? c0.a : a0.a, h ? c0.b : a0.b, h ? c0.c : a0.c, h ? c0.d : a0.d,
                                   h ? c1.a : a1.a, h ? c1.b : a1.b, h ? c1.c : a1.c, h ? c1.d : a1.d};
            if (q + h >= passes) break;
            ColSum<kForm> s = column_sum<kForm>(it, T, base, u, c.one);
            if (alone) {
                uint32_t xb = 0u;
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (u[i] < T[i]) xb |= 1u << i;
                s_x[t & 1][(q + h) * kThreads + tid] = (uint8_t)xb;
            }
            if (m.lanes == 32) {
                s = column_warp_sum<kForm>(s);
            } else {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    if (o < m.lanes) {
                        if constexpr (kForm == 2) {
                            s.w += __shfl_xor_sync(0xffffffffu, s.w, o);
                            s.v += __shfl_xor_sync(0xffffffffu, s.v, o);
                        } else {
                            s.a += __shfl_xor_sync(0xffffffffu, s.a, o);
                            if constexpr (kForm == 1) s.b += __shfl_xor_sync(0xffffffffu, s.b, o);
                        }
                    }
                }
            }
            if (b.leader && (q + h) * m.rpp + b.r_sub < rows) column_add<kForm>(s, acc0 + h * m.rpp + b.r_sub, s_acc32, s_acc64);
        }
        q += 2;
        // flush when the accumulators are used up or the share is done
        if (q < passes && (q * m.rpp) % kColSmallRows != 0) continue;
        const int done = min(rows, q * m.rpp), first = (max(done, 1) - 1) / kColSmallRows * kColSmallRows;
        __syncthreads();
        ColSync *const sy = alone || posted ? s_sync + (t & 3) : c.sync + (t & 3);
        for (int i = tid; i < ((done - first + 31) & ~31); i += kThreads) {
            const unsigned long long key = first + i < done
                ? column_row_done<kForm>(p, c.sum_bits, m.ntile, row0 + first + i, i, s_fix, s_acc32, s_acc64) : 0ull;
            const uint32_t hi = (uint32_t)(key >> 32), mh = __reduce_max_sync(0xffffffffu, hi);
            const uint32_t lo = hi == mh ? (uint32_t)key : 0u, ml = __reduce_max_sync(0xffffffffu, lo);
            if ((tid & 31) == 0 && (mh | ml) != 0u) {
                const unsigned long long k = ((unsigned long long)mh << 32) | ml;
                if ((alone || posted) && rows <= 32) sy->key = k;       // (this thread's alone)
                else atomicMax(&sy->key, k);
            }
        }
        __syncthreads();
        if (q < passes) continue;
        // generation t is done here: tell the others, then what need not be told first. (Words are
        // cleared two generations ahead: parts of t + 1 may be written by now.)
        if (tid == 0) {
            if (rec && !alone && !posted) c.sync[(t + 2) & 3] = ColSync{};
            if (posted) {
                const unsigned long long hi = (unsigned long long)((uint32_t)t + 1u) | ((unsigned long long)sy->drops << 32);
                asm volatile("{ .reg .b128 q; mov.b128 q, {%0, %1}; st.relaxed.gpu.global.b128 [%2], q; }"
                             :: "l"(sy->key), "l"(hi), "l"(c.post + (size_t)(t & 1) * kColPosted + blockIdx.x) : "memory");
            } else if (!alone) {
                asm volatile("red.release.gpu.global.add.u32 [%0], 1;" :: "l"(&sy->arrived) : "memory");
            }
            s_sync[(t + 2) & 3] = ColSync{};
        }
        if (rec && f != INT64_MIN) column_record(p, t - 1, e, f, improved, run, nv + ns);
        if (__any_sync(0xffffffffu, lead_share))
            column_lead<kForm>(p, c, it, x, t, improved, lead_share,
                               &(alone || posted ? s_sync : c.sync)[(t + 1) & 3].drops);
        x = 0u;
        q = 0;
        ++g;
        have = false;
    }
    if (blockIdx.x != 0) return;
    const bool over = m.items != 0;
    if (over && rec) column_record(p, t0 + g - 1, e, f, improved, run, nv + ns);
    __syncthreads();
    column_finish(p, c, t0, g, G, t0 + g - 1, over, stop, best_f, prev_f, run, s_fix);
}

// The angle indices that generation t (t_last, or the one before it) observed, of quad q: a
// quad fixed when the run began was never on its list.
__device__ __forceinline__ uint2 observed_quad(const ColParams &c, int32_t svec, int q, int32_t t, uint32_t off_top)
{
    const uint2 s = c.canon[q];
    return quad_fixed(s, off_top) ? s : column_parity(c, svec, t)[q];
}

// The allele plane of the run's last generation (and, when the run stopped early, of the one
// before, which the plane of the other parity holds): byte v of row r is the alleles of vector
// v. A thread keeps one vector for its rows; vectors at the bounds store their sides.
__device__ __forceinline__ void column_plane(const GenParams &p, const ColParams &c, int block, int blocks,
                                             const uint32_t *s_thr)
{
    if (!c.ctl[kCtlRan]) return;
    // no block of this launch reads the head; the next launch fills it again
    if (block == 0 && threadIdx.x == 0 && c.ctl[kCtlRebuild]) *c.head = ColSlot{};
    const int tiles = (p.svec + kThreads - 1) / kThreads;
    const unsigned char *thr_bytes = reinterpret_cast<const unsigned char *>(s_thr);
    const uint32_t off_top = (uint32_t)(8 * p.K);
    const int tile = block % tiles, part = block / tiles;
    const int parts = blocks / tiles;
    if (part >= parts) return;
    const int ra = (int)((int64_t)p.np * part / parts), rb = (int)((int64_t)p.np * (part + 1) / parts);
    const int vec = tile * kThreads + (int)threadIdx.x;
    const int32_t t_last = c.ctl[kCtlLast];
    const int planes = c.ctl[kCtlEarly] && t_last > c.ctl[kCtlFirst] ? 2 : 1;
    if (vec < p.svec) {
        for (int k = 0; k < planes; ++k) {
            const int32_t t = t_last - k;
            const uint2 sa = observed_quad(c, p.svec, 2 * vec, t, off_top), sb = observed_quad(c, p.svec, 2 * vec + 1, t, off_top);
            uint8_t *x = p.xbits + (size_t)(t & 1) * p.xplane + (size_t)ra * p.xstride + vec;
            if (quad_fixed(sa, off_top) && quad_fixed(sb, off_top)) {
                const uint8_t bits = (uint8_t)(quad_sides(sa) | (quad_sides(sb) << 4));
                for (int r = ra; r < rb; ++r, x += p.xstride) *x = bits;
            } else {
                // thresholds and the sides of the genes at pi/2 in registers, as in a run
                const uint32_t sp[4] = {sa.x, sa.y, sb.x, sb.y};
                uint32_t T[8], top = 0u;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const uint32_t off = (i & 1) ? (sp[i >> 1] >> 16) : (sp[i >> 1] & 0xffffu);
                    T[i] = *reinterpret_cast<const uint32_t *>(thr_bytes + off);      // 0 at both bounds
                    if (off == off_top) top |= 1u << i;
                }
                const RowKeys key = row_keys(p, (uint32_t)t);
                const QuadWords wa = quad_words(p, 2u * (uint32_t)vec, (uint32_t)t);
                const QuadWords wb = quad_words(p, 2u * (uint32_t)vec + 1u, (uint32_t)t);
#pragma unroll 2
                for (int r = ra; r < rb; ++r, x += p.xstride) {
                    const uint64_t z = row_product(key, (uint32_t)r);
                    const Draw4 d0 = quad_draw(key, wa, z), d1 = quad_draw(key, wb, z);
                    const uint32_t u[8] = {d0.a, d0.b, d0.c, d0.d, d1.a, d1.b, d1.c, d1.d};
                    uint32_t bits = top;
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        if (u[i] < T[i]) bits |= 1u << i;
                    *x = (uint8_t)bits;
                }
            }
        }
    }
}

__global__ void __launch_bounds__(kThreads) column_plane_kernel(const GenParams p, const ColParams c)
{
    __shared__ uint32_t s_thr[kMaxThr];
    load_thresholds(p, s_thr);
    grid_dependency_wait();
    __syncthreads();
    column_plane(p, c, (int)blockIdx.x, (int)gridDim.x, s_thr);
    allow_dependent_launch();
}

__device__ __forceinline__ void column_clear_words(const ColParams &c)
{
    for (int i = 0; i < 3; ++i) c.slot[i] = ColSlot{};
    for (int i = 0; i < 4; ++i) c.sync[i] = ColSync{};
}

// Sums of the items of a fixed vector's quad (32-bit item arrays; zero on padding genes).
__device__ __forceinline__ void quad_sums(const GenParams &p, int q, uint2 s, int64_t &w, int64_t &v)
{
    const int4 a = __ldg(p.w4 + q), b = __ldg(p.v4 + q);
    const int32_t wi[4] = {a.x, a.y, a.z, a.w}, vi[4] = {b.x, b.y, b.z, b.w};
    const uint32_t x = quad_sides(s);
#pragma unroll
    for (int i = 0; i < 4; ++i)
        if ((x >> i) & 1u) {
            w += wi[i];
            v += vi[i];
        }
}

// The end of a run, per vector: the CIP of its last generation into the state between runs, the
// best row (its alleles from the last generation's elite, from the alleles recorded when the
// best was found, or, for quads fixed before that, from their side), and the list the next run
// starts with; the last block advances the generation counter and clears the run's words.
// from_rows: instead, the state between runs is taken from row 0 of the full state (whose rows
// are equal), after a run in a row-by-row form or a checkpoint.
__device__ __forceinline__ void column_end(const GenParams &p, const ColParams &c, int32_t from_rows, int block,
                                           int blocks, const uint32_t *s_thr)
{
    const unsigned char *thr_bytes = reinterpret_cast<const unsigned char *>(s_thr);
    const uint32_t off_top = (uint32_t)(8 * p.K), k8 = off_top * 0x00010001u;
    for (int i = block * kThreads + threadIdx.x; i < 2 * kColPosted; i += blocks * kThreads) c.post[i] = ColSync{};
    for (int i = block * kThreads + threadIdx.x; i < 4 * kColQueues; i += blocks * kThreads) c.qctr[i] = 0u;
    const bool ran = from_rows || c.ctl[kCtlRan] != 0;
    const bool rebuild = from_rows || (ran && c.ctl[kCtlRebuild] != 0);
    const int32_t t_last = c.ctl[kCtlLast], t0 = c.ctl[kCtlFirst];
    const int32_t e = *p.elite_idx;
    const int64_t tb = p.best[1];
    const int vec = block * kThreads + threadIdx.x;
    if (ran) {
        const bool act = vec < p.svec;
        uint2 s[2] = {make_uint2(0u, 0u), make_uint2(0u, 0u)};
        uint32_t best = 0u;
        if (act) {
            for (int h = 0; h < 2; ++h) {
                const int q = 2 * vec + h;
                if (from_rows) {
                    s[h] = reinterpret_cast<const uint2 *>(p.state)[q];
                } else {
                    const uint2 o = observed_quad(c, p.svec, q, t_last, off_top);
                    const Draw4 d = philox4x32_10_rk((uint32_t)q, (uint32_t)e, (uint32_t)t_last, 0u, p.rk0, p.rk1);
                    const uint32_t x = observe_quad(d, o, thr_bytes, off_top);
                    s[h] = step_quad(o, x, k8);
                    const int2 rec = c.best_nib[q];
                    const uint32_t bx = tb == t_last ? x : rec.x == tb ? (uint32_t)rec.y : quad_sides(o);
                    best |= bx << (4 * h);
                }
                c.canon[q] = s[h];
            }
            if (!from_rows && tb >= t0) p.best_row[vec] = (uint8_t)best;
        }
        if (rebuild) {
            const bool fa = quad_fixed(s[0], off_top), fb = quad_fixed(s[1], off_top);
            int64_t fw = 0, fv = 0;
            if (act && fa) quad_sums(p, 2 * vec, s[0], fw, fv);
            if (act && fb) quad_sums(p, 2 * vec + 1, s[1], fw, fv);
            column_append(c.head, column_list(c, p.svec, 0), p.svec, act, true, 2 * vec, 2 * vec + 1, fa, fb, fw, fv);
        }
    }
    __shared__ int s_last;
    __syncthreads();
    if (threadIdx.x == 0) s_last = atom_add_acq_rel(reinterpret_cast<unsigned int *>(c.ctl + kCtlTicket), 1u) == (unsigned int)blocks - 1u ? 1 : 0;
    __syncthreads();
    if (!s_last || threadIdx.x != 0) return;
    c.ctl[kCtlTicket] = 0;
    if (from_rows) return;
    if (ran) {
        *p.gen = t_last + 1;
        *p.bar_gen = t_last + 1;
    }
    *p.ticket = 0u;
    p.keys[0] = p.keys[1] = p.keys[2] = 0ull;
    p.qctr[0] = p.qctr[1] = p.qctr[2] = 0u;
    column_clear_words(c);
    c.ctl[kCtlRebuilt] = 0;
    c.ctl[kCtlPhase] = 0;
}

__global__ void __launch_bounds__(kThreads) column_end_kernel(const GenParams p, const ColParams c, int32_t from_rows)
{
    __shared__ uint32_t s_thr[kMaxThr];
    load_thresholds(p, s_thr);
    grid_dependency_wait();
    __syncthreads();
    column_end(p, c, from_rows, (int)blockIdx.x, (int)gridDim.x, s_thr);
}

// Generation 0 of an instance that runs in the column form: the words every form shares, one row
// at pi/4, every vector on the list, no recorded best row. The full state is written if state_words
// is not 0 (column_expand_kernel makes it otherwise, when another form needs it).
__global__ void __launch_bounds__(kThreads) column_reset_kernel(const GenParams p, const ColParams c, size_t state_words,
                                                                size_t xbytes, size_t acc_words, size_t hist_words)
{
    grid_dependency_wait();
    init_words(p, state_words, xbytes, acc_words, hist_words);
    const uint32_t kk = (uint32_t)(4 * p.K) * 0x00010001u;
    const int i0 = blockIdx.x * kThreads + threadIdx.x, stride = (int)gridDim.x * kThreads;
    for (int vec = i0; vec < p.svec; vec += stride) {
        c.canon[2 * vec] = c.canon[2 * vec + 1] = make_uint2(kk, kk);
        c.best_nib[2 * vec] = c.best_nib[2 * vec + 1] = make_int2(-1, 0);
        column_list(c, p.svec, 0)[vec] = vec;
    }
    for (int i = i0; i < 2 * kColPosted; i += stride) c.post[i] = ColSync{};
    for (int i = i0; i < 4 * kColQueues; i += stride) c.qctr[i] = 0u;
    if (i0 == 0) {
        ColSlot h{};
        h.nv = (unsigned int)p.svec;
        *c.head = h;
        column_clear_words(c);
        for (int i = 0; i < 16; ++i) c.ctl[i] = 0;
    }
}

// Whether a row of the full state differs from row 0 (a checkpoint's may). Bound by memory; a host
// comparison of the checkpoint's 20 MB (1,024 x 10,000) took 1 ms of the load's 2.6.
__global__ void __launch_bounds__(kThreads) column_compare_kernel(const GenParams p, const ColParams c)
{
    grid_dependency_wait();
    const size_t total = (size_t)p.np * p.svec, stride = (size_t)gridDim.x * kThreads;
    bool differ = false;
    for (size_t i = (size_t)blockIdx.x * kThreads + threadIdx.x; i < total; i += stride) {
        const uint4 a = p.state[i], b = __ldg(p.state + i % (size_t)p.svec);
        differ = differ || a.x != b.x || a.y != b.y || a.z != b.z || a.w != b.w;
    }
    if (differ) c.ctl[kCtlDiffer] = 1;
}

// The full state from the state between runs (every row equal), for the row-by-row forms.
__global__ void __launch_bounds__(kThreads) column_expand_kernel(const GenParams p, const ColParams c)
{
    grid_dependency_wait();
    const uint4 *row = reinterpret_cast<const uint4 *>(c.canon);
    const size_t total = (size_t)p.np * p.svec, stride = (size_t)gridDim.x * kThreads;
    for (size_t i = (size_t)blockIdx.x * kThreads + threadIdx.x; i < total; i += stride)
        p.state[i] = __ldg(row + i % (size_t)p.svec);
}

template <int kForm>
struct ColObserveShared {
    uint32_t thr[kMaxThr];
    unsigned long long acc64[kForm == 2 ? 2 * kColRows : 1];
    uint32_t acc32[kForm == 2 ? 1 : 2 * kColRows];
    int32_t row[kColRows];
    int64_t fix[2];
};

// Before column_observe, whose first barrier follows.
template <int kForm>
__device__ __forceinline__ void column_observe_begin(const GenParams &p, ColObserveShared<kForm> &sh)
{
    load_thresholds(p, sh.thr);
    for (int i = threadIdx.x; i < 2 * kColRows; i += kThreads) {
        if constexpr (kForm == 2) sh.acc64[i] = 0ull;
        else sh.acc32[i] = 0u;
    }
    if (threadIdx.x < 2) sh.fix[threadIdx.x] = 0;
}

// One generation from equal rows: the alleles, fitness and best key of np rows. A block keeps one
// tile's thresholds and items for its rows, as in a run.
//   t >= 0: generation t of a row block (a population sharded by rows, whose elite is picked outside);
//     the angle indices stay as they are until column_rotate_kernel.
//   t = -1 - g: generation g of an instance's run, which column_step_kernel ends. From the second on
//     (kNext) the block first takes the generation before's CIP, toward the elite of its key: the
//     leading blocks leave the angle indices in their parity and the best row, block 0 the records.
// Bound by the integer pipes and, with 50 rows a block, by its start: 1,500 rows of 20,000 genes
// 30 us, 38 us row by row with the state read (and the rotation 2.5 us, 15 us row by row).
template <int kForm, bool kNext>
__device__ __forceinline__ void column_observe(const GenParams &p, const ColParams &c, int32_t t, int32_t part_rows,
                                               int block, int blocks, ColObserveShared<kForm> &sh)
{
    const int tid = threadIdx.x;
    __syncthreads();
    const bool step = t < 0, rec = block == 0 && tid == 0;
    const int32_t g = kNext ? -1 - t : 0;
    unsigned long long last = 0ull;               // the key and the best fitness before generation t - 1
    int64_t best = 0;
    if (step) {
        if (column_stopped(p, c, block)) return;
        // (every word that may be needed is asked for at once: one trip to L2)
        const int32_t failed = *p.error, t0 = *p.gen;
        unsigned long long k0 = 0ull, k1 = 0ull, k2 = 0ull;
        int64_t b0 = 0, b1 = 0;
        if (kNext) {
            k0 = p.keys[0];
            k1 = p.keys[1];
            k2 = p.keys[2];
            b0 = c.run_best[0];
            b1 = c.run_best[1];
        } else if (rec) {
            b0 = p.best[0];
            b1 = p.best[1];
        }
        if (failed) {                             // (no launch before this one is still running)
            if (rec) c.ctl[kCtlRan] = 0;
            return;
        }
        t = t0 + g;
        if (kNext) {
            const int32_t slot = (t + 2) % 3;
            last = slot == 0 ? k0 : slot == 1 ? k1 : k2;
            best = (t & 1) ? b0 : b1;
        }
        if (rec) {
            p.keys[(t + 1) % 3] = 0ull;           // (generation t - 2's, which nobody reads any more)
            if (!kNext) {
                // (no block of this launch reads the list's counts; column_step_kernel fills them again)
                c.ctl[kCtlRan] = 1;
                *c.head = ColSlot{};
                c.run_best[t & 1] = b1 < 0 ? INT64_MIN : b0;
            }
        }
    }
    const ColGeom m = column_geometry((uint32_t)p.svec, 0u, p.np, blocks);
    const BlockShare b = tile_geometry(m.lanes, m.warps);
    const int tile = block % m.ntile, part = block / m.ntile;
    const int r_end = (int)min((int64_t)p.np, (int64_t)(part + 1) * part_rows);
    const int vec = tile * m.width + b.v_in;
    const bool active = b.v_in < m.width && vec < p.svec;
    ColItem<kForm> it;
    it.qa = active ? 2 * vec : -1;
    it.qb = active ? 2 * vec + 1 : -1;
    it.whole = true;
    column_load<kForm>(p, it, g < 2 ? c.canon : column_parity(c, p.svec, t - 1));
    const unsigned char *thr_bytes = reinterpret_cast<const unsigned char *>(sh.thr);
    const uint32_t off_top = (uint32_t)(8 * p.K);
    uint32_t T[8], top = 0u;
    ColSum<kForm> base;
    column_thresholds<kForm>(it, thr_bytes, off_top, T, top, base);
    if (kNext) {
        const int32_t e0 = (int32_t)(0xffffffu - (uint32_t)(last & 0xffffffull)), e = e0 >= 0 && e0 < p.np ? e0 : 0;
        const int64_t f = (int64_t)(last >> 24) - kKeyBias;
        const bool improved = f > best;
        const uint32_t x = column_cip<kForm>(p, it, e, t, T, top, off_top * 0x00010001u);
        column_thresholds<kForm>(it, thr_bytes, off_top, T, top, base);
        if (part == 0 && b.r_sub == 0 && active) {
            uint2 *row = column_parity(c, p.svec, t);
            row[it.qa] = it.sa;
            row[it.qb] = it.sb;
            if (improved) p.best_row[vec] = (uint8_t)x;
        }
        if (rec) {
            c.run_best[t & 1] = improved ? f : best;
            if (e != e0) atomicOr(p.error, kErrEliteRange);
            column_record(p, t - 1, e, f, improved, 0, (uint32_t)p.svec);
        }
    }
    const RowKeys k = row_keys(p, (uint32_t)t);
    const QuadWords wa = quad_words(p, (uint32_t)it.qa, (uint32_t)t), wb = quad_words(p, (uint32_t)it.qb, (uint32_t)t);
    uint8_t *const plane = p.xbits + (size_t)(t & 1) * p.xplane + vec;
    unsigned long long *const key = p.keys + t % 3;
    for (int ra = part * part_rows; ra < r_end; ra += kColRows) {
        const int n = min(kColRows, r_end - ra);
        if (tid < n) sh.row[tid] = ra + tid;
#pragma unroll 2
        for (int q = b.r_sub; q < n + b.r_sub; q += m.rpp) {         // the same trips for every thread
            const uint64_t z = row_product(k, (uint32_t)(p.row0 + ra + q));
            const Draw4 d0 = quad_draw(k, wa, z), d1 = quad_draw(k, wb, z);
            const uint32_t u[8] = {d0.a, d0.b, d0.c, d0.d, d1.a, d1.b, d1.c, d1.d};
            ColSum<kForm> s = column_sum<kForm>(it, T, base, u, c.one);
            uint32_t bits = top;
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (u[i] < T[i]) bits |= 1u << i;
            if (active && q < n) plane[(size_t)(ra + q) * p.xstride] = (uint8_t)bits;
            if (m.lanes == 32) {
                s = column_warp_sum<kForm>(s);
            } else {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    if (o < m.lanes) {
                        if constexpr (kForm == 2) {
                            s.w += __shfl_xor_sync(0xffffffffu, s.w, o);
                            s.v += __shfl_xor_sync(0xffffffffu, s.v, o);
                        } else {
                            s.a += __shfl_xor_sync(0xffffffffu, s.a, o);
                            if constexpr (kForm == 1) s.b += __shfl_xor_sync(0xffffffffu, s.b, o);
                        }
                    }
                }
            }
            if (b.leader && q < n) column_add<kForm>(s, q, sh.acc32, sh.acc64);
        }
        column_flush<kForm>(p, c.sum_bits, m.ntile, sh.row, n, sh.fix, key, sh.acc32, sh.acc64);
    }
    // the generation counter then names the next generation, as after a run
    if (!step && rec) *p.gen = t + 1;
}

template <int kForm, bool kNext>
__global__ void __launch_bounds__(kThreads, 2) column_observe_kernel(const GenParams p, const ColParams c, int32_t t,
                                                                     int32_t part_rows)
{
    __shared__ ColObserveShared<kForm> sh;
    column_observe_begin(p, sh);
    grid_dependency_wait();
    column_observe<kForm, kNext>(p, c, t, part_rows, (int)blockIdx.x, (int)gridDim.x, sh);
    allow_dependent_launch();
}

// Ends a run of column_observe_kernel's generations, of which g is the last: its elite from its key, CIP
// of the one row, the best row if it improved, the list the next run starts with, and by the
// last block the records. (When a run is worth these launches: see step_run.)
__device__ __forceinline__ void column_step(const GenParams &p, const ColParams &c, int32_t g, int block, int blocks,
                                            const uint32_t *s_thr)
{
    __shared__ int s_last;
    const unsigned char *thr_bytes = reinterpret_cast<const unsigned char *>(s_thr);
    const uint32_t off_top = (uint32_t)(8 * p.K), k8 = off_top * 0x00010001u;
    // (every word that may be needed is asked for at once: one trip to L2)
    const int32_t ran = c.ctl[kCtlRan], t = *p.gen + g, slot = t % 3;
    const unsigned long long k0 = p.keys[0], k1 = p.keys[1], k2 = p.keys[2], key = slot == 0 ? k0 : slot == 1 ? k1 : k2;
    const int64_t best_f = p.best[0], best_t = p.best[1];
    if (ran == 0) return;                         // (stopped by convergence)
    const uint2 *state = g == 0 ? c.canon : column_parity(c, p.svec, t);
    const int32_t e0 = (int32_t)(0xffffffu - (uint32_t)(key & 0xffffffull)), e = e0 >= 0 && e0 < p.np ? e0 : 0;
    const int64_t f = (int64_t)(key >> 24) - kKeyBias;
    const bool improved = best_t < 0 || f > best_f;
    const int vec = block * kThreads + threadIdx.x;
    const bool act = vec < p.svec;
    uint2 s[2] = {make_uint2(0u, 0u), make_uint2(0u, 0u)};
    uint32_t bits = 0u;
    if (act) {
        for (int h = 0; h < 2; ++h) {
            const int q = 2 * vec + h;
            const uint2 o = state[q];
            const Draw4 d = philox4x32_10_rk((uint32_t)q, (uint32_t)e, (uint32_t)t, 0u, p.rk0, p.rk1);
            const uint32_t x = observe_quad(d, o, thr_bytes, off_top);
            s[h] = step_quad(o, x, k8);
            c.canon[q] = s[h];
            bits |= x << (4 * h);
        }
        if (improved) p.best_row[vec] = (uint8_t)bits;
    }
    const bool fa = quad_fixed(s[0], off_top), fb = quad_fixed(s[1], off_top);
    int64_t fw = 0, fv = 0;
    if (act && fa) quad_sums(p, 2 * vec, s[0], fw, fv);
    if (act && fb) quad_sums(p, 2 * vec + 1, s[1], fw, fv);
    column_append(c.head, column_list(c, p.svec, 0), p.svec, act, true, 2 * vec, 2 * vec + 1, fa, fb, fw, fv);
    __syncthreads();
    if (threadIdx.x == 0) s_last = atom_add_acq_rel(reinterpret_cast<unsigned int *>(c.ctl + kCtlTicket), 1u) == (unsigned int)blocks - 1u ? 1 : 0;
    __syncthreads();
    if (!s_last || threadIdx.x != 0) return;
    c.ctl[kCtlTicket] = 0;
    if (e != e0) atomicOr(p.error, kErrEliteRange);
    int32_t run = 0;
    if (p.converge) {
        const int32_t before = t > 0 ? p.conv[(t - 1) & 1] : 0;
        run = before > 0 && f == p.hist_f[t - 1] ? before + 1 : 1;
        if (run >= kConvergeWindow) {
            p.conv[3] = t;
            p.conv[2] = kStopped;
        }
    }
    column_record(p, t, e, f, improved, run, (uint32_t)p.svec);      // (column_observe_kernel draws every vector)
    *p.gen = t + 1;
    *p.bar_gen = t + 1;
    p.keys[0] = p.keys[1] = p.keys[2] = 0ull;
}

__global__ void __launch_bounds__(kThreads) column_step_kernel(const GenParams p, const ColParams c, int32_t g)
{
    __shared__ uint32_t s_thr[kMaxThr];
    load_thresholds(p, s_thr);
    grid_dependency_wait();
    __syncthreads();
    column_step(p, c, g, (int)blockIdx.x, (int)gridDim.x, s_thr);
}

// CIP of a row block with equal rows toward an elite row supplied from outside: bytes of 0 or 1,
// 8 a vector.
__global__ void __launch_bounds__(kThreads) column_rotate_kernel(const GenParams p, const ColParams c, const uint2 *elite)
{
    const uint32_t k8 = (uint32_t)(8 * p.K) * 0x00010001u;
    const int vec = (int)(blockIdx.x * kThreads + threadIdx.x);
    if (vec >= p.svec) return;
    const uint2 e = elite[vec];
    const auto nib = [](uint32_t w) { return (w & 1u) | (w >> 7 & 2u) | (w >> 14 & 4u) | (w >> 21 & 8u); };
    c.canon[2 * vec] = step_quad(c.canon[2 * vec], nib(e.x), k8);
    c.canon[2 * vec + 1] = step_quad(c.canon[2 * vec + 1], nib(e.y), k8);
}

// Many instances in one launch (batches, a server's steps). The members do not depend on one
// another, so each has its own blocks for the whole run: a list of tasks per block, where a member
// that is worth several blocks comes first on them and small members follow one another on one
// block (see plan_column_batch, which cuts the blocks so that all end at about the same time).
// A member's short list stays with its blocks (column_run's kMember: there is no hand-over to
// column_small_kernel, whose shorter chain matters less where other members fill the SM).
//
// Bound by the integer pipes like column_run_kernel; the blocks' ends spread over the last third of
// the run, since a member gets whole blocks. 96 members (50 to 20,000 genes, 32 to 512 rows),
// 200 generations with the resets and the results read back: 7.7 ms, 5.3 of them in this kernel;
// 21.6 ms in the row-by-row form, whose members share every generation's launch.
struct ColMember {
    GenParams p;
    ColParams c;
};

struct ColTask {
    int32_t member;
    int32_t block, blocks;        // of the member's blocks
    int32_t gens;                 // most generations of this run (column_batch_observe_kernel: rows a block)
};

// A member's words in shared memory (whole block).
__device__ __forceinline__ void load_member(ColMember &s_m, const ColMember *m)
{
    static_assert(sizeof(ColMember) % 4 == 0, "copied by words");
    __syncthreads();
    for (int i = threadIdx.x; i < (int)(sizeof(ColMember) / 4); i += kThreads)
        reinterpret_cast<uint32_t *>(&s_m)[i] = __ldg(reinterpret_cast<const uint32_t *>(m) + i);
    __syncthreads();
}

// Every generation of the members' runs in one cooperative launch: block b's tasks are
// [first[b], first[b + 1]).
template <int kForm>
__global__ void __launch_bounds__(kThreads, 2) column_batch_kernel(const ColMember *members, const ColTask *tasks,
                                                                   const int32_t *first, int32_t G)
{
    __shared__ ColMember s_m;
    __shared__ ColRunShared<kForm> sh;
    for (int i = first[blockIdx.x]; i < first[blockIdx.x + 1]; ++i) {
        const ColTask k = tasks[i];
        load_member(s_m, members + k.member);
        column_run<kForm, true>(s_m.p, s_m.c, min(G, k.gens), k.block, k.blocks, sh);
    }
}

// A run of one generation, task by task: column_observe and column_step (see qieo_batch_run for when).
template <int kForm>
__global__ void __launch_bounds__(kThreads, 2) column_batch_observe_kernel(const ColMember *members, const ColTask *tasks)
{
    __shared__ ColMember s_m;
    __shared__ ColObserveShared<kForm> sh;
    grid_dependency_wait();
    const ColTask k = tasks[blockIdx.x];
    load_member(s_m, members + k.member);
    column_observe_begin(s_m.p, sh);
    column_observe<kForm, false>(s_m.p, s_m.c, -1, k.gens, k.block, k.blocks, sh);
}

__global__ void __launch_bounds__(kThreads) column_batch_step_kernel(const ColMember *members, const ColTask *tasks)
{
    __shared__ ColMember s_m;
    __shared__ uint32_t s_thr[kMaxThr];
    grid_dependency_wait();
    const ColTask k = tasks[blockIdx.x];
    load_member(s_m, members + k.member);
    load_thresholds(s_m.p, s_thr);
    __syncthreads();
    column_step(s_m.p, s_m.c, 0, k.block, k.blocks, s_thr);
}

// column_plane_kernel and column_end_kernel for every member, task by task. (A plane task of no blocks
// only clears the head: a server's solves have no use for the plane.)
__global__ void __launch_bounds__(kThreads) column_batch_plane_kernel(const ColMember *members, const ColTask *tasks)
{
    __shared__ ColMember s_m;
    __shared__ uint32_t s_thr[kMaxThr];
    grid_dependency_wait();
    const ColTask k = tasks[blockIdx.x];
    load_member(s_m, members + k.member);
    load_thresholds(s_m.p, s_thr);
    __syncthreads();
    column_plane(s_m.p, s_m.c, k.block, k.blocks, s_thr);
}

__global__ void __launch_bounds__(kThreads) column_batch_end_kernel(const ColMember *members, const ColTask *tasks)
{
    __shared__ ColMember s_m;
    __shared__ uint32_t s_thr[kMaxThr];
    grid_dependency_wait();
    const ColTask k = tasks[blockIdx.x];
    load_member(s_m, members + k.member);
    load_thresholds(s_m.p, s_thr);
    __syncthreads();
    column_end(s_m.p, s_m.c, 0, k.block, k.blocks, s_thr);
}

}  // namespace qieo
