// crk_pass.cuh -- warp-per-tile skeleton of the pair passes.
//
// One warp owns one i-tile (lane = particle i of 32 consecutive sorted
// particles) and walks the tile's interaction list.  Each neighbour tile J is
// staged once in shared memory (lane l loads record J*32+l, coalesced) and
// every lane then loops over the 32 staged records, testing the exact
// fixed-point predicate and accumulating in registers.  No atomics, no
// inter-warp synchronisation: results are deterministic.
#pragma once

#include "crk_internal.cuh"

#include <type_traits>

namespace crk {

struct PassGeom {
    int n;
    int ntiles;
    const uint2 *ofs;        // per i-tile (offset, count) into list
    const uint32_t *list;    // neighbour tile ids
    unsigned long long *pairs;  // optional pair counter
};

// P must provide: Params, JRec, IState,
//   init(IState&, int i, bool valid, const Params&)
//   stage(JRec&, int j, const Params&)
//   pair(IState&, const JRec&, int j, int i, bool valid, const Params&)
//   finish(IState&, int i, const Params&)           (valid lanes only)
//   count(const IState&) -> pairs of this lane
template <class P, int WARPS>
__global__ void __launch_bounds__(WARPS * 32) k_pass(PassGeom g, typename P::Params prm) {
    grid_wait();
    __shared__ typename P::JRec sj[WARPS][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int tile = blockIdx.x * WARPS + w;
    if (tile >= g.ntiles) return;
    const int i = tile * TILE + lane;
    const bool valid = i < g.n;
    typename P::IState st;
    P::init(st, i, valid, prm);
    const uint2 lo = g.ofs[tile];
    for (uint32_t t = 0; t < lo.y; t++) {
        const int J = (int)g.list[lo.x + t];
        const int j0 = J * TILE;
        const int cnt = min(TILE, g.n - j0);
        __syncwarp();
        if (lane < cnt) P::stage(sj[w][lane], j0 + lane, prm);
        __syncwarp();
        for (int jj = 0; jj < cnt; jj++) P::pair(st, sj[w][jj], j0 + jj, i, valid, prm);
    }
    if (valid) P::finish(st, i, prm);
    if (g.pairs) {
        unsigned c = valid ? (unsigned)P::count(st) : 0u;
        c = __reduce_add_sync(0xffffffffu, c);
        if (lane == 0 && c) atomicAdd(g.pairs, (unsigned long long)c);
    }
}

template <class P, int WARPS>
int launch_pass(crk_ctx *ctx, int prof_id, bool union_list, const typename P::Params &prm,
                unsigned long long *pairs, cudaStream_t s, const char *what) {
    if (ctx->n == 0) return CRK_OK;
    PassGeom g;
    g.n = ctx->n;
    g.ntiles = ctx->ntiles;
    g.ofs = union_list ? ctx->uofs : ctx->gofs;
    g.list = union_list ? ctx->ulist : ctx->glist;
    g.pairs = pairs;
    prof_begin(ctx, prof_id, s);
    launch(s, grid_for(ctx->ntiles, WARPS), WARPS * 32, 0, k_pass<P, WARPS>, g, prm);
    ++ctx->launches;
    prof_end(ctx, s);
    CRK_LAUNCH_CHECK(ctx, what);
    return CRK_OK;
}

// Pair-sum accumulator: plain FP32, or Kahan-compensated (precision mode 1),
// whose error stays near one rounding of the final sum however much the terms
// cancel (the odd moments and grad m1 = delta m0 + sum V x grad W do).
template <bool COMP>
struct Acc {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void add(float v) {
        if (COMP) {
            float y = v - c;
            float t = s + y;
            c = (t - s) - y;
            s = t;
        } else {
            s += v;
        }
    }
    __device__ __forceinline__ float value() const { return COMP ? s - c : s; }
};

// ---------------------------------------------------------------- list passes



// Per-particle lists.  A tile has kcap columns of 32 lanes, stored as blocks of
// four columns: a lane's four entries of a block are 16 contiguous bytes and a
// block is 512, so a warp reads a block in one coalesced 128-bit load per lane,
// and the walk writes 16 bytes at a time.  Gather neighbours fill blocks from
// the front, the other pair-set neighbours fill blocks from the back; a lane
// pads the last block of either segment with its own index i.  A pair (i, i)
// adds exactly zero to every sum of differences (x = 0, v_i - v_j = 0, F_ii = 0);
// the passes whose self term is not zero (W(0)) get `ok` = false for a pad.
constexpr int LB = 4;   // entries of a block

__host__ __device__ __forceinline__ int list_blocks(int entries) { return (entries + LB - 1) / LB; }

// word of a lane's column 0 of block b within its tile's columns
__device__ __forceinline__ size_t block_at(int b, int lane) { return ((size_t)b * 32 + lane) * LB; }

// Block b of the pair-set sequence of a lane with nbg gather blocks: its
// gather blocks, then the others from the tile's last block down.
__device__ __forceinline__ int pair_block(int b, int nbg, int kcap) { return b < nbg ? b : kcap / LB - 1 - (b - nbg); }

// Warp per tile, lane = particle i; lane i walks its own list, block by block.
// Gather passes walk the gather blocks, pair-set passes all blocks; entry u of
// block b has its stored force (P4 -> P5) in row 4 b + u of the tile, pads
// included (F = 0, j = i).  P must provide Params, IState, Rec, GATHER,
// PREFETCH, UNROLL, PERSISTENT, ENTRIES (false: the pass reads only its stored
// entries, and `entry` is passed as 0),
//   init(IState&, int i, bool valid, const Params&)
//   load(uint32_t entry, size_t pos, const Params&) -> Rec   (the neighbour's data)
//   pair(IState&, const Rec&, uint32_t entry, size_t pos, bool ok, const Params&)
//   finish(IState&, int i, const Params&)            (valid lanes only)
struct ListGeom {
    int n, ntiles, kcap;
    const uint32_t *fbase;             // per-tile stored-force base, units of 32 entries
    const uint32_t *len_g, *len_u;     // per-tile rows of the longest lane (multiples of LB)
    const int32_t *cnt_g, *cnt_u;
    const uint32_t *ent;
    const unsigned long long *heavy;   // set: tiles with more pair-set rows than *heavy are left to the split form
};

// A tile with more rows than HEAVY_ROWS and than one and a half times the mean tile's
// (CNT_LONG_ROWS) is shared by the warps of a CTA: a warp that walks the 1000 to
// 2000 neighbours of a particle in an evacuated region runs on alone when the
// others are done.  P1 to P5 of Sedov 64^3 after 500 steps (mean 320 entries, longest
// 1460): no tile shared 2.90 ms, beyond 576 rows and 1, 1.25, 1.5, 2, 2.5, 3 means
// 2.49, 2.48, 2.49, 2.49, 2.54, 2.78; beyond 1.5 means and 384 to 800 rows within 1%.
// (Clustered 64^3 after 60 steps, longest lists milder: 2.33 unshared, 2.42 at 1.5.)
// Where all lists are long the warps are even, and sharing every tile only costs:
// 80^3 with 600 neighbours each 6.76 ms, 9.15 with a fixed line of 576.
constexpr int HEAVY_ROWS = 576;

// The blocks of lists stream once from HBM (or L2, just written by the walk),
// the longest latency of the loop, so the next block is always read ahead.
// Passes with 16-32-byte records (mostly L1 hits) gather U neighbours' records
// at a time (U = 1, 2 or 4; 4 is the measured best).  P4, whose record already
// fills the registers, evaluates one pair at a time with the next record in
// flight (P::PREFETCH), alternating two register sets (measured 7% faster than
// copying the prefetched record into the current one).
// passes that declare SKIPPABLE take a device flag (Params::skip, may be null)
template <class P, class = void>
struct has_skip : std::false_type {};
template <class P>
struct has_skip<P, std::void_t<decltype(P::SKIPPABLE)>> : std::bool_constant<P::SKIPPABLE> {};

// passes that declare NOTUNE run their own loop form only (no autotuner variants)
template <class P, class = void>
struct has_notune : std::false_type {};
template <class P>
struct has_notune<P, std::void_t<decltype(P::NOTUNE)>> : std::bool_constant<P::NOTUNE> {};

template <class P>
__device__ __forceinline__ bool pass_skipped(const typename P::Params &prm) {
    if constexpr (has_skip<P>::value) return prm.skip && *(volatile const unsigned long long *)prm.skip;
    return false;
}

// What a lane reads ahead for a block: its four list entries (P::ENTRIES), or,
// for a pass that reads only what an earlier pass stored per entry, those four
// stored records (P::Stored, from P::stored(pos)), which then stream from HBM.
template <class P, bool = P::ENTRIES>
struct BlockOf {
    uint32_t e[LB];
};
template <class P>
struct BlockOf<P, false> {
    typename P::Stored e[LB];
};

// One lane's list: where its blocks are and how many it has.
template <class P>
struct LaneList {
    const uint32_t *tile_ent;   // the tile's columns
    size_t fb;                  // stored-force position of row 0
    int lane, kcap, mg, nbg, nb;
    __device__ __forceinline__ LaneList(const ListGeom &g, int tile, int lane_, int i, bool valid) {
        lane = lane_;
        kcap = g.kcap;
        tile_ent = g.ent + (size_t)tile * g.kcap * 32;
        fb = (size_t)g.fbase[tile] * 32 + lane;
        // counts beyond kcap only occur in a walk that overflowed (the host then
        // grows kcap and walks again, or discards a replayed step): never read
        // past the tile's columns
        const int all = g.kcap / LB;
        mg = valid ? min(g.cnt_g[i], g.kcap) : 0;
        nbg = list_blocks(mg);
        nb = P::GATHER ? nbg : (valid ? min(nbg + list_blocks(max(g.cnt_u[i] - g.cnt_g[i], 0)), all) : 0);
    }
    __device__ __forceinline__ BlockOf<P> fetch(int b, const typename P::Params &prm) const {
        BlockOf<P> r;
        if constexpr (P::ENTRIES) {
            const int c = P::GATHER ? b : pair_block(b, nbg, kcap);
            const uint4 v = __ldg(reinterpret_cast<const uint4 *>(tile_ent + block_at(c, lane)));
            r.e[0] = v.x;
            r.e[1] = v.y;
            r.e[2] = v.z;
            r.e[3] = v.w;
        } else {
#pragma unroll
            for (int u = 0; u < LB; u++) r.e[u] = P::stored(fb + (size_t)(LB * b + u) * 32, prm);
        }
        return r;
    }
    // entry u of block b is a neighbour, not a pad (gather passes)
    __device__ __forceinline__ bool ok(int b, int u) const { return LB * b + u < mg; }
};

// Blocks [b0, b1) of this lane, the warp looping over [b0, bw): U independent
// gathers and pair evaluations in flight per lane and the next block read ahead.
template <class P, int U>
__device__ __forceinline__ void list_loop(typename P::IState &st, const typename P::Params &prm,
                                          const LaneList<P> &ll, int b0, int b1, int bw) {
    BlockOf<P> en = {};
    if (b0 < b1) en = ll.fetch(b0, prm);
    for (int b = b0; b < bw; b++) {
        const BlockOf<P> ec = en;
        if (b + 1 < b1) en = ll.fetch(b + 1, prm);
        if (b < b1) {
            const size_t pos = ll.fb + (size_t)b * (LB * 32);
#pragma unroll
            for (int q = 0; q < LB; q += U) {
                typename P::Rec r[U];
#pragma unroll
                for (int u = 0; u < U; u++) r[u] = P::load(ec.e[q + u], pos + 32 * (q + u), prm);
#pragma unroll
                for (int u = 0; u < U; u++)
                    P::pair(st, r[u], ec.e[q + u], pos + 32 * (q + u), ll.ok(b, q + u), prm);
            }
        }
    }
}

// list_loop with the neighbour records ahead as well (RP variants): while the
// U pairs of one group are evaluated the records of the next group are in
// flight, so a record that misses L1 is waited for only if it takes longer
// than a whole group.  Same entries, same order: bitwise the same sums.
template <class P, int U>
__device__ __forceinline__ void list_loop_rp(typename P::IState &st, const typename P::Params &prm,
                                             const LaneList<P> &ll, int b0, int b1, int bw) {
    BlockOf<P> ec = {}, en = {};
    typename P::Rec rc[U] = {};
    if (b0 < b1) {
        ec = ll.fetch(b0, prm);
#pragma unroll
        for (int u = 0; u < U; u++) rc[u] = P::load(ec.e[u], ll.fb + (size_t)b0 * (LB * 32) + 32 * u, prm);
    }
    if (b0 + 1 < b1) en = ll.fetch(b0 + 1, prm);
    for (int b = b0; b < bw; b++) {
        if (b < b1) {
            const size_t pos = ll.fb + (size_t)b * (LB * 32);
#pragma unroll
            for (int q = 0; q < LB; q += U) {
                typename P::Rec rn[U] = {};
#pragma unroll
                for (int u = 0; u < U; u++) {
                    if (q + U < LB)
                        rn[u] = P::load(ec.e[(q + U + u) % LB], pos + 32 * (q + U + u), prm);
                    else if (b + 1 < b1)
                        rn[u] = P::load(en.e[u], pos + LB * 32 + 32 * u, prm);
                }
#pragma unroll
                for (int u = 0; u < U; u++)
                    P::pair(st, rc[u], ec.e[q + u], pos + 32 * (q + u), ll.ok(b, q + u), prm);
#pragma unroll
                for (int u = 0; u < U; u++) rc[u] = rn[u];
            }
        }
        ec = en;
        if (b + 2 < b1) en = ll.fetch(b + 2, prm);
    }
}

template <class P, int U, bool RP = false>
__device__ __forceinline__ void lpass_tile(const ListGeom &g, const typename P::Params &prm, int tile, int lane) {
    if (pass_skipped<P>(prm)) return;   // the sums were formed by an earlier pass
    if (g.heavy && g.len_u[tile] > *g.heavy) return;
    const int i = tile * TILE + lane;
    const bool valid = i < g.n;
    typename P::IState st;
    P::init(st, i, valid, prm);
    const LaneList<P> ll(g, tile, lane, i, valid);
    const int bw = (int)((P::GATHER ? g.len_g[tile] : g.len_u[tile]) / LB);
    if constexpr (!P::PREFETCH) {
        if constexpr (RP)
            list_loop_rp<P, U>(st, prm, ll, 0, ll.nb, bw);
        else
            list_loop<P, U>(st, prm, ll, 0, ll.nb, bw);
    } else {
        // one pair at a time with the next record in flight, in alternating
        // register sets, so no record is copied from one to the other
        BlockOf<P> e = {};
        typename P::Rec ra{}, rb{};
        if (ll.nb > 0) {
            e = ll.fetch(0, prm);
            ra = P::load(e.e[0], ll.fb, prm);
        }
        for (int b = 0; b < bw; b++) {
            if (b < ll.nb) {
                const size_t pos = ll.fb + (size_t)b * (LB * 32);
                BlockOf<P> en = e;
                if (b + 1 < ll.nb) en = ll.fetch(b + 1, prm);
                rb = P::load(e.e[1], pos + 32, prm);
                P::pair(st, ra, e.e[0], pos, true, prm);
                ra = P::load(e.e[2], pos + 64, prm);
                P::pair(st, rb, e.e[1], pos + 32, true, prm);
                rb = P::load(e.e[3], pos + 96, prm);
                P::pair(st, ra, e.e[2], pos + 64, true, prm);
                ra = P::load(en.e[0], pos + 128, prm);   // past the last block: this block's first record again
                P::pair(st, rb, e.e[3], pos + 96, true, prm);
                e = en;
            }
        }
    }
    if (valid) P::finish(st, i, prm);
}

// Grid form: warp w of block b takes tile order[b WARPS + w] (order null:
// tiles in Morton order).
template <class P, int WARPS, int U, bool RP = false>
__global__ void __launch_bounds__(WARPS * 32) k_lpass(ListGeom g, typename P::Params prm, const int32_t *order) {
    grid_wait();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int t = blockIdx.x * WARPS + w;
    if (t >= g.ntiles) return;
    lpass_tile<P, U, RP>(g, prm, order ? order[t] : t, lane);
}

// Persistent form (one warp per block, as many blocks as fit at once): SM s
// owns the contiguous tile range [s chunk, (s+1) chunk) and its warps claim
// tiles from it in order with an atomic counter, so the warps resident on one
// SM work on neighbouring tiles, whose neighbour records they share in L1.  A
// warp whose range is exhausted claims tiles from the other ranges.  Every
// claim is one atomicAdd; a range's counter runs past chunk at most once per
// warp, so the loop is bounded.
template <class P, int U, bool RP = false>
__global__ void __launch_bounds__(32) k_lpass_sm(ListGeom g, typename P::Params prm, uint32_t *next, int nrange,
                                                 int chunk) {
    grid_wait();
    const int lane = threadIdx.x & 31;
    unsigned smid;
    asm volatile("mov.u32 %0, %%smid;" : "=r"(smid));
    const int home = (int)(smid % (unsigned)nrange);
    for (int r = 0; r < nrange; r++) {
        const int range = (home + r) % nrange;
        for (;;) {
            uint32_t t = 0;
            if (lane == 0) t = atomicAdd(&next[range], 1u);
            t = __shfl_sync(0xffffffffu, t, 0);
            if (t >= (uint32_t)chunk) break;
            const long long tile = (long long)range * chunk + t;
            if (tile >= g.ntiles) break;
            lpass_tile<P, U, RP>(g, prm, (int)tile, lane);
        }
    }
}

// Split form, for passes over few tiles (small boxes; time bins: the leaves
// ending a step at a deep level): S warps share one tile, warp w walking one
// contiguous range of every lane's blocks, so a tile's pairs take 1/S of the
// time of one warp walking them all.  Warps w > 0 start from empty sums
// (P::zero) and leave them in shared memory (P::sums); warp 0 adds them in warp
// order (P::merge, deterministic) and finishes.  The stored forces of P4 go to
// the same rows as in the other forms; the sums differ from them by rounding.
template <class P>
constexpr int split_warps() {   // as many as their sums fit static shared memory (48 KB)
    return (7 * 32 * sizeof(typename P::Sums) <= 44 * 1024) ? 8
           : ((3 * 32 * sizeof(typename P::Sums) <= 44 * 1024) ? 4 : 2);
}

// Blocks of the split form per SM that the compiler is told to leave registers for
// (0: its own choice).  With 16 warps' worth it keeps more of a block's records in
// flight, which P4, the float-float P2 and the density pass gain from (44^3 P4 383 -> 376 us,
// 40^3 P2 546 -> 518, 24^3 density 22 -> 19) and P3 and P5 lose by (48^3 119 -> 135, 134 -> 146).
template <class P, class = void>
struct split_blocks : std::integral_constant<int, 0> {};
template <class P>
struct split_blocks<P, std::void_t<decltype(P::SPLIT_WARPS)>>
    : std::integral_constant<int, P::SPLIT_WARPS / split_warps<P>()> {};

// One tile, by the S warps of the block.
template <class P, int S, int U>
__device__ __forceinline__ void split_tile(const ListGeom &g, const typename P::Params &prm, int tile, int lane, int w,
                                           typename P::Sums *part) {
    const int i = tile * TILE + lane;
    const bool valid = i < g.n;
    typename P::IState st;
    P::init(st, i, valid, prm);
    if (w > 0) P::zero(st);
    const LaneList<P> ll(g, tile, lane, i, valid);
    const int bw = (int)((P::GATHER ? g.len_g[tile] : g.len_u[tile]) / LB);
    const int chunk = (bw + S - 1) / S;
    const int b0 = w * chunk, b1 = min(bw, b0 + chunk);
    list_loop<P, U>(st, prm, ll, b0, min(ll.nb, b1), b1);
    if (w > 0) part[(w - 1) * 32 + lane] = P::sums(st);
    __syncthreads();
    if (w == 0) {
#pragma unroll 1
        for (int v = 1; v < S; v++) P::merge(st, part[(v - 1) * 32 + lane]);
        if (valid) P::finish(st, i, prm);
    }
}

// Block b takes tile order[b] (order null: tile b).
template <class P, int S, int U>
__global__ void __launch_bounds__(S * 32, split_blocks<P>::value)
k_lpass_split(ListGeom g, typename P::Params prm, const int32_t *order) {
    grid_wait();
    __shared__ __align__(16) unsigned char part[(S - 1) * 32 * sizeof(typename P::Sums)];
    if (pass_skipped<P>(prm)) return;
    split_tile<P, S, U>(g, prm, order ? order[blockIdx.x] : (int)blockIdx.x, threadIdx.x & 31, threadIdx.x >> 5,
                        reinterpret_cast<typename P::Sums *>(part));
}

// The blocks share those of the tiles listed[0 .. *count) that have more than
// *g.heavy rows, looking at 32 of them at a time.  As few blocks run as there are long
// tiles, so each needs its loads in flight more than neighbours: with registers for 16
// warps an SM, Sedov 64^3 after 250 plain steps P2 84 -> 59 us, P3 73 -> 37, P4 120 -> 104,
// P5 57 -> 38.
template <class P, int S, int U>
__global__ void __launch_bounds__(S * 32, 16 / S) k_lpass_long(ListGeom g, typename P::Params prm, const int32_t *listed,
                                                       const unsigned long long *count) {
    grid_wait();
    __shared__ __align__(16) unsigned char part[(S - 1) * 32 * sizeof(typename P::Sums)];
    if (pass_skipped<P>(prm)) return;
    const int lane = threadIdx.x & 31, end = (int)*count;
    for (int t0 = blockIdx.x; t0 < end; t0 += 32 * gridDim.x) {
        const int t = t0 + lane * (int)gridDim.x, mine = t < end ? listed[t] : 0;
        unsigned todo = __ballot_sync(0xffffffffu, t < end && g.len_u[mine] > *g.heavy);
        for (; todo; todo &= todo - 1u) {
            split_tile<P, S, U>(g, prm, __shfl_sync(0xffffffffu, mine, __ffs(todo) - 1), lane, threadIdx.x >> 5,
                                reinterpret_cast<typename P::Sums *>(part));
            __syncthreads();   // `part` is free for the next tile
        }
    }
}

// Tiles per SM below which a pass splits them: a warp per tile then leaves the
// SMs short of warps, or the last wave of warps nearly empty.  P1 to P5 together,
// us, a warp per tile (long lists by CTAs) / split:
//   jittered lattice, tiles per SM   8: 449/326   15: 643/558   26: 924/894   38: 1276/1286
//   Sedov after 400 to 500 steps    13: 1112/658  23: 1360/1035 36: 1888/1541
//                                   54: 2494/2252 105: 3937/3982
// On an even lattice the passes cross one by one, P2 and P3 from 10 to 15 tiles per SM
// (at 26: 144/158 and 113/141, P4 500/426); a run leaves that state within a few
// steps, and then a line of 10 to 25 for P1 to P3 costs 4% of the whole step at 23.
constexpr int SPLIT_TILES = 40;

// merge a partial pair sum into another (the compensated sum keeps the
// partial's correction term)
template <bool C>
__device__ __forceinline__ void merge_acc(Acc<C> &d, const Acc<C> &o) {
    d.add(o.s);
    if (C) d.add(-o.c);
}

// ---------------------------------------------------------------- autotuner
//
// Variants of a list pass: the loop form (U pairs per iteration for the small
// records; U is 1 for P4's prefetching loop) and the order tiles are taken in
// (Morton in the grid; contiguous per-SM ranges in the persistent form;
// longest list first in the grid).  Every variant visits each particle's list
// in the same order, so all give bitwise identical results; the tuner times
// each once on the first evaluation after crk_autotune(ctx, 1) and keeps the
// fastest per pass.  A set below SPLIT_TILES tiles per SM has one form whatever
// the variant: that one is timed and the default reported (TUNED_SPLIT), and the
// first evaluation above the line still sweeps.
enum { TUNED = 1, TUNED_SPLIT = 2 };   // crk_ctx::tune_done (0: not tuned)
enum { ORD_GRID = 0, ORD_SM = 1, ORD_LONGEST = 2 };
struct LVariant {
    int U, ord;
    int warps;   // tiles per CTA in the grid form (32 particles each); 0 = the pass's own
    bool rp;     // records one iteration ahead (list_loop_rp)
    bool tma;    // records brought into shared memory by TMA gathers (passes with P::TMA)
};
// 0-3: grid, U = 1..4; 4-7: longest first, U = 1..4; 8: per-SM ranges;
// 9-12: grid with the pass's own U and CTAs of 1, 2, 4, 8 tiles (32-256 particles);
// 13-16: grid, U = 1..4, records one iteration ahead, CTAs of one tile;
// 17-20: the same with the pass's own CTA width (passes without their own
// record prefetch: all but P4); 21: records by TMA gathers (P4); 22: per-SM
// ranges with the pass's own U and records one iteration ahead (all but P4)
__host__ __device__ constexpr LVariant lvariant(int v) {
    return v < 4 ? LVariant{v + 1, ORD_GRID, 0, false, false}
                 : (v < 8 ? LVariant{v - 3, ORD_LONGEST, 0, false, false}
                          : (v == 8 ? LVariant{1, ORD_SM, 0, false, false}
                                    : (v < 13 ? LVariant{0, ORD_GRID, 1 << (v - 9), false, false}
                                              : (v < 17 ? LVariant{v - 12, ORD_GRID, 1, true, false}
                                                        : (v < 21 ? LVariant{v - 16, ORD_GRID, 0, true, false}
                                                                  : (v == 21 ? LVariant{1, ORD_GRID, 0, false, true}
                                                                             : LVariant{0, ORD_SM, 0, true, false}))))));
}

// passes with a TMA-fed variant (21)
template <class P, class = void>
struct has_tma : std::false_type {};
template <class P>
struct has_tma<P, std::void_t<decltype(P::TMA)>> : std::bool_constant<P::TMA> {};

int tile_order_by_length(crk_ctx *ctx, cudaStream_t s);   // ctx->tile_order, longest pair-set list first

template <class P, int WARPS, int U>
static int launch_variant_u(crk_ctx *ctx, const ListGeom &g, const typename P::Params &prm, int ord,
                             cudaStream_t s) {
    if (ord == ORD_SM) {
        static int per_sm = 0;
        if (!per_sm) {
            if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_lpass_sm<P, U>, 32, 0) != cudaSuccess ||
                per_sm < 1)
                per_sm = 1;
        }
        const int nrange = ctx->nsm > 0 ? (ctx->nsm < 1024 ? ctx->nsm : 1024) : 1;
        const int chunk = (ctx->ntiles + nrange - 1) / nrange;
        CRK_TRY(zero_async(ctx, ctx->sm_next, sizeof(uint32_t) * nrange, s));
        launch(s, nrange * per_sm, 32, 0, k_lpass_sm<P, U>, g, prm, ctx->sm_next, nrange, chunk);
    } else {
        launch(s, grid_for(ctx->ntiles, WARPS), WARPS * 32, 0, k_lpass<P, WARPS, U>, g, prm,
               ord == ORD_LONGEST ? ctx->tile_order : nullptr);
    }
    return CRK_OK;
}

// per-SM tile ranges, the pass's own entries per iteration, records one
// iteration ahead
template <class P>
static int launch_sm_rp(crk_ctx *ctx, const ListGeom &g, const typename P::Params &prm, cudaStream_t s) {
    constexpr int U = P::UNROLL;
    static int per_sm = 0;
    if (!per_sm) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_lpass_sm<P, U, true>, 32, 0) != cudaSuccess ||
            per_sm < 1)
            per_sm = 1;
    }
    const int nrange = ctx->nsm > 0 ? (ctx->nsm < 1024 ? ctx->nsm : 1024) : 1;
    const int chunk = (ctx->ntiles + nrange - 1) / nrange;
    CRK_TRY(zero_async(ctx, ctx->sm_next, sizeof(uint32_t) * nrange, s));
    launch(s, nrange * per_sm, 32, 0, k_lpass_sm<P, U, true>, g, prm, ctx->sm_next, nrange, chunk);
    return CRK_OK;
}

template <class P, int W>
static void launch_width(crk_ctx *ctx, const ListGeom &g, const typename P::Params &prm, cudaStream_t s) {
    constexpr int U = P::PREFETCH ? 1 : P::UNROLL;
    launch(s, grid_for(ctx->ntiles, W), W * 32, 0, k_lpass<P, W, U>, g, prm, nullptr);
}

template <class P, int W, int U>
static void launch_rp(crk_ctx *ctx, const ListGeom &g, const typename P::Params &prm, cudaStream_t s) {
    launch(s, grid_for(ctx->ntiles, W), W * 32, 0, k_lpass<P, W, U, true>, g, prm, nullptr);
}

template <class P, int W>
static void launch_rp_u(crk_ctx *ctx, const ListGeom &g, const typename P::Params &prm, int U, cudaStream_t s) {
    switch (U) {   // 3 does not divide a block: it runs as 4
    case 1: launch_rp<P, W, 1>(ctx, g, prm, s); break;
    case 2: launch_rp<P, W, 2>(ctx, g, prm, s); break;
    default: launch_rp<P, W, 4>(ctx, g, prm, s); break;
    }
}

template <class P, int WARPS>
static int launch_variant(crk_ctx *ctx, const ListGeom &g, const typename P::Params &prm, int v, cudaStream_t s) {
    const LVariant lv = lvariant(v);
    if (lv.tma) {
        if constexpr (has_tma<P>::value) return P::launch_tma(ctx, g, prm, s);
        return CRK_OK;
    }
    if (lv.rp && lv.ord == ORD_SM) {
        if constexpr (!P::PREFETCH) return launch_sm_rp<P>(ctx, g, prm, s);
        return CRK_OK;
    }
    if (lv.rp) {   // records one iteration ahead (passes without their own prefetch)
        if constexpr (!P::PREFETCH) {
            if (lv.warps == 1)
                launch_rp_u<P, 1>(ctx, g, prm, lv.U, s);
            else
                launch_rp_u<P, WARPS>(ctx, g, prm, lv.U, s);
        }
        return CRK_OK;
    }
    if (lv.warps) {   // CTA width variants (the pass's own loop form)
        switch (lv.warps) {
        case 1: launch_width<P, 1>(ctx, g, prm, s); break;
        case 2: launch_width<P, 2>(ctx, g, prm, s); break;
        case 4: launch_width<P, 4>(ctx, g, prm, s); break;
        default: launch_width<P, 8>(ctx, g, prm, s); break;
        }
        return CRK_OK;
    }
    if (lv.ord == ORD_LONGEST) {
        int rc = tile_order_by_length(ctx, s);
        if (rc) return rc;
    }
    if constexpr (P::PREFETCH) {
        return launch_variant_u<P, WARPS, 1>(ctx, g, prm, lv.ord, s);
    } else {
        switch (lv.U) {
        case 1: return launch_variant_u<P, WARPS, 1>(ctx, g, prm, lv.ord, s);
        case 2: return launch_variant_u<P, WARPS, 2>(ctx, g, prm, lv.ord, s);
        default: return launch_variant_u<P, WARPS, 4>(ctx, g, prm, lv.ord, s);
        }
    }
}

// the measured default of each pass (before or without tuning)
template <class P>
constexpr int default_variant() {
    return P::PREFETCH ? (P::PERSISTENT ? 8 : 0) : P::UNROLL - 1;
}

template <class P>
constexpr bool variant_applies(int v) {
    if (lvariant(v).tma) return has_tma<P>::value;
    if (lvariant(v).rp) return !P::PREFETCH;
    return P::PREFETCH ? (lvariant(v).U <= 1) : true;
}

// the time between the tuner's events
inline int tune_time(crk_ctx *ctx, float *ms) {
    CRK_CUDA(ctx, cudaEventSynchronize(ctx->tune_ev[1]));
    CRK_CUDA(ctx, cudaEventElapsedTime(ms, ctx->tune_ev[0], ctx->tune_ev[1]));
    return CRK_OK;
}

// tune_slot: the autotuner's record for this pass (default: its profiling id;
// a pass with a different record layout, such as the two-kick P5, keeps its own)
template <class P, int WARPS, int MINB = 1>
int launch_lpass(crk_ctx *ctx, int prof_id, const typename P::Params &prm, cudaStream_t s, const char *what,
                 int tune_slot = -1) {
    const int ts = tune_slot >= 0 ? tune_slot : prof_id;
    if (ctx->n == 0) return CRK_OK;
    if (!ctx->lists_valid) return crk_set_error(ctx, CRK_ESTATE, "%s: neighbour lists are not built", what);
    ListGeom g{ctx->n,   ctx->ntiles, ctx->kcap,  ctx->tbase, ctx->len_g,
               ctx->len_u, ctx->cnt_g, ctx->cnt_u, ctx->ent,  nullptr};
    int rc;
    const int nsm = ctx->nsm > 0 ? ctx->nsm : 152;
    constexpr int U = P::PREFETCH ? 1 : P::UNROLL;
    // the tiles ctx->act[0 .. nact) only (time bins): each pass's default loop
    // form over that list, no tuning
    if (ctx->act) g.ntiles = ctx->nact;
    if (g.ntiles == 0) return CRK_OK;
    const bool forms = !ctx->act && !has_notune<P>::value;
    const bool split = g.ntiles < SPLIT_TILES * nsm;   // whatever the variant: its warps would not fill the SMs
    // long lists by CTAs (a captured step does not know whether there are any)
    const bool heavy = !split && !ctx->act &&
                       (ctx->graph_mode || ctx->h_counters[CNT_MAXCNT] > ctx->h_counters[CNT_LONG_ROWS]);
    if (heavy) g.heavy = ctx->counters + CNT_LONG_ROWS;
    const bool tuning = forms && ctx->tune_on && !ctx->graph_mode && ctx->tune_done[ts] != TUNED;
    float ms = 0.f;
    if (tuning && !split) {
        // time every applicable variant once (each recomputes the same outputs)
        float best = 3.0e38f;
        int bestv = default_variant<P>();
        for (int v = 0; v < NVAR; v++) {
            // the TMA-fed variant is measured 3x slower than the L1 forms on
            // GB300 (128^3: 20.5 ms, 7.4): it runs only when pinned (crk_tune_set)
            if (!variant_applies<P>(v) || lvariant(v).tma) continue;
            CRK_CUDA(ctx, cudaEventRecord(ctx->tune_ev[0], s));
            rc = launch_variant<P, WARPS>(ctx, g, prm, v, s);
            if (rc) return rc;
            CRK_CUDA(ctx, cudaEventRecord(ctx->tune_ev[1], s));
            ++ctx->launches;
            CRK_LAUNCH_CHECK(ctx, what);
            rc = tune_time(ctx, &ms);
            if (rc) return rc;
            if (ms < best) {
                best = ms;
                bestv = v;
            }
        }
        ctx->tune_choice[ts] = bestv;
        ctx->tune_ms[ts] = best;
        ctx->tune_done[ts] = TUNED;
    }
    const int v = ctx->tune_choice[ts] >= 0 ? ctx->tune_choice[ts] : default_variant<P>();
    if (forms && !variant_applies<P>(v))   // only a variant pinned by crk_tune_set can be one the pass lacks
        return crk_set_error(ctx, CRK_EINVAL, "%s: the pass has no variant %d", what, v);
    prof_begin(ctx, prof_id, s);
    rc = CRK_OK;
    constexpr int S = split_warps<P>();
    if (split) {
        if (tuning) CRK_CUDA(ctx, cudaEventRecord(ctx->tune_ev[0], s));
        launch(s, g.ntiles, S * 32, 0, k_lpass_split<P, S, U>, g, prm, ctx->act);
        if (tuning) CRK_CUDA(ctx, cudaEventRecord(ctx->tune_ev[1], s));
    } else if (ctx->act) {
        launch(s, grid_for(g.ntiles, WARPS), WARPS * 32, 0, k_lpass<P, WARPS, U>, g, prm, ctx->act);
    } else {
        if (heavy) {
            launch(s, 2 * nsm, S * 32, 0, k_lpass_long<P, S, U>, g, prm, ctx->heavy, ctx->counters + CNT_HEAVY);
            ++ctx->launches;
            CRK_LAUNCH_CHECK(ctx, what);
        }
        if (forms)
            rc = launch_variant<P, WARPS>(ctx, g, prm, v, s);
        else
            launch(s, grid_for(g.ntiles, WARPS), WARPS * 32, 0, k_lpass<P, WARPS, U>, g, prm, nullptr);
    }
    if (rc) return rc;
    ++ctx->launches;
    prof_end(ctx, s);
    CRK_LAUNCH_CHECK(ctx, what);
    if (tuning && split) {   // the one form such a set has; a later set above the line is still swept
        rc = tune_time(ctx, &ms);
        if (rc) return rc;
        ctx->tune_choice[ts] = default_variant<P>();
        ctx->tune_ms[ts] = ms;
        ctx->tune_done[ts] = TUNED_SPLIT;
    }
    return CRK_OK;
}

// ---------------------------------------------------------------- kernel maths

// C4 Wendland kernel (eq:C4) with eta = r/h and t = 1 - eta:
//   W = 495/(32 pi h^3) t^6 (1 + 6 eta + 35/3 eta^2)
//   grad_i W = -1155/(4 pi h^5) (1 + 5 eta) t^5 x_ij
// The constants are evaluated from their definitions at compile time (a
// hand-typed 1155/(4 pi) was once 6e-7 off, which the cancellation in the
// diagonal of grad m1 = delta m0 + cG sum V x x Gu amplified ~100-fold).
constexpr double KW_D = 495.0 / (32.0 * PI_D);
constexpr double KG_D = 1155.0 / (4.0 * PI_D);
constexpr float KW = (float)KW_D;         // 495 / (32 pi)
constexpr float KG = (float)KG_D;         // 1155 / (4 pi)
constexpr float K35_3 = (float)(35.0 / 3.0);
constexpr float K4PI_3 = (float)(4.0 * PI_D / 3.0);   // eq:hi

// Two float4 of a record in one 256-bit read-only load (p on a 32-byte
// boundary): one L1 sector per lane per instruction.
__device__ __forceinline__ void ldg_v8(const float4 *p, float4 &a, float4 &b) {
    asm("ld.global.nc.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
        : "=f"(a.x), "=f"(a.y), "=f"(a.z), "=f"(a.w), "=f"(b.x), "=f"(b.y), "=f"(b.z), "=f"(b.w)
        : "l"(p));
}

__device__ __forceinline__ float sqrt_approx(float v) {
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}

struct Sep {
    float x, y, z, r2, r;
};

__device__ __forceinline__ Sep separation(int dx, int dy, int dz) {
    Sep s;
    s.x = (float)dx * TWO_M32;
    s.y = (float)dy * TWO_M32;
    s.z = (float)dz * TWO_M32;
    s.r2 = fmaf(s.x, s.x, fmaf(s.y, s.y, s.z * s.z));
    s.r = sqrt_approx(s.r2);
    return s;
}

// The separation in fixed-point units, 2^32 times the above (the scaling is
// exact, so sums of products with it are the same bits up to that power of
// two): the passes apply 2^-32 to their constants instead of to every pair.
__device__ __forceinline__ Sep separation32(int dx, int dy, int dz) {
    Sep s;
    s.x = (float)dx;
    s.y = (float)dy;
    s.z = (float)dz;
    s.r2 = fmaf(s.x, s.x, fmaf(s.y, s.y, s.z * s.z));
    s.r = sqrt_approx(s.r2);
    return s;
}
__device__ __forceinline__ float distance32(int dx, int dy, int dz) { return separation32(dx, dy, dz).r; }

// An unevaluated sum hi + lo of two floats, for per-particle coefficients: each
// is rounded once, from products that carry about 45 bits.
struct F2 {
    float hi, lo;
};
__device__ __forceinline__ F2 f2_mul(F2 a, F2 b) {
    const float p = __fmul_rn(a.hi, b.hi);
    return F2{p, fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, fmaf(a.hi, b.hi, -p)))};
}
__device__ __forceinline__ F2 f2_mul(F2 a, float b) {
    const float p = __fmul_rn(a.hi, b);
    return F2{p, fmaf(a.lo, b, fmaf(a.hi, b, -p))};
}
__device__ __forceinline__ float f2_sum(F2 a, F2 b) {   // TwoSum of the high parts
    const float s = __fadd_rn(a.hi, b.hi), t = __fsub_rn(s, a.hi);
    const float e = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, t)), __fsub_rn(b.hi, t));
    return s + (e + (a.lo + b.lo));
}
constexpr float KW_LO = (float)(KW_D - (double)KW);
constexpr float KGW = (float)(-KG_D / KW_D);   // -56/3
constexpr float KGW_LO = (float)(-KG_D / KW_D - (double)KGW);

// -56/3 h^-2 as the passes form it from 1/h
__device__ __forceinline__ float grad_factor(float ih) { return KGW * (ih * ih); }

// The corrected kernel gradient of a particle with separation x, eq:gRK, is
// affine in x up to two radial factors:
//   grad W^R_g = t^6 (1 + 6 eta + 35/3 eta^2) (c_g + M_g . x) - 56/3 h^-2 t^5 (1 + 5 eta) (A' + B' . x) x_g,
//   c_g = cW (dA_g + A B_g), M_ga = cW (dA_g B_a + A dB^a_g), A' = cW A, B' = cW A B, cW = 495/(32 pi h^3).
struct Affine {
    float c[3], M[3][3], A, B[3];   // M[a][g]: the coefficient of x_a in component g
};
__device__ __forceinline__ Affine affine_of(const CorrRec &r, float h, float ih) {
    const float B[3] = {r.c0.y, r.c0.z, r.c0.w}, dA[3] = {r.c1.x, r.c1.y, r.c1.z};
    const float dB[9] = {r.c1.w, r.c2.x, r.c2.y, r.c2.z, r.c2.w, r.c3.x, r.c3.y, r.c3.z, r.c3.w};   // [a][g]
    const F2 i1 = {ih, __fmul_rn(fmaf(-ih, h, 1.f), ih)}, i2 = f2_mul(i1, i1);
    const F2 cW = f2_mul(F2{KW, KW_LO}, f2_mul(i2, i1)), cA = f2_mul(cW, r.c0.x);
    // A', B' also carry the rounding of grad_factor: its product with them is
    // cG A, cG A B to their own rounding
    const float gf = grad_factor(ih);
    const F2 g2 = f2_mul(F2{KGW, KGW_LO}, i2);
    const float fix = ((g2.hi - gf) + g2.lo) / gf;
    const F2 gA = F2{cA.hi, fmaf(cA.hi, fix, cA.lo)};
    Affine o;
#pragma unroll
    for (int g = 0; g < 3; g++) {
        const F2 d = f2_mul(cW, dA[g]);
        o.c[g] = f2_sum(d, f2_mul(cA, B[g]));
#pragma unroll
        for (int a = 0; a < 3; a++) o.M[a][g] = f2_sum(f2_mul(d, B[a]), f2_mul(cA, dB[3 * a + g]));
        const F2 v = f2_mul(gA, B[g]);
        o.B[g] = v.hi + v.lo;
    }
    o.A = gA.hi + gA.lo;
    return o;
}

}  // namespace crk
