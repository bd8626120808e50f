// crk_walk.cu -- per-particle neighbour lists, built once per evaluation from
// the tile interaction lists (CRK-HACC Sec. 2.3: interaction lists assembled
// once per hydro step and reused by every hydro kernel), and P1 volumes
// (Sec. 1.2 eq:vol, Sec. 2.6 eq:hi) over those lists.
//
// One walk: warp per i-tile over the pair-set tile list; every staged
// neighbour is tested once.  Lane i writes its list into the tile's columns in
// blocks of four entries (layout: crk_pass.cuh): gather neighbours (j != i,
// |dq|^2 < H_i^2) from the first block up, the other pair-set neighbours from
// the last block down, the last block of each padded with i.  A particle with
// more than KCAP / 4 blocks sets the overflow maximum; the host then grows KCAP
// and walks again.  Stored pair forces use a compact layout: per-tile base (in
// units of 32 entries) from a scan of the per-tile maximum row count.
#include "crk_pass.cuh"

namespace crk {

constexpr int WALK_WARPS = 8;
constexpr int WALK_WIDE = 8;       // fewer tiles than this per SM: CTAs of 32 warps
constexpr int WALK_ALL = 20;       // fewer tiles than this per SM: every tile is shared by a CTA's warps
// Candidate tiles above which a tile is shared.  The walk, us, with the line at 192, 256,
// 384, 512, 768, none: clustered 64^3 (mean 134 candidates) 762, 698, 749, 838, 912, 1086;
// 128^3 (126) 4629, 4396, 4285, 4340, 4482, 6068; Sedov 80^3 after 400 steps (160) 2748, 2710,
// 2512, 2473, 2494, 8048; no tile of the Hilbert order is near it.
constexpr int WALK_HEAVY = 384;

struct WalkArgs {
    int n, ntiles, kcap;
    const uint4 *q4;
    const float *hs;
    const uint2 *ofs;        // pair-set tile list per tile
    const uint32_t *tiles;
    const uint4 *tlo, *thi;  // tile boxes (xlo, ylo, zlo, Hmax), (xhi, yhi, zhi, count)
    float *V, *Nn;
    uint4 *qV;               // (qx, qy, qz, V bits)
    int32_t *cnt_g, *cnt_u;
    uint32_t *len_g, *len_u; // per-tile max counts
    unsigned long long *pairs_g, *pairs_u, *maxcnt;
    uint32_t *ent;
    const int32_t *sbox;     // batched boxes: box of each slot (BATCH only)
    const uint32_t *nbox;    // box range of each tile (BATCH only)
    const int32_t *act;      // may be null: walk the tiles act[0 .. ntiles) only
    int32_t *long_list;      // tiles with more than HEAVY_ROWS rows (the passes take the long ones), and their count
    unsigned long long *nlong;
    int heavy;               // tiles with more candidate tiles than this are shared by the warps of a CTA
    int hblocks;             // CTAs that take them (all: one per tile, every tile is shared)
    int all;
    unsigned long long *tests;   // lane tests of the exact predicate (LISTS walk)
};

// circular distance (fixed point) from coordinate q to the arc [lo, hi]
// (which may wrap, lo > hi); differences modulo 2^32
__device__ __forceinline__ float point_gap(uint32_t q, uint32_t lo, uint32_t hi) {
    return q - lo <= hi - lo ? 0.f : (float)min(lo - q, q - hi);
}

// One segment of a lane's list on its way to memory: the last up to three
// entries wait in registers (newest in p3) until their block is full.  A lane
// of a shared tile (PART) may start inside a block, `start` entries of the
// segment coming from the warps before it: that block's and the last block's
// entries are written singly.
template <bool PART>
struct Seg {
    uint32_t p1, p2, p3;
    int n, start;   // entries of the segment so far, and before this lane's first
    int at;         // word of the current block in the tile's columns
    __device__ __forceinline__ void push(uint32_t j, uint32_t *cols, int kcap, int step) {
        ++n;
        if ((n & (LB - 1)) == 0) {
            if (n <= kcap) {
                if (!PART || n - LB >= start) {
                    *reinterpret_cast<uint4 *>(cols + at) = make_uint4(p1, p2, p3, j);
                } else {
                    if (n - 3 >= start) cols[at + 1] = p2;
                    if (n - 2 >= start) cols[at + 2] = p3;
                    cols[at + 3] = j;
                }
            }
            at += step;
        }
        p1 = p2;
        p2 = p3;
        p3 = j;
    }
    // the entries of the last, partial block
    __device__ __forceinline__ void close(uint32_t *cols, int kcap) const {
        const int r = n & (LB - 1), m = PART ? min(r, n - start) : r;
        if (m == 0 || n > kcap) return;
        cols[at + r - 1] = p3;
        if (m > 1) cols[at + r - 2] = p2;
        if (m > 2) cols[at + r - 3] = p1;
    }
    // its pads: the lane's own index
    __device__ __forceinline__ void pad(uint32_t self, uint32_t *cols, int kcap) const {
        const int r = n & (LB - 1);
        if (r == 0 || n > kcap) return;
        for (int k = r; k < LB; k++) cols[at + k] = self;
    }
};
constexpr int BLOCK_WORDS = LB * 32;

// Rounding margins of the walk's FP32 comparisons, u = 2^-24.
// Relative form: a particle within reach of the tile (gap to its box below the
// support R < 2^32 / 3) lies at an offset in (-R, E + R) of the box corner, E the
// tile's largest extent; with E + R < 2^31 that offset is the minimum image, and
// the differences of two such offsets are too.  Offsets are exact integers of
// at most M = E + R rounded to FP32: each is off by at most u M, a difference d
// by 3 u M, a squared distance r^2 <= 3 M^2 by 2 sqrt(3) r 3 u M + 3 u r^2 <=
// 27 u M^2 and a squared support by 3 u M^2: a comparison that clears 48 u M^2
// has the sign of the exact one.
// Integer form (tiles with E beyond that): the minimum-image difference is an
// exact integer rounded once, so r^2 is off by at most 5 u r^2 and a comparison
// with H^2 that clears 16 u H^2 (H the largest support) has the exact sign.
constexpr float MARGIN_REL = 48.f / 16777216.f, MARGIN_INT = 16.f / 16777216.f;
constexpr int RING = 64;   // kept particles a warp holds: a batch of 32 and up to 32 more

// What is the same for the warp's lanes: kept in shared memory, out of the
// loops' registers (64 a thread are four CTAs per SM).
struct WalkBox {
    uint4 lo;        // box corner, largest support
    float ex, ey, ez;   // extents
    uint32_t Ie;     // the largest
};

// Batches of masks a warp of a shared tile keeps between counting and writing.
constexpr int MASKS = 8;
struct WalkMasks {
    uint32_t g[MASKS][32], j[MASKS][32], id[MASKS][32];
};

template <bool VOL, bool BATCH>
struct WalkShm {
    WalkBox B;
    uint4 r[RING];                      // x, y, z relative or fixed point; H^2
    uint32_t id[VOL ? 1 : RING];        // sorted index
    int32_t box[BATCH ? RING : 1];
};

// Shared memory of a CTA of W warps.
template <bool LISTS, bool VOL, bool BATCH, int W>
struct WalkCta {
    WalkShm<VOL, BATCH> shm[W];
    WalkMasks masks[LISTS ? W : 1];
    int part[2][W][32];
};

// A tile and this lane's particle of it.
struct WalkTile {
    int tile, i;
    bool valid, raw;          // raw: integer form
    float fx, fy, fz;         // this lane relative to the box corner
    float Hf, Hf2;
    int32_t bi;               // box of the particle, box range of the tile (batched boxes)
    uint32_t Ib;
};

// fixed-point record of this lane's particle (0 for invalid lanes): read again
// where the rarer paths need it, which keeps it out of the loops' registers
__device__ __forceinline__ uint4 own_record(const WalkArgs &a, const WalkTile &T) {
    return T.valid ? __ldg(a.q4 + T.i) : make_uint4(0, 0, 0, 0);
}

template <bool BATCH>
__device__ __forceinline__ WalkTile walk_tile(const WalkArgs &a, int tile, int lane, WalkBox &B) {
    WalkTile T;
    T.tile = tile;
    T.i = tile * TILE + lane;
    T.valid = T.i < a.n;
    const uint4 qi = own_record(a, T);
    const uint4 Ilo = __ldg(a.tlo + tile), Ihi = __ldg(a.thi + tile);
    const uint32_t x = Ihi.x - Ilo.x, y = Ihi.y - Ilo.y, z = Ihi.z - Ilo.z, e = max(max(x, y), z);
    T.raw = e >= 0x80000000u - 0x55555556u;   // E + R may reach 2^31
    __syncwarp();
    if (lane == 0) B = WalkBox{Ilo, (float)x, (float)y, (float)z, e};
    __syncwarp();
    T.fx = (float)(qi.x - Ilo.x);
    T.fy = (float)(qi.y - Ilo.y);
    T.fz = (float)(qi.z - Ilo.z);
    T.Hf = (float)qi.w;
    T.Hf2 = T.Hf * T.Hf;
    T.bi = BATCH && T.valid ? a.sbox[T.i] : 0;
    T.Ib = BATCH ? __ldg(a.nbox + tile) : 0u;
    return T;
}

// The candidate tiles [t0, t1) of a tile's list, by one warp.  Lane jj stages
// particle jj of a candidate and keeps it if it can be in the pair set (VOL: the
// gather set) of some particle of the tile; the kept particles of successive
// candidates fill batches of 32 in shared memory.  visit(gm, jm, ring, c) gets a
// batch of c kept particles in ring[ring ..]: bit p of gm: slot p is in
// gather(i); of jm: i is in gather(slot p) (VOL: visit(ring, c), no masks).
// `kept` counts the kept particles: every lane tests each of them.
template <bool VOL, bool BATCH, class Visit>
__device__ __forceinline__ void walk_range(const WalkArgs &a, const WalkTile &T, int lane, uint2 lo, int t0, int t1,
                                           WalkShm<VOL, BATCH> &S, uint32_t &kept, Visit &&visit) {
    uint32_t head = 0, done = 0;   // kept particles staged, and handed on
    uint32_t exact_to = 0;         // batches that start below take the integer predicate (mixed boxes)
    int self = -1;                 // the staged number of this lane's own particle
    float margin = 0.f;            // of the tests so far
    auto batch = [&](int c) {
        const uint32_t ring = done & (RING - 1);
        if constexpr (VOL) {
            visit(ring, c);
        } else {
            unsigned gm = 0u, jm = 0u;
            const unsigned live = c == 32 ? 0xffffffffu : (1u << c) - 1u;
            bool exact = done < exact_to;
            if (!exact) {
                float amb = 3.0e38f;
                const int top = (c + 3) & ~3;
                if (!T.raw) {
                    for (int p = top - 4; p >= 0; p -= 4) {   // independent chains; slot 0 ends at bit 0
#pragma unroll
                        for (int u = 3; u >= 0; u--) {
                            const float4 f = reinterpret_cast<const float4 *>(S.r)[ring + p + u];
                            const float dx = T.fx - f.x, dy = T.fy - f.y, dz = T.fz - f.z;
                            const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
                            const float ti = r2 - T.Hf2, tj = r2 - f.w;
                            amb = fminf(amb, fminf(fabsf(ti), fabsf(tj)));
                            gm = __funnelshift_l(__float_as_uint(ti), gm, 1);
                            jm = __funnelshift_l(__float_as_uint(tj), jm, 1);
                        }
                    }
                } else {
                    const uint4 qi = own_record(a, T);
                    for (int p = top - 4; p >= 0; p -= 4) {
#pragma unroll
                        for (int u = 3; u >= 0; u--) {
                            const uint4 q = S.r[ring + p + u];
                            const float dx = (float)(int)(qi.x - q.x), dy = (float)(int)(qi.y - q.y),
                                        dz = (float)(int)(qi.z - q.z);
                            const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
                            const float ti = r2 - T.Hf2, tj = r2 - __uint_as_float(q.w);
                            amb = fminf(amb, fminf(fabsf(ti), fabsf(tj)));
                            gm = __funnelshift_l(__float_as_uint(ti), gm, 1);
                            jm = __funnelshift_l(__float_as_uint(tj), jm, 1);
                        }
                    }
                }
                exact = __any_sync(0xffffffffu, T.valid && amb < margin);
            }
            if (exact) {
                gm = jm = 0u;
                const uint4 qi = own_record(a, T);
                const unsigned long long Hi2 = (unsigned long long)qi.w * qi.w;
                for (int p = 0; p < c; p++) {
                    const uint4 q = __ldg(a.q4 + S.id[ring + p]);
                    unsigned long long R2 = r2_fixed((int)(qi.x - q.x), (int)(qi.y - q.y), (int)(qi.z - q.z));
                    if (BATCH && S.box[ring + p] != T.bi) R2 = ~0ull;
                    gm |= (R2 < Hi2 ? 1u : 0u) << p;
                    jm |= (R2 < (unsigned long long)q.w * q.w ? 1u : 0u) << p;
                }
            }
            unsigned use = T.valid ? live : 0u;
            const int me = self - (int)done;   // j != i
            if (me >= 0 && me < 32) use &= ~(1u << me);
            visit(gm & use, jm & use, ring);
        }
        done += (uint32_t)c;
    };
    // software pipeline over the candidate tiles: the tile id two ahead, and
    // the box and this lane's staged particle of the next tile, are in flight
    // while the current tile is tested (each is otherwise a dependent L2 trip)
    const uint32_t *tl = a.tiles + lo.x;
    int J1 = t0 < t1 ? (int)__ldg(tl + t0) : 0, J2 = t0 + 1 < t1 ? (int)__ldg(tl + t0 + 1) : 0;
    uint4 qn = make_uint4(0, 0, 0, 0);
    uint32_t H1 = 0;
    if (t0 < t1) {
        H1 = __ldg(&a.tlo[J1].w);
        if (J1 * TILE + lane < a.n) qn = __ldg(a.q4 + J1 * TILE + lane);
    }
    for (int t = t0; t < t1; t++) {
        const int J = J1;
        const uint4 qc = qn;
        const uint32_t JH = H1;
        J1 = J2;
        if (t + 2 < t1) J2 = (int)__ldg(tl + t + 2);
        if (t + 1 < t1) {
            H1 = __ldg(&a.tlo[J1].w);
            if (J1 * TILE + lane < a.n) qn = __ldg(a.q4 + J1 * TILE + lane);
        }
        const int j0 = J * TILE;
        const int cnt = min(TILE, a.n - j0);
        const uint4 Ilo = S.B.lo;
        const uint32_t R = VOL ? Ilo.w : max(Ilo.w, JH), M = S.B.Ie + R;   // warp-uniform
        // Keep a particle whose gap to the tile's box is below the larger support:
        // conservative, so the lists are unchanged.  (Skipping candidates whose
        // box no lane's sphere touches, too, took 30 instructions a candidate
        // and dropped few: 128^3 clustered 3.80 ms with that test, 3.20 without.)
        bool keep;
        float jx = 0.f, jy = 0.f, jz = 0.f;
        const float edge = T.raw ? (float)R : (float)M;
        const float mrg = (T.raw ? MARGIN_INT : MARGIN_REL) * (edge * edge);
        if (!T.raw) {
            jx = (float)(int)(qc.x - Ilo.x);
            jy = (float)(int)(qc.y - Ilo.y);
            jz = (float)(int)(qc.z - Ilo.z);
            const float hx = fmaxf(fmaxf(-jx, jx - S.B.ex), 0.f), hy = fmaxf(fmaxf(-jy, jy - S.B.ey), 0.f),
                        hz = fmaxf(fmaxf(-jz, jz - S.B.ez), 0.f);
            const float rj = (float)(VOL ? Ilo.w : max(qc.w, Ilo.w));
            keep = lane < cnt && fmaf(hx, hx, fmaf(hy, hy, hz * hz)) < fmaf(rj, rj, mrg);
        } else {
            const uint4 Ihi = __ldg(a.thi + T.tile);
            const float hx = point_gap(qc.x, Ilo.x, Ihi.x), hy = point_gap(qc.y, Ilo.y, Ihi.y),
                        hz = point_gap(qc.z, Ilo.z, Ihi.z), rj = (float)(VOL ? Ilo.w : max(qc.w, Ilo.w));
            keep = lane < cnt && fmaf(hx, hx, fmaf(hy, hy, hz * hz)) < fmaf(rj, rj, mrg);
        }
        bool mixed = false;   // the pair's boxes must be compared
        int32_t bj = 0;
        if constexpr (BATCH) {
            const uint32_t Jb = __ldg(a.nbox + J);
            mixed = T.Ib != Jb || (T.Ib & 0xffffu) != (T.Ib >> 16);
            bj = (int32_t)(Jb & 0xffffu);
            if (mixed && lane < cnt) {
                bj = __ldg(a.sbox + j0 + lane);
                keep = keep && (uint32_t)bj >= (T.Ib & 0xffffu) && (uint32_t)bj <= (T.Ib >> 16);
            }
        }
        const unsigned mask = __ballot_sync(0xffffffffu, keep);
        if (mask == 0u) continue;
        const uint32_t at = head + (uint32_t)__popc(mask & lanemask_lt());
        if (J == T.tile) self = (int)at;   // this tile's particles are all kept
        __syncwarp();
        if (keep) {
            const uint32_t k = at & (RING - 1);
            const float hj = (float)qc.w;
            const bool fix = VOL || T.raw;
            S.r[k] = make_uint4(fix ? qc.x : __float_as_uint(jx), fix ? qc.y : __float_as_uint(jy),
                                fix ? qc.z : __float_as_uint(jz), __float_as_uint(hj * hj));
            if (!VOL) S.id[k] = (uint32_t)(j0 + lane);
            if (BATCH) S.box[k] = bj;
        }
        __syncwarp();
        head += (uint32_t)__popc(mask);
        margin = fmaxf(margin, mrg);
        if (mixed) exact_to = head;
        if (head - done >= 32u) batch(32);
    }
    if (head > done) batch((int)(head - done));
    kept += head;
}

// Neighbour lists (LISTS) or volumes (VOL).  BATCH: the particles belong to
// independent boxes; j can be a neighbour of i only in i's box (the box ranges
// of tiles prune the rest).
//
// LISTS.  Bound by instruction issue: each lane tests every kept particle, and
// about one test in five finds an entry.  A test is an FP32 difference against
// both squared supports (3 add, 3 multiply-add, 2 add, a running minimum of the
// distance to either threshold and a funnel shift per mask: 13 instructions
// against 27 of the 64-bit integer test); the integer predicate runs only for a
// batch where some lane came within the rounding margin of a threshold, or that
// holds several batched boxes, so the lists are the exact ones.  Batches span
// candidate tiles (a tile keeps about 15 of a candidate's 32), so the loops run
// full and each lane's divergent writing of its entries runs half as often.
//
// VOL.  Sums n_i instead of writing lists: W vanishes beyond h_i, so every kept
// particle is summed without the predicate, and only particles within the
// tile's own supports are kept.
//
// A warp takes a tile, except where that leaves the chip waiting for a few
// warps: tiles with more than a.heavy candidates (a run of the Morton order
// that jumps across the box: at 64^3 clustered the largest has 16 times the
// mean's candidates), and every tile of a set that does not fill the chip.
// Those are shared by the W warps of a CTA, each taking a range of the
// candidates (W = 32 below WALK_WIDE tiles per SM, where the CTA of the slowest
// tile is the time: Sedov 17^3 97 -> 43 us, 16^3 36 -> 24, the tiles of a 48^3
// cycle 2.20 -> 1.46 ms; at 13 tiles per SM it is even, and a loss at 20): a
// first sweep counts and keeps its masks, the prefix over the
// warps gives each its place in the lists, and the entries are written from the
// masks (a warp with more than MASKS batches sweeps again), so the lists are
// exactly the one-warp walk's.
template <bool LISTS, bool VOL, bool BATCH, int W>
__global__ void __launch_bounds__(W * 32, 32 / W) k_walk(WalkArgs a) {
    grid_wait();
    extern __shared__ __align__(16) unsigned char walk_smem[];
    WalkCta<LISTS, VOL, BATCH, W> &C = *reinterpret_cast<WalkCta<LISTS, VOL, BATCH, W> *>(walk_smem);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    WalkShm<VOL, BATCH> &S = C.shm[w];
    const int kcap = a.kcap;
    // V_i, N_i from the kernel sum of a lane
    auto volume = [&](const WalkTile &T, float acc) {
        const float h = a.hs[T.i], inv_h = 1.f / h;
        const float ih3 = inv_h * inv_h * inv_h;
        const float nsum = KW * ih3 * acc;                         // n_i, eq:vol
        a.V[T.i] = 1.f / nsum;
        if (a.Nn) a.Nn[T.i] = (K4PI_3 * h * h * h) * nsum;         // eq:hi
    };
    auto sum_batch = [&](const WalkTile &T, const uint4 &qi, float inv_h, uint32_t ring, int c, float &acc) {
        auto term = [&](int p, bool live) {
            const uint4 q = S.r[ring + p];
            const float eta = distance32((int)(qi.x - q.x), (int)(qi.y - q.y), (int)(qi.z - q.z)) * inv_h;
            float t = __saturatef(1.f - eta);
            if (!live || (BATCH && S.box[ring + p] != T.bi)) t = 0.f;
            const float t2 = t * t, t3 = t2 * t;
            acc = fmaf(t3 * t3, fmaf(eta, fmaf(eta, K35_3, 6.f), 1.f), acc);
        };
        if (c == 32) {
            for (int p = 0; p < 32; p += 4) {
#pragma unroll
                for (int u = 0; u < 4; u++) term(p + u, true);
            }
        } else {
            for (int p = 0; p < c; p += 2) {
                term(p, true);
                term(p + 1, p + 1 < c);
            }
        }
    };
    // counts, per-tile rows and totals of a finished tile (one warp)
    auto close = [&](const WalkTile &T, int cg, int co) {
        const int rg = LB * list_blocks(cg), ru = rg + LB * list_blocks(co);   // rows with the pads
        if (T.valid) {
            a.cnt_g[T.i] = cg;
            a.cnt_u[T.i] = cg + co;
        }
        const uint32_t mg = __reduce_max_sync(0xffffffffu, (uint32_t)rg);
        const uint32_t mu = __reduce_max_sync(0xffffffffu, (uint32_t)ru);
        const uint32_t sg = __reduce_add_sync(0xffffffffu, (uint32_t)cg);
        const uint32_t su = __reduce_add_sync(0xffffffffu, (uint32_t)(cg + co));
        if (lane == 0) {
            a.len_g[T.tile] = min(mg, (uint32_t)kcap);
            a.len_u[T.tile] = min(mu, (uint32_t)kcap);
            atomicAdd(a.pairs_g, (unsigned long long)sg);
            atomicAdd(a.pairs_u, (unsigned long long)su);
            atomicMax(a.maxcnt, (unsigned long long)mu);
            if (LISTS && mu > (uint32_t)HEAVY_ROWS) a.long_list[atomicAdd(a.nlong, 1ull)] = T.tile;
        }
    };
    auto shared_tile = [&](int tile, uint2 lo) {   // by all warps of the CTA
        const WalkTile T = walk_tile<BATCH>(a, tile, lane, S.B);
        const int nt = (int)lo.y, chunk = (nt + W - 1) / W;
        const int t0 = min(nt, w * chunk), t1 = min(nt, t0 + chunk);
        uint32_t kept = 0;
        if constexpr (VOL) {
            const uint4 qi = own_record(a, T);
            const float inv_h = TWO_M32 * (1.f / (T.valid ? a.hs[T.i] : 1.f));
            float acc = 0.f;
            walk_range<VOL, BATCH>(a, T, lane, lo, t0, t1, S, kept,
                                   [&](uint32_t ring, int c) { sum_batch(T, qi, inv_h, ring, c, acc); });
            C.part[0][w][lane] = __float_as_int(acc);
            __syncthreads();
            if (w == 0) {
                for (int v = 1; v < W; v++) acc += __int_as_float(C.part[0][v][lane]);
                if (T.valid) volume(T, acc);
                close(T, 0, 0);
            }
        } else {
            uint32_t *const col0 = a.ent + (size_t)tile * kcap * 32;
            WalkMasks &K = C.masks[w];
            int cg = 0, co = 0, nb = 0;
            walk_range<VOL, BATCH>(a, T, lane, lo, t0, t1, S, kept, [&](unsigned gm, unsigned jm, uint32_t ring) {
                jm &= ~gm;
                cg += __popc(gm);
                co += __popc(jm);
                if (nb < MASKS) {
                    K.g[nb][lane] = gm;
                    K.j[nb][lane] = jm;
                    K.id[nb][lane] = S.id[ring + lane];
                }
                nb++;
            });
            if (lane == 0) atomicAdd(a.tests, 32ull * kept);
            C.part[0][w][lane] = cg;
            C.part[1][w][lane] = co;
            __syncthreads();
            int pg = 0, po = 0, tg = 0, to = 0;   // this warp's place, the totals
            for (int v = 0; v < W; v++) {
                if (v == w) pg = tg, po = to;
                tg += C.part[0][v][lane];
                to += C.part[1][v][lane];
            }
            Seg<true> G{0u, 0u, 0u, pg, pg, (int)block_at(pg / LB, lane)};
            Seg<true> O{0u, 0u, 0u, po, po, (int)block_at(kcap / LB - 1 - po / LB, lane)};
            auto write = [&](unsigned gm, unsigned jm, const uint32_t *id) {
                for (; gm; gm &= gm - 1u) G.push(id[__ffs(gm) - 1], col0, kcap, BLOCK_WORDS);
                for (; jm; jm &= jm - 1u) O.push(id[__ffs(jm) - 1], col0, kcap, -BLOCK_WORDS);
            };
            if (nb <= MASKS) {
                for (int b = 0; b < nb; b++) write(K.g[b][lane], K.j[b][lane], K.id[b]);
            } else {
                walk_range<VOL, BATCH>(a, T, lane, lo, t0, t1, S, kept, [&](unsigned gm, unsigned jm, uint32_t ring) {
                    write(gm, jm & ~gm, S.id + ring);
                });
            }
            if (T.valid) {
                G.close(col0, kcap);
                O.close(col0, kcap);
                if (w == W - 1) {   // its segments end where the lists end
                    G.pad((uint32_t)T.i, col0, kcap);
                    O.pad((uint32_t)T.i, col0, kcap);
                }
            }
            if (w == 0) close(T, tg, to);
        }
        __syncthreads();   // `part` is free for the next tile
    };
    if ((int)blockIdx.x < a.hblocks) {
        if (a.all) {
            const int tile = a.act ? a.act[blockIdx.x] : (int)blockIdx.x;
            shared_tile(tile, a.ofs[tile]);
            return;
        }
        // neighbouring tiles, which are heavy together, go to different CTAs
        for (int t0 = (int)blockIdx.x; t0 < a.ntiles; t0 += a.hblocks * 32) {
            const int t = t0 + lane * a.hblocks;
            const int mine = t < a.ntiles ? (a.act ? a.act[t] : t) : -1;
            unsigned m = __ballot_sync(0xffffffffu, mine >= 0 && (int)a.ofs[max(mine, 0)].y > a.heavy);
            for (; m; m &= m - 1u) {
                const int tile = __shfl_sync(0xffffffffu, mine, __ffs(m) - 1);
                shared_tile(tile, a.ofs[tile]);
            }
        }
        return;
    }
    const int tw = ((int)blockIdx.x - a.hblocks) * W + w;
    if (tw >= a.ntiles) return;
    const int tile = a.act ? a.act[tw] : tw;
    const uint2 lo = a.ofs[tile];
    if ((int)lo.y > a.heavy) return;
    const WalkTile T = walk_tile<BATCH>(a, tile, lane, S.B);
    uint32_t kept = 0;
    if constexpr (VOL) {
        const uint4 qi = own_record(a, T);
        const float inv_h = TWO_M32 * (1.f / (T.valid ? a.hs[T.i] : 1.f));
        float acc = 0.f;
        walk_range<VOL, BATCH>(a, T, lane, lo, 0, (int)lo.y, S, kept,
                               [&](uint32_t ring, int c) { sum_batch(T, qi, inv_h, ring, c, acc); });
        if (T.valid) volume(T, acc);
        close(T, 0, 0);
    } else {
        uint32_t *const col0 = a.ent + (size_t)tile * kcap * 32;
        Seg<false> G{0u, 0u, 0u, 0, 0, (int)block_at(0, lane)};
        Seg<false> O{0u, 0u, 0u, 0, 0, (int)block_at(kcap / LB - 1, lane)};
        walk_range<VOL, BATCH>(a, T, lane, lo, 0, (int)lo.y, S, kept, [&](unsigned gm, unsigned jm, uint32_t ring) {
            jm &= ~gm;
            for (; gm; gm &= gm - 1u) G.push(S.id[ring + __ffs(gm) - 1], col0, kcap, BLOCK_WORDS);
            for (; jm; jm &= jm - 1u) O.push(S.id[ring + __ffs(jm) - 1], col0, kcap, -BLOCK_WORDS);
        });
        if (T.valid) {
            G.close(col0, kcap);
            O.close(col0, kcap);
            G.pad((uint32_t)T.i, col0, kcap);
            O.pad((uint32_t)T.i, col0, kcap);
        }
        close(T, G.n, O.n);
        if (lane == 0) atomicAdd(a.tests, 32ull * kept);
    }
}

// total stored-force units (32 entries each) = base[last] + len_u[last], and the
// rows above which a tile's list is a long one
__global__ void k_total(int ntiles, const uint32_t *__restrict__ base, const uint32_t *__restrict__ len,
                        unsigned long long *counters) {
    grid_wait();
    const unsigned long long total = (unsigned long long)base[ntiles - 1] + len[ntiles - 1];
    counters[CNT_ENTRIES] = total;
    counters[CNT_LONG_ROWS] =
        max((unsigned long long)HEAVY_ROWS, 3ull * total / (2ull * (unsigned long long)ntiles));
}

static WalkArgs walk_args(crk_ctx *ctx) {
    WalkArgs a;
    a.n = ctx->n;
    a.ntiles = ctx->ntiles;
    a.kcap = ctx->kcap;
    a.q4 = ctx->q4;
    a.hs = ctx->hs;
    a.ofs = ctx->uofs;
    a.tiles = ctx->ulist;
    a.tlo = ctx->node_lo;
    a.thi = ctx->node_hi;
    a.V = ctx->V;
    a.Nn = ctx->Nn;
    a.qV = ctx->qV;
    a.cnt_g = ctx->cnt_g;
    a.cnt_u = ctx->cnt_u;
    a.len_g = ctx->len_g;
    a.len_u = ctx->len_u;
    a.pairs_g = ctx->counters + CNT_PAIRS_G;
    a.pairs_u = ctx->counters + CNT_PAIRS_U;
    a.maxcnt = ctx->counters + CNT_MAXCNT;
    a.ent = ctx->volumes_only ? nullptr : ctx->ent;
    a.sbox = ctx->nbox > 1 ? ctx->sbox : nullptr;
    a.nbox = ctx->nbox > 1 ? ctx->node_box : nullptr;
    a.act = ctx->act;
    if (ctx->act) a.ntiles = ctx->nact;
    a.tests = ctx->counters + CNT_WALK_TESTS;
    a.long_list = ctx->heavy;
    a.nlong = ctx->counters + CNT_HEAVY;
    const int nsm = ctx->nsm > 0 ? ctx->nsm : 152;
    a.all = a.ntiles < WALK_ALL * nsm;
    a.heavy = a.all ? -1 : WALK_HEAVY;
    a.hblocks = a.all ? a.ntiles : 4 * nsm;   // a full wave of CTAs
    return a;
}

template <bool LISTS, bool VOL, bool BATCH, int W>
static int launch_walk_wide(crk_ctx *ctx, const WalkArgs &a, cudaStream_t s) {
    using Cta = WalkCta<LISTS, VOL, BATCH, W>;
    if (sizeof(Cta) > 48 * 1024)
        CRK_CUDA(ctx, cudaFuncSetAttribute(k_walk<LISTS, VOL, BATCH, W>,
                                           cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Cta)));
    const int g = a.hblocks + (a.all ? 0 : grid_for(a.ntiles, W));
    launch(s, g, W * 32, sizeof(Cta), k_walk<LISTS, VOL, BATCH, W>, a);
    return CRK_OK;
}

template <bool LISTS, bool VOL, bool BATCH>
static int launch_walk_form(crk_ctx *ctx, const WalkArgs &a, cudaStream_t s) {
    const int nsm = ctx->nsm > 0 ? ctx->nsm : 152;
    if (a.ntiles < WALK_WIDE * nsm) return launch_walk_wide<LISTS, VOL, BATCH, 32>(ctx, a, s);
    return launch_walk_wide<LISTS, VOL, BATCH, WALK_WARPS>(ctx, a, s);
}

static int launch_walk(crk_ctx *ctx, cudaStream_t s) {
    if (!ctx->volumes_only) {
        int rc = crk_ensure_entries(ctx, (long long)ctx->ntiles * 32 * ctx->kcap, -1);
        if (rc) return rc;
    }
    CRK_TRY(zero_async(ctx, ctx->counters + CNT_PAIRS_G, 5 * sizeof(unsigned long long), s));
    if (ctx->act && !ctx->volumes_only) {   // tiles left out of the walk take no list columns and no stored forces
        CRK_TRY(zero_async(ctx, ctx->len_g, sizeof(uint32_t) * ctx->ntiles, s));
        CRK_TRY(zero_async(ctx, ctx->len_u, sizeof(uint32_t) * ctx->ntiles, s));
    }
    if (ctx->act && ctx->nact == 0) return CRK_OK;
    prof_begin(ctx, PROF_LISTS, s);
    const WalkArgs a = walk_args(ctx);
    const bool b = ctx->nbox > 1;
    int rc = CRK_OK;
    if (ctx->volumes_only && b)
        rc = launch_walk_form<false, true, true>(ctx, a, s);
    else if (ctx->volumes_only)
        rc = launch_walk_form<false, true, false>(ctx, a, s);
    else if (b)
        rc = launch_walk_form<true, false, true>(ctx, a, s);
    else
        rc = launch_walk_form<true, false, false>(ctx, a, s);
    if (rc) return rc;
    ++ctx->launches;
    prof_end(ctx, s);
    CRK_LAUNCH_CHECK(ctx, "neighbour walk");
    return CRK_OK;
}

// The walk and the list layout (synchronises once): on overflow grow KCAP and
// walk again; then lay out the stored pair forces.
int run_lists(crk_ctx *ctx, cudaStream_t s) {
    if (ctx->lists_valid) return CRK_OK;
    if (ctx->volumes_only) return crk_set_error(ctx, CRK_ESTATE, "no neighbour lists in this context");
    if (ctx->n == 0) {
        ctx->lists_valid = 1;
        return CRK_OK;
    }
    int nt = ctx->ntiles;
    for (int attempt = 0; attempt < 3; attempt++) {
        int rc = launch_walk(ctx, s);
        if (rc) return rc;
        rc = scan_u32(ctx, ctx->len_u, ctx->tbase, nt, s);
        if (rc) return rc;
        launch(s, 1, 1, 0, k_total, nt, ctx->tbase, ctx->len_u, ctx->counters);
        ++ctx->launches;
        CRK_LAUNCH_CHECK(ctx, "list layout");
        if (ctx->graph_mode) {   // captured step: capacities were fixed beforehand, overflow checked after
            ctx->lists_valid = 1;
            return CRK_OK;
        }
        rc = crk_sync_counters(ctx, s);
        if (rc) return rc;
        long long maxc = (long long)ctx->h_counters[CNT_MAXCNT];
        if (maxc <= ctx->kcap) {
            long long units = (long long)ctx->h_counters[CNT_ENTRIES];
            rc = crk_ensure_entries(ctx, -1, units * 32);
            if (rc) return rc;
            ctx->entries = units * 32;
            ctx->lists_valid = 1;
            return CRK_OK;
        }
        ctx->kcap = (int)((maxc + maxc / 4 + 31) / 32 * 32);
    }
    return crk_set_error(ctx, CRK_ECAPACITY, "neighbour lists keep overflowing");
}

// The lists the passes walk, exported in caller order, from off[perm[s]] for slot
// s: mode 0: its gather set (self first, then the gather entries) as caller index |
// (i in gather(j)) << 31; mode 1: its pair set (gather entries, then the others) as
// caller indices.  A warp takes a particle, so that the output is written in whole
// lines (a thread per particle wrote single words: mode 0 at 16^3, 40^3, 64^3 70, 136,
// 713 us, 14, 71, 215 so).
__global__ void k_export_lists(int n, int kcap, int mode, const int32_t *__restrict__ perm,
                               const int32_t *__restrict__ cnt_g, const int32_t *__restrict__ cnt_u,
                               const uint32_t *__restrict__ ent, const uint4 *__restrict__ q4,
                               const long long *__restrict__ off, int32_t *__restrict__ out) {
    grid_wait();
    const int s = (int)((blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (s >= n) return;
    const int tile = s / TILE, i = s % TILE;
    const uint32_t *col0 = ent + (size_t)tile * kcap * 32;
    const int ci = perm[s], cg = min(cnt_g[s], kcap), nbg = list_blocks(cg), co = min(cnt_u[s] - cnt_g[s], kcap);
    const uint4 qi = q4[s];
    int32_t *o = out + off[ci];
    if (mode == 0) {
        if (lane == 0) o[0] = (int32_t)((uint32_t)ci | 0x80000000u);
        for (int k = lane; k < cg; k += 32) {
            const uint32_t e = col0[block_at(k / LB, i) + k % LB];
            const uint4 qj = q4[e];
            const unsigned long long R2 = r2_fixed((int)(qi.x - qj.x), (int)(qi.y - qj.y), (int)(qi.z - qj.z));
            o[1 + k] = (int32_t)((uint32_t)perm[e] | (R2 < (unsigned long long)qj.w * qj.w ? 0x80000000u : 0u));
        }
    } else {
        for (int k = lane; k < cg + co; k += 32) {
            const int r = k - cg, b = r < 0 ? k / LB : pair_block(nbg + r / LB, nbg, kcap);
            o[k] = perm[col0[block_at(b, i) + (r < 0 ? k : r) % LB]];
        }
    }
}

int run_export_lists(crk_ctx *ctx, int mode, const long long *off, int32_t *out, cudaStream_t s) {
    if (ctx->n == 0) return CRK_OK;
    int rc = run_lists(ctx, s);
    if (rc) return rc;
    launch(s, grid_for(32ll * ctx->n, 256), 256, 0, k_export_lists, ctx->n, ctx->kcap, mode, ctx->perm, ctx->cnt_g,
           ctx->cnt_u, ctx->ent, ctx->q4, off, out);
    ++ctx->launches;
    CRK_LAUNCH_CHECK(ctx, "export lists");
    return CRK_OK;
}

// P1 volumes over the gather lists (eq:vol, eq:hi), self included.
struct P1 {
    static constexpr bool GATHER = true;
    static constexpr int UNROLL = 4;
    static constexpr bool ENTRIES = true;
    static constexpr bool PERSISTENT = false;
    static constexpr bool PREFETCH = false;
    using Rec = uint4;
    struct Params {
        const uint4 *q4;
        const float *hs;
        float *V, *Nn;
        uint4 *qV;
    };
    struct IState {
        uint4 q;
        float h, inv_h, acc;
    };
    __device__ static void init(IState &s, int i, bool valid, const Params &p) {
        s.q = valid ? p.q4[i] : make_uint4(0, 0, 0, 0);
        s.h = valid ? p.hs[i] : 1.f;
        s.inv_h = 1.f / s.h;
        s.acc = 1.f;                                   // self: W(0) / (495/(32 pi h^3)) = 1
    }
    __device__ static void zero(IState &s) { s.acc = 0.f; }
    using Sums = float;
    __device__ static Sums sums(const IState &s) { return s.acc; }
    __device__ static void merge(IState &s, Sums o) { s.acc += o; }
    __device__ static Rec load(uint32_t j, size_t, const Params &p) { return __ldg(p.q4 + j); }
    __device__ static void pair(IState &s, const Rec &r, uint32_t, size_t, bool ok, const Params &) {
        const float eta =
            distance32((int)(s.q.x - r.x), (int)(s.q.y - r.y), (int)(s.q.z - r.z)) * (TWO_M32 * s.inv_h);
        float t = ok ? __saturatef(1.f - eta) : 0.f;
        float t2 = t * t, t3 = t2 * t;
        s.acc = fmaf(t3 * t3, fmaf(eta, fmaf(eta, K35_3, 6.f), 1.f), s.acc);
    }
    __device__ static void finish(IState &s, int i, const Params &p) {
        float ih3 = s.inv_h * s.inv_h * s.inv_h;
        float nsum = KW * ih3 * s.acc;                       // n_i, eq:vol
        float V = 1.f / nsum;
        p.V[i] = V;
        if (p.Nn) p.Nn[i] = (K4PI_3 * s.h * s.h * s.h) * nsum;   // eq:hi
        p.qV[i] = make_uint4(s.q.x, s.q.y, s.q.z, __float_as_uint(V));
    }
};

// P1 volumes: the walk (if the lists are stale) and the list pass; a
// volumes-only context sums n_i inside the walk instead.
int run_volumes(crk_ctx *ctx, cudaStream_t s) {
    if (ctx->n == 0) return CRK_OK;
    if (ctx->volumes_only) {
        ctx->lists_valid = 0;
        return launch_walk(ctx, s);
    }
    int rc = run_lists(ctx, s);
    if (rc) return rc;
    P1::Params p{ctx->q4, ctx->hs, ctx->V, ctx->Nn, ctx->qV};
    return launch_lpass<P1, 8>(ctx, PROF_P1, p, s, "P1 volumes");
}

}  // namespace crk
