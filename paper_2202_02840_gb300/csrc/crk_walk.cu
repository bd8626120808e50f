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
    int2 *lowc;              // may be null: per particle, gather and other entries with j < i
    unsigned long long *tests;   // lane tests of the exact predicate (LISTS walk)
};

// LISTS: write the lists; VOL: sum n_i in the walk (volumes-only contexts).
// circular distance (fixed point) from coordinate q to the arc [lo, hi]
// (which may wrap, lo > hi); differences modulo 2^32
__device__ __forceinline__ unsigned long long point_gap(uint32_t q, uint32_t lo, uint32_t hi) {
    if (q - lo <= hi - lo) return 0ull;
    uint32_t d1 = lo - q, d2 = q - hi;
    return (unsigned long long)(d1 < d2 ? d1 : d2);
}

// One segment of a lane's list on its way to memory: the last up to three
// entries wait in registers (newest in p3) until their block is full.
struct Seg {
    uint32_t p1, p2, p3;
    int n;   // entries so far
    uint32_t *at;   // the next block
    __device__ __forceinline__ void push(uint32_t j, int kcap, ptrdiff_t step) {
        ++n;
        if ((n & (LB - 1)) == 0) {
            if (n <= kcap) *reinterpret_cast<uint4 *>(at) = make_uint4(p1, p2, p3, j);
            at += step;
        }
        p1 = p2;
        p2 = p3;
        p3 = j;
    }
    // the last, partial block, padded with the lane's own index
    __device__ __forceinline__ void close(uint32_t self, int kcap) {
        const int r = n & (LB - 1);
        if (r == 0 || n > kcap) return;
        *reinterpret_cast<uint4 *>(at) = r == 1 ? make_uint4(p3, self, self, self)
                                       : (r == 2 ? make_uint4(p2, p3, self, self) : make_uint4(p1, p2, p3, self));
    }
};
constexpr ptrdiff_t BLOCK_WORDS = LB * 32;

// Rounding margin of the walk's FP32 comparisons.  Coordinates are offsets from
// the tile's box corner, exact integers of at most M (the two tiles' extents
// plus the larger support, < 2^31, so an offset is the minimum image) rounded
// to FP32: each is off by at most u M (u = 2^-24), a difference d by 3 u M, a
// squared distance r^2 <= 3 M^2 by 2 sqrt(3) r 3 u M + 3 u r^2 <= 27 u M^2 and a
// squared support by 3 u M^2.  A comparison of the two that clears 48 u M^2 has
// the sign of the exact one.
constexpr float WALK_MARGIN = 48.f / 16777216.f;
constexpr float FAR = 1e18f;   // coordinate of the padding slots: in nobody's reach

// The exact predicate of one kept particle (bits of its slot p): in gather(i), i in gather(j).
__device__ __forceinline__ void exact_bits(const uint4 &qi, unsigned long long Hi2, const uint4 &qj, bool same_box,
                                           int p, unsigned &gm, unsigned &jm) {
    const unsigned long long R2 =
        same_box ? r2_fixed((int)(qi.x - qj.x), (int)(qi.y - qj.y), (int)(qi.z - qj.z)) : ~0ull;
    gm |= (R2 < Hi2 ? 1u : 0u) << p;
    jm |= (R2 < (unsigned long long)qj.w * qj.w ? 1u : 0u) << p;
}

// BATCH: the particles belong to independent boxes; j can be a neighbour of i
// only in i's box (the box ranges of tiles prune the rest).
//
// LISTS.  Bound by instruction issue: each lane tests every kept particle of
// each candidate tile, and about one test in five finds an entry.  A test is
// the FP32 difference of tile-relative coordinates against both squared
// supports (3 add, 3 multiply-add, 2 add, a running minimum of the distance to
// either threshold and one funnel shift per mask: 13 instructions against 27 of
// the 64-bit integer test); the integer predicate runs only for a candidate
// tile where some lane came within the rounding margin of a threshold (about 1
// in 500), whose tiles span half the box or more, or which holds several
// batched boxes, so the lists are the exact ones.  The kept particles are
// compacted in shared memory, so the loop has no bit scans.
//
// VOL.  Sums n_i instead of writing lists: W vanishes beyond h_i, so every kept
// particle is summed without the predicate, and only particles within the
// tile's own supports are kept.
template <bool LISTS, bool VOL, bool BATCH>
__global__ void __launch_bounds__(WALK_WARPS * 32, 4) k_walk(WalkArgs a) {
    __shared__ float4 sf[LISTS ? WALK_WARPS : 1][32];        // kept: x, y, z (tile-relative), H^2
    __shared__ uint4 sq[WALK_WARPS][32];                     // kept: fixed-point record
    __shared__ uint32_t sid[LISTS ? WALK_WARPS : 1][32];     // kept: sorted index
    __shared__ int32_t sb[WALK_WARPS][BATCH ? 32 : 1];       // kept: box
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int tw = blockIdx.x * WALK_WARPS + w;
    if (tw >= a.ntiles) return;
    const int tile = a.act ? a.act[tw] : tw;
    const int i = tile * TILE + lane;
    const bool valid = i < a.n;
    const uint4 qi = valid ? a.q4[i] : make_uint4(0, 0, 0, 0);
    const unsigned long long Hi2 = (unsigned long long)qi.w * qi.w;   // 0 for invalid lanes
    const float h = VOL && valid ? a.hs[i] : 1.f;
    const float inv_h = 1.f / h;
    const int kcap = a.kcap;
    uint32_t *const col0 = LISTS ? a.ent + (size_t)tile * kcap * 32 : nullptr;
    float acc = 0.f;
    Seg G{0u, 0u, 0u, 0, LISTS ? col0 + block_at(0, lane) : nullptr};
    Seg O{0u, 0u, 0u, 0, LISTS ? col0 + block_at(kcap / LB - 1, lane) : nullptr};
    int lg = 0, lo_ = 0;   // entries with j < i: the candidate tiles come in ascending order
    uint32_t ntest = 0;    // kept staged particles (warp-uniform)
    const uint2 lo = a.ofs[tile];
    const uint4 Ilo = __ldg(a.tlo + tile), Ihi = __ldg(a.thi + tile);   // this tile's box, max H
    const int32_t bi = BATCH && valid ? a.sbox[i] : 0;
    const uint32_t Ib = BATCH ? __ldg(a.nbox + tile) : 0u;
    // this tile and this lane relative to the box corner
    const uint32_t Iex = Ihi.x - Ilo.x, Iey = Ihi.y - Ilo.y, Iez = Ihi.z - Ilo.z;
    const uint32_t Ie = max(max(Iex, Iey), Iez);
    const float ex = (float)Iex, ey = (float)Iey, ez = (float)Iez;
    const float fx = (float)(qi.x - Ilo.x), fy = (float)(qi.y - Ilo.y), fz = (float)(qi.z - Ilo.z);
    const float Hf = (float)qi.w, Hf2 = Hf * Hf;
    // software pipeline over the candidate tiles: the tile id two ahead, and
    // the box and this lane's staged particle of the next tile, are in flight
    // while the current tile is tested (each is otherwise a dependent L2 trip)
    const uint32_t *tl = a.tiles + lo.x;
    const int nt = (int)lo.y;
    int J1 = nt > 0 ? (int)__ldg(tl) : 0, J2 = nt > 1 ? (int)__ldg(tl + 1) : 0;
    uint4 lo1 = make_uint4(0, 0, 0, 0), hi1 = lo1, qn = lo1;
    if (nt > 0) {
        lo1 = __ldg(a.tlo + J1);
        hi1 = __ldg(a.thi + J1);
        if (J1 * TILE + lane < a.n) qn = __ldg(a.q4 + J1 * TILE + lane);
    }
    for (int t = 0; t < nt; t++) {
        const int J = J1;
        const uint4 Jlo = lo1, Jhi = hi1, qc = qn;
        J1 = J2;
        if (t + 2 < nt) J2 = (int)__ldg(tl + t + 2);
        if (t + 1 < nt) {
            lo1 = __ldg(a.tlo + J1);
            hi1 = __ldg(a.thi + J1);
            if (J1 * TILE + lane < a.n) qn = __ldg(a.q4 + J1 * TILE + lane);
        }
        const int j0 = J * TILE;
        const int cnt = min(TILE, a.n - j0);
        const uint32_t Jex = Jhi.x - Jlo.x, Jey = Jhi.y - Jlo.y, Jez = Jhi.z - Jlo.z;
        const uint32_t HJ = VOL ? 0u : Jlo.w;   // the volumes take gather(i) only
        const uint32_t Hm = max(Ilo.w, HJ);
        const unsigned long long M =
            (unsigned long long)Ie + max(max(Jex, Jey), Jez) + max(Ilo.w, Jlo.w);   // warp-uniform
        const bool wide = M >= 0x7fffffffull;   // offsets may not be the minimum image
        const float margin = WALK_MARGIN * ((float)M * (float)M);
        // lane jj stages particle j0 + jj and keeps it only if it can be in the
        // pair set (VOL: the gather set) of some particle of this tile: its gap
        // to the tile's box below the larger support.  Skip a tile that no
        // lane's sphere touches.  Conservative, so the lists are unchanged.
        bool near, keep;
        float jx = 0.f, jy = 0.f, jz = 0.f;
        if (!wide) {
            const int ox = (int)(Jlo.x - Ilo.x), oy = (int)(Jlo.y - Ilo.y), oz = (int)(Jlo.z - Ilo.z);
            const float lx = (float)ox, ly = (float)oy, lz = (float)oz;
            const float gx = fmaxf(fmaxf(lx - fx, fx - (float)(int)((uint32_t)ox + Jex)), 0.f);
            const float gy = fmaxf(fmaxf(ly - fy, fy - (float)(int)((uint32_t)oy + Jey)), 0.f);
            const float gz = fmaxf(fmaxf(lz - fz, fz - (float)(int)((uint32_t)oz + Jez)), 0.f);
            const float re = fmaxf(Hf, (float)HJ);
            near = valid && fmaf(gx, gx, fmaf(gy, gy, gz * gz)) < fmaf(re, re, margin);
            jx = (float)(int)(qc.x - Ilo.x);
            jy = (float)(int)(qc.y - Ilo.y);
            jz = (float)(int)(qc.z - Ilo.z);
            const float hx = fmaxf(fmaxf(-jx, jx - ex), 0.f), hy = fmaxf(fmaxf(-jy, jy - ey), 0.f),
                        hz = fmaxf(fmaxf(-jz, jz - ez), 0.f);
            const float rj = (float)(VOL ? Ilo.w : max(qc.w, Ilo.w));
            keep = lane < cnt && fmaf(hx, hx, fmaf(hy, hy, hz * hz)) < fmaf(rj, rj, margin);
        } else {
            const unsigned long long gx = point_gap(qi.x, Jlo.x, Jhi.x), gy = point_gap(qi.y, Jlo.y, Jhi.y),
                                     gz = point_gap(qi.z, Jlo.z, Jhi.z);
            const unsigned long long reach = max(qi.w, HJ);
            near = valid && gx * gx + gy * gy + gz * gz < reach * reach;
            const unsigned long long hx = point_gap(qc.x, Ilo.x, Ihi.x), hy = point_gap(qc.y, Ilo.y, Ihi.y),
                                     hz = point_gap(qc.z, Ilo.z, Ihi.z);
            const unsigned long long rj = VOL ? Hm : max(qc.w, Ilo.w);
            keep = lane < cnt && hx * hx + hy * hy + hz * hz < rj * rj;
        }
        bool mixed = false;   // the pair's boxes must be compared
        int32_t bj = 0;
        if constexpr (BATCH) {
            const uint32_t Jb = __ldg(a.nbox + J);
            near = near && (uint32_t)bi >= (Jb & 0xffffu) && (uint32_t)bi <= (Jb >> 16);
            mixed = Ib != Jb || (Ib & 0xffffu) != (Ib >> 16);
            if (mixed && lane < cnt) {
                bj = __ldg(a.sbox + j0 + lane);
                keep = keep && (uint32_t)bj >= (Ib & 0xffffu) && (uint32_t)bj <= (Ib >> 16);
            }
        }
        if (__ballot_sync(0xffffffffu, near) == 0u) continue;
        const unsigned mask = __ballot_sync(0xffffffffu, keep);
        if (mask == 0u) continue;
        const int nk = __popc(mask), nk4 = (nk + 3) & ~3;
        ntest += (uint32_t)nk;   // every lane tests every kept particle
        const int slot = __popc(mask & lanemask_lt());
        __syncwarp();
        if (keep) {
            sq[w][slot] = qc;
            if (LISTS) {
                const float hj = (float)qc.w;
                sf[w][slot] = make_float4(jx, jy, jz, hj * hj);
                sid[w][slot] = (uint32_t)(j0 + lane);
            }
            if (BATCH) sb[w][slot] = bj;
        }
        if (lane < nk4 - nk) {
            if (LISTS) sf[w][nk + lane] = make_float4(FAR, FAR, FAR, 0.f);
            if (VOL) sq[w][nk + lane] = make_uint4(0, 0, 0, 0);
        }
        __syncwarp();
        if constexpr (LISTS) {
            // gm: j in gather(i); jm: i in gather(j); bit = slot
            unsigned gm = 0u, jm = 0u;
            bool exact = wide || mixed;
            if (!exact) {
                float amb = 3.0e38f;
                for (int p = nk4 - 4; p >= 0; p -= 4) {   // four independent chains; slot 0 ends at bit 0
#pragma unroll
                    for (int u = 3; u >= 0; u--) {
                        const float4 f = sf[w][p + u];
                        const float dx = fx - f.x, dy = fy - f.y, dz = fz - f.z;
                        const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
                        const float ti = r2 - Hf2, tj = r2 - f.w;
                        amb = fminf(amb, fminf(fabsf(ti), fabsf(tj)));
                        gm = __funnelshift_l(__float_as_uint(ti), gm, 1);
                        jm = __funnelshift_l(__float_as_uint(tj), jm, 1);
                    }
                }
                exact = __any_sync(0xffffffffu, valid && amb < margin);
            }
            if (exact) {
                gm = jm = 0u;
                for (int p = 0; p < nk; p++)
                    exact_bits(qi, Hi2, sq[w][p], !BATCH || !mixed || sb[w][p] == bi, p, gm, jm);
            }
            if (!valid) gm = jm = 0u;
            if (J <= tile) {
                unsigned below = 0xffffffffu;
                if (J == tile) {   // j != i (particle i is kept, in slot `slot`)
                    below = (1u << slot) - 1u;
                    gm &= ~(1u << slot);
                    jm &= ~(1u << slot);
                }
                lg = G.n + __popc(gm & below);
                lo_ = O.n + __popc(jm & ~gm & below);
            }
            // each lane appends its own entries in staging order
            jm &= ~gm;
            while (gm) {
                const int p = __ffs(gm) - 1;
                gm &= gm - 1u;
                G.push(sid[w][p], kcap, BLOCK_WORDS);
            }
            while (jm) {
                const int p = __ffs(jm) - 1;
                jm &= jm - 1u;
                O.push(sid[w][p], kcap, -BLOCK_WORDS);
            }
        } else {
            for (int p = 0; p < nk4; p += 4) {
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    const uint4 qj = sq[w][p + u];
                    Sep d = separation((int)(qi.x - qj.x), (int)(qi.y - qj.y), (int)(qi.z - qj.z));
                    const float eta = d.r * inv_h;
                    float tt = __saturatef(1.f - eta);
                    if (p + u >= nk) tt = 0.f;
                    if (BATCH && mixed && p + u < nk && sb[w][p + u] != bi) tt = 0.f;
                    const float t2 = tt * tt, t3 = t2 * tt;
                    acc = fmaf(t3 * t3, fmaf(eta, fmaf(eta, K35_3, 6.f), 1.f), acc);
                }
            }
        }
    }
    const int cu = G.n + O.n;
    const int rg = LB * list_blocks(G.n), ru = rg + LB * list_blocks(O.n);   // rows with the pads
    if (valid) {
        if (VOL) {
            float ih3 = inv_h * inv_h * inv_h;
            float nsum = KW * ih3 * acc;                       // n_i, eq:vol
            a.V[i] = 1.f / nsum;
            if (a.Nn) a.Nn[i] = (K4PI_3 * h * h * h) * nsum;   // eq:hi
        }
        if (LISTS) {
            G.close((uint32_t)i, kcap);
            O.close((uint32_t)i, kcap);
        }
        a.cnt_g[i] = G.n;
        a.cnt_u[i] = cu;
        if (LISTS && a.lowc) a.lowc[i] = make_int2(lg, lo_);
    }
    uint32_t mg = __reduce_max_sync(0xffffffffu, (uint32_t)rg);
    uint32_t mu = __reduce_max_sync(0xffffffffu, (uint32_t)ru);
    uint32_t sg = __reduce_add_sync(0xffffffffu, (uint32_t)G.n);
    uint32_t su = __reduce_add_sync(0xffffffffu, (uint32_t)cu);
    if (lane == 0) {
        a.len_g[tile] = min(mg, (uint32_t)kcap);
        a.len_u[tile] = min(mu, (uint32_t)kcap);
        atomicAdd(a.pairs_g, (unsigned long long)sg);
        atomicAdd(a.pairs_u, (unsigned long long)su);
        atomicMax(a.maxcnt, (unsigned long long)mu);
        if (LISTS) atomicAdd(a.tests, 32ull * ntest);
    }
}

// The walk for few tiles (time bins, act set): S warps share one tile, warp w
// testing the candidate tiles [w chunk, (w+1) chunk) of its list.  A first
// sweep counts every lane's gather and other neighbours per warp; their
// prefix over the warps gives each warp its columns, and a second sweep
// writes the entries there, so every list is exactly the one-warp walk's.
template <int S>
__global__ void __launch_bounds__(S * 32) k_walk_split(WalkArgs a) {
    __shared__ uint4 sq[S][32];
    __shared__ int cnt[2][S][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int tile = a.act[blockIdx.x];
    const int i = tile * TILE + lane;
    const bool valid = i < a.n;
    const uint4 qi = valid ? a.q4[i] : make_uint4(0, 0, 0, 0);
    const unsigned long long Hi2 = (unsigned long long)qi.w * qi.w;
    const int kcap = a.kcap;
    uint32_t *const col0 = a.ent + (size_t)tile * kcap * 32;
    auto word = [&](int c) -> uint32_t * { return col0 + block_at(c / LB, lane) + c % LB; };   // gather entry c
    auto back = [&](int c) -> uint32_t * { return col0 + block_at(kcap / LB - 1 - c / LB, lane) + c % LB; };
    const uint2 lo = a.ofs[tile];
    const uint4 Ilo = __ldg(a.tlo + tile), Ihi = __ldg(a.thi + tile);
    const int nt = (int)lo.y;
    const int chunk = (nt + S - 1) / S;
    const int t0 = w * chunk, t1 = min(nt, t0 + chunk);
    int base_g = 0, base_o = 0, tot_g = 0, tot_o = 0;
    for (int phase = 0; phase < 2; phase++) {
        int cg = 0, co = 0;
        for (int t = t0; t < t1; t++) {
            const int J = (int)__ldg(a.tiles + lo.x + t);
            const uint4 Jlo = __ldg(a.tlo + J), Jhi = __ldg(a.thi + J);
            const unsigned long long gx = point_gap(qi.x, Jlo.x, Jhi.x), gy = point_gap(qi.y, Jlo.y, Jhi.y),
                                     gz = point_gap(qi.z, Jlo.z, Jhi.z);
            const unsigned long long reach = qi.w > Jlo.w ? qi.w : Jlo.w;
            const bool near = valid && gx * gx + gy * gy + gz * gz < reach * reach;
            if (__ballot_sync(0xffffffffu, near) == 0u) continue;
            const int j0 = J * TILE;
            const int cj = min(TILE, a.n - j0);
            __syncwarp();
            bool keep = false;
            if (lane < cj) {
                const uint4 q = __ldg(a.q4 + j0 + lane);
                sq[w][lane] = q;
                const unsigned long long hx = point_gap(q.x, Ilo.x, Ihi.x), hy = point_gap(q.y, Ilo.y, Ihi.y),
                                         hz = point_gap(q.z, Ilo.z, Ihi.z);
                const unsigned long long rj = q.w > Ilo.w ? q.w : Ilo.w;
                keep = hx * hx + hy * hy + hz * hz < rj * rj;
            }
            unsigned mask = __ballot_sync(0xffffffffu, keep);
            __syncwarp();
            auto visit = [&](int jj, const uint4 &qj, unsigned long long R2) {
                const uint32_t j = (uint32_t)(j0 + jj);
                if (valid && (int)j != i) {
                    const bool in_i = R2 < Hi2;
                    const bool in_j = R2 < (unsigned long long)qj.w * qj.w;
                    if (in_i) {
                        const int c = base_g + cg;
                        if (phase == 1 && c < kcap) *word(c) = j;
                        cg++;
                    } else if (in_j) {
                        const int c = base_o + co;
                        if (phase == 1 && c < kcap) *back(c) = j;
                        co++;
                    }
                }
            };
            while (mask) {   // two staged neighbours per iteration, in staging order
                const int ja = __ffs(mask) - 1;
                mask &= mask - 1u;
                const bool two = mask != 0u;
                const int jb = two ? __ffs(mask) - 1 : ja;
                if (two) mask &= mask - 1u;
                const uint4 qa = sq[w][ja], qb = sq[w][jb];
                const unsigned long long Ra = r2_fixed((int)(qi.x - qa.x), (int)(qi.y - qa.y), (int)(qi.z - qa.z));
                const unsigned long long Rb = r2_fixed((int)(qi.x - qb.x), (int)(qi.y - qb.y), (int)(qi.z - qb.z));
                visit(ja, qa, Ra);
                if (two) visit(jb, qb, Rb);
            }
        }
        if (phase == 0) {
            cnt[0][w][lane] = cg;
            cnt[1][w][lane] = co;
            __syncthreads();
            for (int v = 0; v < S; v++) {
                if (v < w) {
                    base_g += cnt[0][v][lane];
                    base_o += cnt[1][v][lane];
                }
                tot_g += cnt[0][v][lane];
                tot_o += cnt[1][v][lane];
            }
        }
    }
    if (w != 0) return;
    const int cu = tot_g + tot_o;
    const int rg = LB * list_blocks(tot_g), ru = rg + LB * list_blocks(tot_o);
    if (valid) {
        for (int c = tot_g; c < min(rg, kcap); c++) *word(c) = (uint32_t)i;   // pads
        for (int c = tot_o; c < min(ru - rg, kcap); c++) *back(c) = (uint32_t)i;
        a.cnt_g[i] = tot_g;
        a.cnt_u[i] = cu;
    }
    uint32_t mg = __reduce_max_sync(0xffffffffu, (uint32_t)rg);
    uint32_t mu = __reduce_max_sync(0xffffffffu, (uint32_t)ru);
    uint32_t sg = __reduce_add_sync(0xffffffffu, (uint32_t)tot_g);
    uint32_t su = __reduce_add_sync(0xffffffffu, (uint32_t)cu);
    if (lane == 0) {
        a.len_g[tile] = min(mg, (uint32_t)kcap);
        a.len_u[tile] = min(mu, (uint32_t)kcap);
        atomicAdd(a.pairs_g, (unsigned long long)sg);
        atomicAdd(a.pairs_u, (unsigned long long)su);
        atomicMax(a.maxcnt, (unsigned long long)mu);
    }
}

// total stored-force units (32 entries each) = base[last] + len_u[last]
__global__ void k_total(int ntiles, const uint32_t *__restrict__ base, const uint32_t *__restrict__ len,
                        unsigned long long *out) {
    *out = ntiles ? (unsigned long long)base[ntiles - 1] + len[ntiles - 1] : 0ull;
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
    a.lowc = ctx->volumes_only ? nullptr : ctx->lowc;
    a.tests = ctx->counters + CNT_WALK_TESTS;
    return a;
}

static int launch_walk(crk_ctx *ctx, cudaStream_t s) {
    if (!ctx->volumes_only) {
        int rc = crk_ensure_entries(ctx, (long long)ctx->ntiles * 32 * ctx->kcap, -1);
        if (rc) return rc;
    }
    CRK_CUDA(ctx, cudaMemsetAsync(ctx->counters + CNT_PAIRS_G, 0, 2 * sizeof(unsigned long long), s));
    CRK_CUDA(ctx, cudaMemsetAsync(ctx->counters + CNT_MAXCNT, 0, sizeof(unsigned long long), s));
    CRK_CUDA(ctx, cudaMemsetAsync(ctx->counters + CNT_WALK_TESTS, 0, sizeof(unsigned long long), s));
    if (ctx->act) {   // tiles left out of the walk take no list columns and no stored forces
        CRK_CUDA(ctx, cudaMemsetAsync(ctx->len_g, 0, sizeof(uint32_t) * ctx->ntiles, s));
        CRK_CUDA(ctx, cudaMemsetAsync(ctx->len_u, 0, sizeof(uint32_t) * ctx->ntiles, s));
        if (ctx->nact == 0) return CRK_OK;
    }
    prof_begin(ctx, PROF_LISTS, s);
    const int g = grid_for(ctx->act ? ctx->nact : ctx->ntiles, WALK_WARPS);
    const bool b = ctx->nbox > 1;
    const int nsm = ctx->nsm > 0 ? ctx->nsm : 152;
    if (ctx->act && !ctx->volumes_only && !b && ctx->nact < 8 * nsm)   // few tiles: 8 warps per tile
        k_walk_split<8><<<ctx->nact, 8 * 32, 0, s>>>(walk_args(ctx));
    else if (ctx->volumes_only && b)
        k_walk<false, true, true><<<g, WALK_WARPS * 32, 0, s>>>(walk_args(ctx));
    else if (ctx->volumes_only)
        k_walk<false, true, false><<<g, WALK_WARPS * 32, 0, s>>>(walk_args(ctx));
    else if (b)
        k_walk<true, false, true><<<g, WALK_WARPS * 32, 0, s>>>(walk_args(ctx));
    else
        k_walk<true, false, false><<<g, WALK_WARPS * 32, 0, s>>>(walk_args(ctx));
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
        k_total<<<1, 1, 0, s>>>(nt, ctx->tbase, ctx->len_u, ctx->counters + CNT_ENTRIES);
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

// The lists the passes walk, exported in caller order: thread per sorted slot
// s writes, from off[perm[s]], mode 0: its gather set (self first, then the
// gather entries) as caller index | (i in gather(j)) << 31; mode 1: its pair
// set (gather entries, then the others) as caller indices.
__global__ void k_export_lists(int n, int kcap, int mode, const int32_t *__restrict__ perm,
                               const int32_t *__restrict__ cnt_g, const int32_t *__restrict__ cnt_u,
                               const uint32_t *__restrict__ ent, const uint4 *__restrict__ q4,
                               const long long *__restrict__ off, int32_t *__restrict__ out) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    const int tile = s / TILE, lane = s % TILE;
    const uint32_t *col0 = ent + (size_t)tile * kcap * 32;
    const int ci = perm[s];
    long long o = off[ci];
    const int cg = min(cnt_g[s], kcap), nbg = list_blocks(cg), co = min(cnt_u[s] - cnt_g[s], kcap);
    const uint4 qi = q4[s];
    if (mode == 0) out[o++] = (int32_t)((uint32_t)ci | 0x80000000u);
    for (int k = 0; k < cg; k++) {
        const uint32_t e = col0[block_at(k / LB, lane) + k % LB];
        uint32_t j = (uint32_t)perm[e];
        if (mode == 0) {
            const uint4 qj = q4[e];
            const unsigned long long R2 = r2_fixed((int)(qi.x - qj.x), (int)(qi.y - qj.y), (int)(qi.z - qj.z));
            if (R2 < (unsigned long long)qj.w * qj.w) j |= 0x80000000u;
        }
        out[o++] = (int32_t)j;
    }
    if (mode == 1)
        for (int k = 0; k < co; k++)
            out[o++] = perm[col0[block_at(pair_block(nbg + k / LB, nbg, kcap), lane) + k % LB]];
}

int run_export_lists(crk_ctx *ctx, int mode, const long long *off, int32_t *out, cudaStream_t s) {
    if (ctx->n == 0) return CRK_OK;
    int rc = run_lists(ctx, s);
    if (rc) return rc;
    k_export_lists<<<grid_for(ctx->n, 256), 256, 0, s>>>(ctx->n, ctx->kcap, mode, ctx->perm, ctx->cnt_g, ctx->cnt_u,
                                                          ctx->ent, ctx->q4, off, out);
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
    __device__ static void merge(IState &s, const IState &o) { s.acc += o.acc; }
    __device__ static Rec load(uint32_t j, size_t, const Params &p) { return __ldg(p.q4 + j); }
    __device__ static void pair(IState &s, const Rec &r, uint32_t, size_t, bool ok, const Params &) {
        int dx = (int)(s.q.x - r.x), dy = (int)(s.q.y - r.y), dz = (int)(s.q.z - r.z);
        Sep d = separation(dx, dy, dz);
        float eta = d.r * s.inv_h;
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
