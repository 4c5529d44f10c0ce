// ds_walk.cuh -- the warp-sized walk of the forward rasteriser: a warp is the
// unit of work, 32 pixels (an 8 x 4 block of a binning tile, eight blocks per
// tile) of one group of samples.
//
// Every warp takes its own blocks from a global counter, culls the tile's list
// against its block 32 triangles at a time (one triangle per lane), keeps the
// survivors in its own shared-memory stage and walks them.  No barrier of the
// CTA is involved.  With one tile per CTA of eight warps (ds_tile.cuh) the
// warps waited for the slowest of them at every staging round, staging used
// one or two of the eight, and the walk stepped over the triangles of the
// other warps.  The 8 x 4 block also keeps more lanes of a covering triangle
// active than rows of 16 or 32 pixels do.  Loops whose iterations are long or
// few are kept rolled: the warps of an SM are in different phases, so that
// large code is fetched again and again (90 KB made warps wait for
// instructions 9 of 24 cycles).
#pragma once

#include "ds_tile.cuh"

namespace ds {

constexpr int kBlkW = 8, kBlkH = 4;              // a warp's pixels
constexpr int kBlocksPerTile = kTilePix / 32;    // 8 in every tile shape
constexpr int kStage = 32;                       // staged triangles per warp and round
constexpr int kWarps = kTilePix / 32;            // warps of a CTA
// Staged triangles between two votes on the early exit (200,000 triangles at
// 1080p, binary opacity: every one 160 us, 2: 154, 4: 150, 8 and 16: 148).
constexpr int kExitEvery = 4;

// A warp's staged set-up: TileStage's terms relative to the block's first
// pixel.
struct WarpStage {
    int4 h0[kStage];      // A0, B0, s0, A1
    int4 h1[kStage];      // B1, s1, A2, B2
    int4 h2[kStage];      // s2, triangle | flags, r0, r1
    int4 h3[kStage];      // r2, k0, k1, k2 (float bits)
    float bound[kStage];  // upper bound on the inverse depth from this entry of the list on
};

// A block: its view, sample group, first pixel and list.
struct Block {
    int v, g, ox, oy;
    uint2 rg;
};

// Blocks are numbered view by view, then sample group, then tile, then block
// of the tile; one outside the view has an empty list.
__device__ __forceinline__ Block find_block(const ViewTable& vt, const uint2* __restrict__ ranges, unsigned id) {
    const int it = (int)(id / kBlocksPerTile), blk = (int)(id % kBlocksPerTile);
    Block b;
    int lo = 0, hi = vt.n - 1;
#pragma unroll 1
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (vt.v[mid].item_base <= it) lo = mid;
        else hi = mid - 1;
    }
    b.v = lo;
    const ViewDesc& V = vt.v[lo];
    const unsigned tiles = (unsigned)(V.tiles_x * V.tiles_y);
    const unsigned local = (unsigned)(it - V.item_base);
    b.g = (int)(local / tiles);
    const unsigned tile = local - b.g * tiles;
    const unsigned ty = tile / (unsigned)V.tiles_x, tx = tile - ty * V.tiles_x;
    const int bw = vt.tile_w >> 3;   // blocks per tile row: 1, 2 or 4
    b.ox = (int)tx * vt.tile_w + (blk & (bw - 1)) * kBlkW;
    b.oy = (int)ty * vt.tile_h + (blk / bw) * kBlkH;
    b.rg = b.ox < V.W && b.oy < V.H ? ranges[V.tile_base + (int)tile] : make_uint2(0u, 0u);
    return b;
}

// Fill the warp's stage from list position c on (at most kStage survivors;
// entries whose triangle covers none of the block's pixel centres, by the
// largest edge value over the block's corners, are dropped).  Returns the
// number staged; c is the first entry not taken.
__device__ __forceinline__ int fill_stage(WarpStage& st, const SetupRec* __restrict__ recs,
                                          const uint32_t* __restrict__ keys, const uint32_t* __restrict__ vals,
                                          uint32_t& c, uint32_t end, int DB, int ox, int oy, int lane) {
    const unsigned lt = (1u << lane) - 1u;
    int ns = 0;
    const int X0 = 256 * ox + 128, Y0 = 256 * oy + 128;
#pragma unroll 1
    while (c < end) {
        bool may = c + lane < end;
        SetupRec r;
        int sv[3], rl[3];
        uint32_t t = 0;
        if (may) {
            t = vals[c + lane];
            r = load_rec(recs + t);
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const long long eb = (long long)r.A[i] * X0 + (long long)r.B[i] * Y0 + r.C[i];
                const long long th = eb >> 8;
                sv[i] = th < -(1LL << 30) ? -(1 << 30) : (th > (1LL << 30) ? (1 << 30) : (int)th);
                rl[i] = (int)(eb & 255) + (int)((r.bias >> i) & 1u);
                const int top = (r.A[i] > 0 ? r.A[i] * (kBlkW - 1) : 0) + (r.B[i] > 0 ? r.B[i] * (kBlkH - 1) : 0);
                may = may && (top + sv[i] >= 0);
            }
        }
        const unsigned m = __ballot_sync(kFullMask, may);
        if (ns + __popc(m) > kStage) break;   // taken again in the next round
        if (may) {
            const int slot = ns + __popc(m & lt);
            if (llabs((long long)r.A[0] * r.B[1] - (long long)r.A[1] * r.B[0]) >= (1LL << 31)) t |= kBig;
            if (max(sv[0], max(sv[1], sv[2])) == 1 << 30) t |= kHuge;
            st.h0[slot] = make_int4(r.A[0], r.B[0], sv[0], r.A[1]);
            st.h1[slot] = make_int4(r.B[1], sv[1], r.A[2], r.B[2]);
            st.h2[slot] = make_int4(sv[2], (int)t, rl[0], rl[1]);
            st.h3[slot] = make_int4(rl[2], __float_as_int(r.k[0]), __float_as_int(r.k[1]), __float_as_int(r.k[2]));
            if (DB > 0) st.bound[slot] = rho_bound(keys[c + lane], DB);
        }
        ns += __popc(m);
        c = min(c + 32u, end);
    }
    __syncwarp();
    return ns;
}

// Coverage of block pixel (lx, ly) by staged triangle j (see tile_cover).
__device__ __forceinline__ bool stage_cover(const WarpStage& st, const SetupRec* __restrict__ recs, int j, int lx, int ly,
                                            int ox, int oy, int& t, Frag& f) {
    const int4 h0 = st.h0[j], h1 = st.h1[j], h2 = st.h2[j];
    const int s0 = h0.x * lx + (h0.y * ly + h0.z);
    const int s1 = h0.w * lx + (h1.x * ly + h1.y);
    const int s2 = h1.z * lx + (h1.w * ly + h2.x);
    if ((s0 | s1 | s2) < 0) return false;
    const int4 h3 = st.h3[j];
    t = h2.y & (int)kTriMask;
    float e0, e1, e2;
    if (!(h2.y & (int)(kBig | kHuge))) {
        e0 = __int2float_rn(h2.z + (s0 << 8));
        e1 = __int2float_rn(h2.w + (s1 << 8));
        e2 = __int2float_rn(h3.x + (s2 << 8));
    } else {
        long long E[3] = {h2.z + 256LL * s0, h2.w + 256LL * s1, h3.x + 256LL * s2};
        if (h2.y & (int)kHuge) cover_exact(load_rec(recs + t), ox + lx, oy + ly, E);
        e0 = __ll2float_rn(E[0]);
        e1 = __ll2float_rn(E[1]);
        e2 = __ll2float_rn(E[2]);
    }
    f = edge_frag(e0, e1, e2, __int_as_float(h3.y), __int_as_float(h3.z), __int_as_float(h3.w));
    return true;
}

// The masked z-test of one block (Eq. 5), as forward_walk.
template <int SG>
__device__ __forceinline__ void block_walk(WarpStage& st, const SetupRec* __restrict__ recs,
                                           const uint32_t* __restrict__ keys, const uint32_t* __restrict__ vals,
                                           const Block& b, int DB, const SoupDev& s, int lane, bool valid,
                                           int ns, uint2 seed, bool stochastic, int (&bt)[SG], float (&brho)[SG],
                                           float (&bb1)[SG], float (&bb2)[SG]) {
    const int lx = lane & (kBlkW - 1), ly = lane / kBlkW;
    uint32_t c = b.rg.x;
#pragma unroll 1
    while (c < b.rg.y) {
        __syncwarp();
        const int n = fill_stage(st, recs, keys, vals, c, b.rg.y, DB, b.ox, b.oy, lane);
#pragma unroll 1
        for (int j = 0; j < n; ++j) {
            if (DB > 0 && j % kExitEvery == 0) {
                bool ldone = true;
                if (valid) {
                    const float bound = st.bound[j];
#pragma unroll
                    for (int q = 0; q < SG; ++q)
                        if (q < ns) ldone = ldone && bt[q] >= 0 && brho[q] > bound;
                }
                if (__all_sync(kFullMask, ldone)) {
                    c = b.rg.y;
                    break;
                }
            }
            int t;
            Frag f;
            if (!valid || !stage_cover(st, recs, j, lx, ly, b.ox, b.oy, t, f)) continue;
            bool want[SG], need = false;
#pragma unroll
            for (int q = 0; q < SG; ++q) {
                want[q] = q < ns && (bt[q] < 0 || in_front(f.rho, t, brho[q], bt[q]));
                need = need || want[q];
            }
            if (!need) continue;
            const float r = __frcp_rn(f.rho);
            const float b1 = __fmul_rn(f.q1, r), b2 = __fmul_rn(f.q2, r);
            const Cell cl = find_cell(s.N, b1, b2);
            const float* aa = s.act_a + (size_t)t * s.V;
            const float alpha = interp(__ldg(aa + cl.k0), __ldg(aa + cl.k1), __ldg(aa + cl.k2), cl.wa, cl.wb);
            const int ka = __float2int_ru(__fmul_rn(alpha, 0x1p24f));
            int k[4] = {1 << 23, 1 << 23, 1 << 23, 1 << 23};   // tau = 1/2
            if (stochastic) {
                const uint4 w = philox4x32_10(make_uint4((uint32_t)(b.ox + lx), (uint32_t)(b.oy + ly), (uint32_t)t,
                                                         (uint32_t)b.g), seed.x, seed.y);
                k[0] = (int)(w.x >> 8);
                k[1] = (int)(w.y >> 8);
                k[2] = (int)(w.z >> 8);
                k[3] = (int)(w.w >> 8);
            }
#pragma unroll
            for (int q = 0; q < SG; ++q)
                if (want[q] && ka > k[q]) {
                    bt[q] = t;
                    brho[q] = f.rho;
                    bb1[q] = b1;
                    bb2[q] = b2;
                }
        }
    }
}

}  // namespace ds
