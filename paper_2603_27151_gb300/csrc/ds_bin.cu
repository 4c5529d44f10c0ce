// ds_bin.cu -- binning of the set-up triangles into tiles: a counting sort by
// tile, then a sort of each tile's list by (depth key, triangle).
//
// The set-up kernel counts the triangles of every tile (k_setup); the counts
// are scanned over the tiles; k_emit places each (tile, triangle) pair at its
// tile's cursor, in whatever order its atomics are served; k_tile_sort (with
// k_list_merge for lists above 2,048 entries) then gives every list its one
// order.  The early exit of the walks wants it front to back.  The triangle
// index breaks ties, and is the whole key when there are no depth bits: the
// forward's results do not depend on the order (its tie-break is by triangle
// index), but the backward sums the opacity terms of neighbouring list entries
// in FP32 before the FP64 accumulators, and those groups have to be the same in
// every call.  A call makes 4 launches here (5 above 4,096 tiles, one more
// where a list is above 2,048 entries or, without a host wait, can be) and a
// memset.  The radix sort of (tile, depth) keys that this replaces made 4
// passes of 5 launches over all pairs: 146 us of a 1.28 ms training step
// (239,566 pairs), 39 us of a 120 us render of 64 triangles.
#include <algorithm>

#include "ds_internal.h"

namespace ds {

namespace {
constexpr unsigned kFull = 0xffffffffu;
constexpr int kBinThreads = 256;
constexpr int kOwnTiles = 32;     // boxes of more tiles are shared by the warp (16 and 64 measure alike),
constexpr int kWarpTiles = 1024;  // those of more than this by the CTA
constexpr int kCtaBoxes = 64;     // as many of them as the CTA's list holds
}  // namespace

// Records per warp of k_setup and k_emit: 32, or fewer while there are not
// enough records for eight such warps per SM, so that a few triangles with
// large boxes are walked by the whole chip (500 full-screen triangles at
// 1280 x 720: k_setup 394 -> 32 us, k_emit 511 -> 41).  Sixteen warps per SM
// cost 1.5 us on 16,000 records.
static int records_per_warp(long long n_records) {
    const long long warps = persistent_grid(1 << 30, 8);
    int per = 1;
    while (per < 32 && n_records > per * warps) per *= 2;
    return per;
}

// A CTA's counter of a tile (its count in k_setup, its cursor in k_emit, which
// have the same records in the same CTAs): tile * step + first.
struct CounterAt {
    int step, first;
    __device__ explicit CounterAt(bool split)
        : step(split ? kSplitWays * kSplitWords : 1), first(split ? (int)(blockIdx.x % kSplitWays) * kSplitWords : 0) {}
};

// The record of this thread (-1: none).
__device__ __forceinline__ long long own_record(long long n_records, int per) {
    const long long warp = blockIdx.x * (long long)(kBinThreads / 32) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    const long long gid = warp * per + lane;
    return lane < per && gid < n_records ? gid : -1;
}

// Upper bound of the biased edge value over the tw x th pixel centres of a
// tile: a linear function peaks at a corner of the centre grid.
__device__ __forceinline__ bool tile_may_cover(const SetupRec& r, int tx, int ty, int tw, int th) {
    const long long X0 = 256LL * (tw * tx) + 128, Y0 = 256LL * (th * ty) + 128;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const long long e0 = (long long)r.A[i] * X0 + (long long)r.B[i] * Y0 + r.C[i];
        const long long up = 256LL * ((long long)(tw - 1) * (r.A[i] > 0 ? r.A[i] : 0) +
                                      (long long)(th - 1) * (r.B[i] > 0 ? r.B[i] : 0));
        if (e0 + up < 0) return false;
    }
    return true;
}

// A box that the CTA walks together.
struct CtaBox {
    SetupRec r;
    int4 box;
    int v, t;
    uint32_t zkey;
};

// Calls f(tiles, in, triangle, depth key) for the tiles of the lane's box, four
// at a time: global tile tiles[k] is one whose pixel centres the triangle may
// cover if in[k].  All threads of the CTA call it (an empty box has z < x).  A
// lane walks a box of a few tiles itself; the tiles of a larger one are spread
// over the warp, those of a very large one over the CTA (a full-screen triangle
// has thousands, and each costs an atomic's round trip in k_emit; four at a
// time share one; 64 of them in a row among 20,000 small ones: k_setup 288 ->
// 112 us, k_emit 411 -> 169).
template <class F>
__device__ __forceinline__ void for_tiles(const ViewTable& vt, int per, int v, const SetupRec& r, int4 box, int t,
                                          uint32_t zkey, F&& f) {
    __shared__ CtaBox s_box[kCtaBoxes];
    __shared__ int s_n;
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    const int nb = box.z < box.x ? 0 : (box.z - box.x + 1) * (box.w - box.y + 1);
    const auto walk = [&](const SetupRec& q, int vq, int x0, int y0, int bw, int i0, int step, int n, int tq, uint32_t zq) {
        const int tiles_x = vt.v[vq].tiles_x, base = vt.v[vq].tile_base;
        for (int i = i0; i < n; i += 4 * step) {
            int tiles[4];
            bool in[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int j = i + k * step, dy = j / bw, tx = x0 + j - dy * bw, ty = y0 + dy;
                tiles[k] = base + ty * tiles_x + tx;
                in[k] = j < n && tile_may_cover(q, tx, ty, vt.tile_w, vt.tile_h);
            }
            f(tiles, in, tq, zq);
        }
    };
    bool cta = nb > kWarpTiles;
    if (cta) {
        const int at = atomicAdd(&s_n, 1);
        cta = at < kCtaBoxes;
        if (cta) s_box[at] = CtaBox{r, box, v, t, zkey};
    }
    // by itself a lane takes nb / 4 rounds, beside the others; shared, a box takes
    // one of the warp's, after the others
    const int own = min(kOwnTiles, 4 * per);
    if (nb <= own) walk(r, v, box.x, box.y, box.z - box.x + 1, 0, 1, nb, t, zkey);
    unsigned wide = __ballot_sync(kFull, nb > own && !cta);
    while (wide) {
        const int src = __ffs(wide) - 1;
        wide &= wide - 1;
        SetupRec q;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            q.A[i] = __shfl_sync(kFull, r.A[i], src);
            q.B[i] = __shfl_sync(kFull, r.B[i], src);
            q.C[i] = __shfl_sync(kFull, r.C[i], src);
        }
        const int x0 = __shfl_sync(kFull, box.x, src), y0 = __shfl_sync(kFull, box.y, src);
        const int bw = __shfl_sync(kFull, box.z, src) - x0 + 1, n = __shfl_sync(kFull, nb, src);
        const int vs = __shfl_sync(kFull, v, src), ts = __shfl_sync(kFull, t, src);
        walk(q, vs, x0, y0, bw, threadIdx.x & 31, 32, n, ts, __shfl_sync(kFull, zkey, src));
    }
    __syncthreads();
    for (int i = 0; i < min(s_n, kCtaBoxes); ++i) {
        const CtaBox& c = s_box[i];
        const int bw = c.box.z - c.box.x + 1;
        walk(c.r, c.v, c.box.x, c.box.y, bw, threadIdx.x, kBinThreads, bw * (c.box.w - c.box.y + 1), c.t, c.zkey);
    }
}

// ---------------------------------------------------------------- set-up
__device__ __forceinline__ int floordiv256(int x) { return x >> 8; }   // arithmetic shift = floor

// The view of set-up record `gid` (records of view v start at rec_base).
__device__ __forceinline__ int view_of_record(const ViewTable& vt, long long gid) {
    int v = 0;
    for (int i = 1; i < vt.n; ++i)
        if (vt.v[i].rec_base <= gid) v = i;
    return v;
}

// One thread per (view, triangle), `per` of them in a warp: project, snap to
// 1/256 pixel, cull, build the oriented edge functions with the top-left fill
// rule (Eq. 1 fragments), the perspective factors k_i and the tile rectangle,
// and count the triangle in every tile whose pixel centres it may cover.
__global__ void __launch_bounds__(kBinThreads) k_setup(const __grid_constant__ ViewTable vt, long long n_records, int per,
                                                       bool split, SetupRec* __restrict__ recs, uint32_t* __restrict__ tile_count,
                                                       int4* __restrict__ tbox, uint32_t* __restrict__ zkeys) {
    const long long gid = own_record(n_records, per);
    const CounterAt at(split);
    int v = 0, t = 0;
    SetupRec r;
    int4 box = make_int4(0, 0, -1, -1);
    if (gid >= 0) {
        v = view_of_record(vt, gid);
        t = (int)(gid - vt.v[v].rec_base);
        const DevCam& cam = view_cam(vt, v);
        const int W = vt.v[v].W, H = vt.v[v].H;
        const float* p = vt.v[v].s_verts + 9LL * t;

        int X[3], Y[3];
        float w[3];
        bool ok = true;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const float px = __ldg(p + 3 * i), py = __ldg(p + 3 * i + 1), pz = __ldg(p + 3 * i + 2);
            const float xc = __fmaf_rn(cam.R[0], px, __fmaf_rn(cam.R[1], py, __fmaf_rn(cam.R[2], pz, cam.t[0])));
            const float yc = __fmaf_rn(cam.R[3], px, __fmaf_rn(cam.R[4], py, __fmaf_rn(cam.R[5], pz, cam.t[1])));
            const float zc = __fmaf_rn(cam.R[6], px, __fmaf_rn(cam.R[7], py, __fmaf_rn(cam.R[8], pz, cam.t[2])));
            ok = ok && (zc > cam.near_z);
            const float sx = __fmaf_rn(cam.fx, __fdiv_rn(xc, zc), cam.cx);
            const float sy = __fmaf_rn(cam.fy, __fdiv_rn(yc, zc), cam.cy);
            ok = ok && (fabsf(sx) <= kGuard) && (fabsf(sy) <= kGuard);
            X[i] = ok ? __float2int_rn(__fmul_rn(sx, 256.0f)) : 0;
            Y[i] = ok ? __float2int_rn(__fmul_rn(sy, 256.0f)) : 0;
            w[i] = zc;
        }
        const long long area =
            (long long)(X[1] - X[0]) * (Y[2] - Y[0]) - (long long)(X[2] - X[0]) * (Y[1] - Y[0]);
        ok = ok && (area != 0);

        uint32_t zk = 0;
        if (ok) {
            const int sg = area > 0 ? 1 : -1;
            r.bias = 0;
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const int j = (i + 1) % 3, k = (i + 2) % 3;
                const int A = sg * (Y[j] - Y[k]);
                const int B = sg * (X[k] - X[j]);
                long long Cc = (long long)sg * ((long long)X[j] * Y[k] - (long long)X[k] * Y[j]);
                const bool owns = A > 0 || (A == 0 && B > 0);
                if (!owns) {
                    Cc -= 1;
                    r.bias |= 1u << i;
                }
                r.A[i] = A;
                r.B[i] = B;
                r.C[i] = Cc;
            }
            const int amax = max(max(max(abs(r.A[0]), abs(r.A[1])), abs(r.A[2])), max(max(abs(r.B[0]), abs(r.B[1])), abs(r.B[2])));
            const int cx = (X[0] >> kCellBits) + 1, cy = (Y[0] >> kCellBits) + 1;
            if (amax <= kSmallEdge && (unsigned)cx < 256u && (unsigned)cy < 256u)
                r.bias |= kSmallTri | ((uint32_t)cx << 4) | ((uint32_t)cy << 12);
            const float fa = __ll2float_rn(area > 0 ? area : -area);
#pragma unroll
            for (int i = 0; i < 3; ++i) r.k[i] = __fdiv_rn(__fdiv_rn(1.0f, w[i]), fa);

            // pixel centres 256 px + 128 inside [min, max] of the snapped vertices
            const int xmin = min(X[0], min(X[1], X[2])), xmax = max(X[0], max(X[1], X[2]));
            const int ymin = min(Y[0], min(Y[1], Y[2])), ymax = max(Y[0], max(Y[1], Y[2]));
            const int px0 = max(floordiv256(xmin - 128 + 255), 0), px1 = min(floordiv256(xmax - 128), W - 1);
            const int py0 = max(floordiv256(ymin - 128 + 255), 0), py1 = min(floordiv256(ymax - 128), H - 1);
            if (px0 <= px1 && py0 <= py1)
                box = make_int4(px0 / vt.tile_w, py0 / vt.tile_h, px1 / vt.tile_w, py1 / vt.tile_h);
            zk = __float_as_uint(fminf(w[0], fminf(w[1], w[2])));
        } else {
            r = SetupRec{};
            r.C[0] = r.C[1] = r.C[2] = -1;   // covers nothing
        }
        int4* dst = reinterpret_cast<int4*>(recs + gid);
        const int4* src = reinterpret_cast<const int4*>(&r);
        dst[0] = src[0];
        dst[1] = src[1];
        dst[2] = src[2];
        dst[3] = src[3];
        tbox[gid] = box;
        zkeys[gid] = zk;
    }
    for_tiles(vt, per, v, r, box, t, 0u, [&](const int (&tiles)[4], const bool (&in)[4], int, uint32_t) {
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (in[k]) atomicAdd(tile_count + tiles[k] * at.step + at.first, 1u);
    });
}

long long view_records(const ViewTable& vt) {
    return vt.n > 0 ? vt.v[vt.n - 1].rec_base + vt.v[vt.n - 1].s_T : 0;
}

void set_view_soups(ViewTable& vt, const SoupDev* const* soups) {
    long long rb = 0;
    for (int v = 0; v < vt.n; ++v) {
        const SoupDev& s = *soups[v];
        ViewDesc& d = vt.v[v];
        d.s_verts = s.verts;
        d.s_act = s.act;
        d.s_act_a = s.act_a;
        d.s_T = s.T;
        d.rec_base = rb;
        rb += s.T;
    }
}

void set_view_soups(ViewTable& vt, const SoupDev& s) {
    const SoupDev* one[DS_MAX_VIEWS];
    for (int v = 0; v < vt.n; ++v) one[v] = &s;
    set_view_soups(vt, one);
}

cudaError_t launch_setup(const ViewTable& vt, int n_tiles, SetupRec* recs, uint32_t* tile_count, int4* tbox,
                         uint32_t* zkeys, cudaStream_t st) {
    const long long n = view_records(vt);
    cudaError_t e = cudaMemsetAsync(tile_count, 0, sizeof(uint32_t) * counter_words(n_tiles), st);
    if (e != cudaSuccess || n <= 0) return e;
    const int per = records_per_warp(n), cta = per * kBinThreads / 32;
    k_setup<<<(unsigned)((n + cta - 1) / cta), kBinThreads, 0, st>>>(vt, n, per, split_counters(n_tiles), recs, tile_count, tbox,
                                                                    zkeys);
    note_launches(1);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- tile offsets
// Sum of one block's kScanBlock tile counts (1024 threads x 4).
__global__ void __launch_bounds__(1024) k_tile_sums(const uint32_t* __restrict__ count, int n,
                                                    uint32_t* __restrict__ block_sum, uint32_t* __restrict__ total) {
    __shared__ uint32_t wsum[32];
    const int tid = threadIdx.x, base = blockIdx.x * kScanBlock + 4 * tid;
    uint32_t s = 0;
    if (blockIdx.x == 0 && tid == 0) total[1] = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) s += base + k < n ? count[base + k] : 0u;
    s = __reduce_add_sync(kFull, s);
    if ((tid & 31) == 0) wsum[tid >> 5] = s;
    __syncthreads();
    if (tid < 32) {
        s = __reduce_add_sync(kFull, wsum[tid]);
        if (tid == 0) block_sum[blockIdx.x] = s;
    }
}

// Exclusive scan of the tile counts: every tile's range in the lists (cut at
// the capacity `cap`) and its cursor for k_emit, the number of pairs total[0],
// the chunks of the lists above kBlockList entries and their number total[1],
// and the tile kernels' work counters set to zero.  A thread has four tiles,
// or the four counters of one (kSplit).  Block b adds up the sums of the
// blocks before it itself (at most 4,096 for the largest call).
template <bool kSplit>
__global__ void __launch_bounds__(1024) k_tile_offsets(const uint32_t* __restrict__ count, int n, uint32_t cap,
                                                       const uint32_t* __restrict__ block_sum, uint2* __restrict__ ranges,
                                                       uint32_t* __restrict__ cursor, uint32_t* __restrict__ total,
                                                       uint2* __restrict__ chunks, int* __restrict__ counters,
                                                       int n_counters) {
    __shared__ uint32_t wsum[32], wpre[32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int base = kSplit ? tid : blockIdx.x * kScanBlock + 4 * tid;
    constexpr int kTiles = kSplit ? 1 : 4;   // tiles of a thread
    if (gridDim.x == 1 && tid == 0) total[1] = 0;   // else k_tile_sums has cleared it
    uint32_t before = 0;
    for (int b = tid; b < (int)blockIdx.x; b += 1024) before += block_sum[b];
    before = __reduce_add_sync(kFull, before);
    const auto slot = [&](int k) { return kSplit ? (base * kSplitWays + k) * kSplitWords : base + k; };
    uint32_t x[4], sum = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        x[k] = base + (kSplit ? 0 : k) < n ? count[slot(k)] : 0u;
        sum += x[k];
    }
    uint32_t inc = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t o = __shfl_up_sync(kFull, inc, d);
        if (lane >= d) inc += o;
    }
    if (lane == 31) wsum[warp] = inc;
    if (lane == 0) wpre[warp] = before;
    __syncthreads();
    uint32_t off = inc - sum;
    for (int w = 0; w < 32; ++w) off += wpre[w] + (w < warp ? wsum[w] : 0u);
#pragma unroll
    for (int t = 0; t < kTiles; ++t) {
        const uint32_t first = off;
        if (base + t >= n) break;
#pragma unroll
        for (int k = t * (4 / kTiles); k < (t + 1) * (4 / kTiles); ++k) {
            cursor[slot(k)] = off;
            off += x[k];
        }
        const uint32_t lo = min(first, cap), hi = min(off, cap);
        ranges[base + t] = make_uint2(lo, hi);
        if (hi - lo > kBlockList) {
            const uint32_t m = (hi - lo + kBlockList - 1) / kBlockList, at = atomicAdd(total + 1, m);
            for (uint32_t c = 0; c < m; ++c) chunks[at + c] = make_uint2((uint32_t)(base + t), c);
        }
        if (base + t == n - 1) *total = off;
    }
    if (blockIdx.x == 0 && tid < n_counters) counters[tid] = 0;
}

cudaError_t launch_tile_offsets(const uint32_t* count, int n_tiles, uint32_t cap, uint32_t* block_sum, uint2* ranges,
                                uint32_t* cursor, uint32_t* total, uint2* chunks, int* counters, int n_counters,
                                cudaStream_t st) {
    const int nblk = (n_tiles + kScanBlock - 1) / kScanBlock;
    if (nblk > 1) {
        k_tile_sums<<<nblk, 1024, 0, st>>>(count, n_tiles, block_sum, total);
        note_launches(1);
    }
    const auto kernel = split_counters(n_tiles) ? k_tile_offsets<true> : k_tile_offsets<false>;
    kernel<<<nblk, 1024, 0, st>>>(count, n_tiles, cap, block_sum, ranges, cursor, total, chunks, counters, n_counters);
    note_launches(1);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- emission
// Each pair to the next place of its tile; the key holds the depth bits (none
// is written without).  Pairs beyond the capacity are dropped and reported.
__global__ void __launch_bounds__(kBinThreads) k_emit(const __grid_constant__ ViewTable vt, long long n_records, int per, bool split,
                                                      const SetupRec* __restrict__ recs, const int4* __restrict__ tbox,
                                                      const uint32_t* __restrict__ zkeys, int DB,
                                                      uint32_t* __restrict__ cursor, uint32_t* __restrict__ keys,
                                                      uint32_t* __restrict__ vals, uint32_t cap,
                                                      int* __restrict__ status) {
    const long long gid = own_record(n_records, per);
    const CounterAt at(split);
    int4 box = make_int4(0, 0, -1, -1);
    if (gid >= 0) box = tbox[gid];
    int v = 0, t = 0;
    uint32_t zk = 0;
    SetupRec r;
    if (box.z >= box.x) {
        v = view_of_record(vt, gid);
        t = (int)(gid - vt.v[v].rec_base);
        r = load_rec(recs + gid);
        zk = DB > 0 ? (zkeys[gid] & 0x7fffffffu) >> (31 - DB) : 0u;
    }
    bool over = false;
    for_tiles(vt, per, v, r, box, t, zk, [&](const int (&tiles)[4], const bool (&in)[4], int tri, uint32_t z) {
        uint32_t o[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) o[k] = in[k] ? atomicAdd(cursor + tiles[k] * at.step + at.first, 1u) : 0u;
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (in[k] && o[k] < cap) {
                vals[o[k]] = (uint32_t)tri;
                if (DB > 0) keys[o[k]] = z;
            } else if (in[k]) {
                over = true;
            }
    });
    if (over && status) atomicOr(status, 1);
}

cudaError_t launch_emit(const ViewTable& vt, int n_tiles, const SetupRec* recs, const int4* tbox, const uint32_t* zkeys, int DB,
                        uint32_t* cursor, uint32_t* keys, uint32_t* vals, uint32_t cap, int* status, cudaStream_t st) {
    const long long n = view_records(vt);
    if (n <= 0) return cudaSuccess;
    const int per = records_per_warp(n), cta = per * kBinThreads / 32;
    k_emit<<<(unsigned)((n + cta - 1) / cta), kBinThreads, 0, st>>>(vt, n, per, split_counters(n_tiles), recs, tbox, zkeys, DB,
                                                                   cursor, keys, vals, cap, status);
    note_launches(1);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- depth order
// Sort times below in us: (a) 100,000 triangles in eight 1080p views, (b)
// 2,000 and (c) 20,000 in a 64 x 64 view (16 lists), (d) 200,000 there with
// lists of 13,000, (e) 1,000,000 there with lists of 45,000, 16 depth bits.
namespace {
constexpr int kSortWarps = 8;       // most tiles per CTA of k_tile_sort
constexpr int kWarpList = 128;      // lists up to this length: one warp, in registers (64: a 76 -> 109, b 24 -> 11)
constexpr int kWarpTriangles = 256; // the same without depth keys
constexpr int kSortThreads = 256;   // 512: a 76 -> 99, d 51 -> 45
}  // namespace

// Ranks of E entries per lane among the warp's n by counting the smaller ones
// ((key, triangle) pairs are distinct), written back in order.
template <int E>
__device__ __forceinline__ void sort_warp(uint32_t* keys, uint32_t* vals, uint32_t lo, int n, int lane) {
    uint32_t k[E], v[E];
    int rank[E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const bool in = lane + 32 * e < n;
        k[e] = in ? keys[lo + lane + 32 * e] : 0u;
        v[e] = in ? vals[lo + lane + 32 * e] : 0u;
        rank[e] = 0;
    }
#pragma unroll
    for (int f = 0; f < E; ++f)
        for (int j = 0; j < min(32, n - 32 * f); ++j) {
            const uint32_t kj = __shfl_sync(kFull, k[f], j), vj = __shfl_sync(kFull, v[f], j);
#pragma unroll
            for (int e = 0; e < E; ++e) rank[e] += kj < k[e] || (kj == k[e] && vj < v[e]) ? 1 : 0;
        }
    __syncwarp();
#pragma unroll
    for (int e = 0; e < E; ++e)
        if (lane + 32 * e < n) {
            keys[lo + rank[e]] = k[e];
            vals[lo + rank[e]] = v[e];
        }
}

// Without depth keys: a bitonic network over the triangles in the warp's 32 E
// registers (the 1080p batch's 1.6 M pairs: counting as above 49 us, the network
// 39, and up to 256 entries in a warp 30).
template <int E>
__device__ __forceinline__ void sort_warp_triangles(uint32_t* vals, uint32_t lo, int n, int lane) {
    uint32_t v[E];
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = lane + 32 * e < n ? vals[lo + lane + 32 * e] : 0xffffffffu;
#pragma unroll
    for (int k = 2; k <= 32 * E; k <<= 1)
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1)
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const bool up = ((lane + 32 * e) & k) == 0;
                if (j < 32) {   // the partner is the same register of another lane
                    const uint32_t o = __shfl_xor_sync(kFull, v[e], j);
                    v[e] = ((lane & j) == 0) == up ? min(v[e], o) : max(v[e], o);
                } else if (!(e & (j >> 5))) {   // another register of this lane
                    const int p = e | (j >> 5);
                    const uint32_t a = min(v[e], v[p]), b = max(v[e], v[p]);
                    v[e] = up ? a : b;
                    v[p] = up ? b : a;
                }
            }
#pragma unroll
    for (int e = 0; e < E; ++e)
        if (lane + 32 * e < n) vals[lo + lane + 32 * e] = v[e];
}

template <bool kKeys>
__device__ __forceinline__ void sort_short(uint32_t* keys, uint32_t* vals, uint32_t lo, int n, int lane) {
    if constexpr (kKeys) {
        if (n > 64) sort_warp<4>(keys, vals, lo, n, lane);
        else if (n > 32) sort_warp<2>(keys, vals, lo, n, lane);
        else if (n > 1) sort_warp<1>(keys, vals, lo, n, lane);
    } else {
        if (n > 128) sort_warp_triangles<8>(vals, lo, n, lane);
        else if (n > 64) sort_warp_triangles<4>(vals, lo, n, lane);
        else if (n > 32) sort_warp_triangles<2>(vals, lo, n, lane);
        else if (n > 1) sort_warp_triangles<1>(vals, lo, n, lane);
    }
}

// n <= kBlockList entries (depth key, triangle) from k, v in order into ko, vo
// (which may be k and v): a bitonic network in shared memory.
__device__ __forceinline__ void sort_block(unsigned long long* s_kv, const uint32_t* k, const uint32_t* v, uint32_t* ko,
                                           uint32_t* vo, int n, bool keys) {
    const int tid = threadIdx.x;
    int m = kSortThreads;
    while (m < n) m <<= 1;
    for (int i = tid; i < m; i += kSortThreads)
        s_kv[i] = i < n ? ((unsigned long long)(keys ? k[i] : 0u) << 32) | v[i] : ~0ull;
    for (int w = 2; w <= m; w <<= 1)
        for (int j = w >> 1; j > 0; j >>= 1) {
            __syncthreads();
            for (int p = tid; p < m / 2; p += kSortThreads) {
                const int i = 2 * p - (p & (j - 1));   // the pair (i, i + j)
                const unsigned long long a = s_kv[i], b = s_kv[i + j];
                if ((a > b) == ((i & w) == 0)) {
                    s_kv[i] = b;
                    s_kv[i + j] = a;
                }
            }
        }
    __syncthreads();
    for (int i = tid; i < n; i += kSortThreads) {
        if (keys) ko[i] = (uint32_t)(s_kv[i] >> 32);
        vo[i] = (uint32_t)s_kv[i];
    }
    __syncthreads();
}

// Every tile's list by (depth key, triangle).  Most lists are short (a few
// dozen triangles): one warp each.  The CTA then takes its tiles with longer
// lists one after the other, and of the lists above kBlockList its
// share of the chunks, which go to (k1, v1) for k_list_merge.  A CTA's `per`
// tiles are gridDim.x apart, since long lists come in neighbouring tiles.
// Bound by the latency of the network's stages (c) or by shared memory (e).
// With eight tiles to every CTA and lists above 2,048 entries in radix passes
// of one CTA: b 49, c 137, d 582, e 2,029 us; now 24, 51, 51 and 132 (a global
// radix sort of all pairs: 64, 80, 109 and 117, and a 171 against 76).
template <bool kKeys>   // there are depth keys
__global__ void __launch_bounds__(kSortThreads) k_tile_sort(const uint2* __restrict__ ranges, int n_tiles, int per,
                                                            const uint32_t* __restrict__ n_chunks,
                                                            const uint2* __restrict__ chunks, uint32_t* __restrict__ k0,
                                                            uint32_t* __restrict__ v0, uint32_t* __restrict__ k1,
                                                            uint32_t* __restrict__ v1) {
    __shared__ unsigned long long s_kv[kBlockList];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    bool lng = false;
    constexpr int kShort = kKeys ? kWarpList : kWarpTriangles;
    const int tile = blockIdx.x + warp * gridDim.x;
    if (warp < per && tile < n_tiles) {
        const uint2 rg = ranges[tile];
        const int n = (int)(rg.y - rg.x);
        if (n > kShort) lng = true;
        else sort_short<kKeys>(k0, v0, rg.x, n, lane);
    }
    const bool any = __syncthreads_or(lng);
    for (int q = 0; any && q < per; ++q) {
        if ((int)(blockIdx.x + q * gridDim.x) >= n_tiles) break;
        const uint2 rg = ranges[blockIdx.x + q * gridDim.x];
        const int n = (int)(rg.y - rg.x);
        if (n > kShort && n <= kBlockList) sort_block(s_kv, k0 + rg.x, v0 + rg.x, k0 + rg.x, v0 + rg.x, n, kKeys);
    }
    const uint32_t nc = n_chunks ? *n_chunks : 0u;
    for (uint32_t i = blockIdx.x; i < nc; i += gridDim.x) {
        const uint2 ch = chunks[i], rg = ranges[ch.x];
        const uint32_t lo = rg.x + ch.y * kBlockList;
        sort_block(s_kv, k0 + lo, v0 + lo, k1 + lo, v1 + lo, (int)min((uint32_t)kBlockList, rg.y - lo), kKeys);
    }
}

// The sorted chunks (k1, v1) of the long lists into one order (k0, v0): an
// entry's place is its place in its chunk plus the number of smaller entries
// of every other chunk of the list, found by bisection with that chunk in
// shared memory.
__global__ void __launch_bounds__(kSortThreads) k_list_merge(const uint2* __restrict__ ranges, int DB,
                                                             const uint32_t* __restrict__ n_chunks,
                                                             const uint2* __restrict__ chunks,
                                                             const uint32_t* __restrict__ k1,
                                                             const uint32_t* __restrict__ v1, uint32_t* __restrict__ k0,
                                                             uint32_t* __restrict__ v0) {
    __shared__ unsigned long long s_kv[kBlockList];
    constexpr int E = kBlockList / kSortThreads;
    const int tid = threadIdx.x;
    const uint32_t nc = *n_chunks;
    const auto entry = [&](uint32_t i) { return ((unsigned long long)(DB > 0 ? k1[i] : 0u) << 32) | v1[i]; };
    for (uint32_t item = blockIdx.x; item < nc; item += gridDim.x) {
        const uint2 ch = chunks[item], rg = ranges[ch.x];
        const uint32_t m = (rg.y - rg.x + kBlockList - 1) / kBlockList, lo = rg.x + ch.y * kBlockList;
        unsigned long long x[E];
        uint32_t rank[E];
#pragma unroll
        for (int e = 0; e < E; ++e) {
            rank[e] = tid + e * kSortThreads;
            x[e] = lo + rank[e] < rg.y ? entry(lo + rank[e]) : ~0ull;
        }
        for (uint32_t o = 0; o < m; ++o) {
            if (o == ch.y) continue;
            const uint32_t from = rg.x + o * kBlockList;
            __syncthreads();
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const uint32_t i = tid + e * kSortThreads;
                s_kv[i] = from + i < rg.y ? entry(from + i) : ~0ull;
            }
            __syncthreads();
            uint32_t pos[E] = {};
#pragma unroll
            for (int step = kBlockList / 2; step > 0; step >>= 1)
#pragma unroll
                for (int e = 0; e < E; ++e)
                    if (s_kv[pos[e] + step - 1] < x[e]) pos[e] += step;
#pragma unroll
            for (int e = 0; e < E; ++e) rank[e] += pos[e] + (s_kv[pos[e]] < x[e] ? 1u : 0u);
        }
#pragma unroll
        for (int e = 0; e < E; ++e)
            if (lo + tid + e * kSortThreads < rg.y) {
                if (DB > 0) k0[rg.x + rank[e]] = (uint32_t)(x[e] >> 32);
                v0[rg.x + rank[e]] = (uint32_t)x[e];
            }
    }
}

bool long_lists(const ViewTable& vt) {
    for (int v = 0; v < vt.n; ++v)
        if (vt.v[v].s_T > kBlockList) return true;
    return false;
}

// CTAs for the chunks of the long lists: as many as full chunks fit the
// buffers, at most what the device holds at once.
static int chunk_grid(uint32_t cap) { return persistent_grid((int)(cap / kBlockList) + 1, 2048 / kSortThreads); }

cudaError_t launch_tile_sort(const ViewTable& vt, const uint2* ranges, int n_tiles, int DB, const uint32_t* n_chunks,
                             const uint2* chunks, uint32_t cap, uint32_t* k0, uint32_t* v0, uint32_t* k1, uint32_t* v1,
                             cudaStream_t st) {
    // Few tiles: fewer of them per CTA, down to one, so that their lists are
    // sorted side by side (eight always: b 24 -> 50, 256 tiles of 740 entries
    // 28 -> 53).  Up to four CTAs per SM; two or eight measure alike.
    const int ctas = persistent_grid(1 << 30, 4);
    int per = 1;
    while (per < kSortWarps && n_tiles > per * ctas) per *= 2;
    const bool lng = long_lists(vt);
    const int grid = std::max((n_tiles + per - 1) / per, lng ? chunk_grid(cap) : 1);
    const auto kernel = DB > 0 ? k_tile_sort<true> : k_tile_sort<false>;
    kernel<<<grid, kSortThreads, 0, st>>>(ranges, n_tiles, per, lng ? n_chunks : nullptr, chunks, k0, v0, k1, v1);
    note_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_list_merge(const uint2* ranges, int DB, const uint32_t* n_chunks, const uint2* chunks, uint32_t cap,
                              uint32_t* k0, uint32_t* v0, const uint32_t* k1, const uint32_t* v1, cudaStream_t st) {
    k_list_merge<<<chunk_grid(cap), kSortThreads, 0, st>>>(ranges, DB, n_chunks, chunks, k1, v1, k0, v0);
    note_launches(1);
    return cudaGetLastError();
}

}  // namespace ds
