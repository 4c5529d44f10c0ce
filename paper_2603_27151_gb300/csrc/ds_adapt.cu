// ds_adapt.cu -- adaptive control of primitives (Sec. 3.4 "Adaptive control
// of primitives"): the GPU measurements that drive it and the rebuild of the
// soup after a round of edge splits and prunes.
//  - k_coverage: pixel-samples won per triangle, from the G-buffers' triangle
//    ids; lanes holding the same id are merged with one match-any vote and
//    a single atomic per id and warp.
//  - k_edge_ratios: per triangle, each edge's largest projected length over
//    the views (those where the triangle lies in front of the near plane and
//    its projected bounding box meets the image), relative to the image
//    height; FP32 in the oracle's order, so that the split decision is the
//    same on both sides.
//  - the plan (host C++): split the longest edge above the threshold, then
//    remove the lowest-coverage triangles until the budget holds; or, for
//    the random initialisation of the supplementary material, remove the
//    uncovered triangles and split the longest edges up to a target count.
//  - k_rebuild_verts / k_rebuild_level: the new soup: copies, or the two
//    children of a split edge (midpoint in FP32), each child's grid sampled
//    from the parent's grid at the child's vertices mapped into the parent.
#include <algorithm>
#include <type_traits>
#include <numeric>
#include <vector>

#include "ds_internal.h"

namespace ds {

namespace {

struct CoverView {
    const int4* gbuf;   // [S][H][W] texels; .x = triangle id
    long long n;        // S * H * W
};
struct CoverTable {
    int n_views, T;
    CoverView v[DS_MAX_VIEWS];
};

__global__ void __launch_bounds__(256) k_coverage(const __grid_constant__ CoverTable ct, int* __restrict__ counts) {
    const CoverView& V = ct.v[blockIdx.y];
    for (long long base = (long long)blockIdx.x * blockDim.x; base < V.n; base += (long long)gridDim.x * blockDim.x) {
        const long long k = base + threadIdx.x;
        int id = -1;
        if (k < V.n) id = __ldg(&V.gbuf[k].x);
        if (id >= ct.T) id = -1;
        const unsigned same = __match_any_sync(0xffffffffu, id);
        const int lead = __ffs(same) - 1;
        if (id >= 0 && (int)(threadIdx.x & 31) == lead) atomicAdd(counts + id, __popc(same));
    }
}

struct RatioCam {
    float fx, fy, cx, cy, R[9], t[3], near_z;
    int W, H;
};
struct RatioTable {
    int n_views;
    RatioCam c[DS_MAX_VIEWS];
};

__global__ void __launch_bounds__(256) k_edge_ratios(const __grid_constant__ RatioTable rt, const float* __restrict__ verts,
                                                     int T, float* __restrict__ out) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= T) return;
    float p[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) p[k] = __ldg(verts + 9 * (size_t)t + k);
    float best[3] = {0.f, 0.f, 0.f};
    for (int v = 0; v < rt.n_views; ++v) {
        const RatioCam& c = rt.c[v];
        float sx[3], sy[3];
        bool ok = true;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const float* q = p + 3 * i;
            const float xc = __fmaf_rn(c.R[0], q[0], __fmaf_rn(c.R[1], q[1], __fmaf_rn(c.R[2], q[2], c.t[0])));
            const float yc = __fmaf_rn(c.R[3], q[0], __fmaf_rn(c.R[4], q[1], __fmaf_rn(c.R[5], q[2], c.t[1])));
            const float zc = __fmaf_rn(c.R[6], q[0], __fmaf_rn(c.R[7], q[1], __fmaf_rn(c.R[8], q[2], c.t[2])));
            ok = ok && (zc > c.near_z);
            sx[i] = __fmaf_rn(c.fx, __fdiv_rn(xc, zc), c.cx);
            sy[i] = __fmaf_rn(c.fy, __fdiv_rn(yc, zc), c.cy);
        }
        if (!ok) continue;
        const float x0 = fminf(sx[0], fminf(sx[1], sx[2])), x1 = fmaxf(sx[0], fmaxf(sx[1], sx[2]));
        const float y0 = fminf(sy[0], fminf(sy[1], sy[2])), y1 = fmaxf(sy[0], fmaxf(sy[1], sy[2]));
        if (x1 < 0.0f || x0 > (float)c.W || y1 < 0.0f || y0 > (float)c.H) continue;
#pragma unroll
        for (int e = 0; e < 3; ++e) {
            const int a = e, b = (e + 1) % 3;
            const float dx = __fsub_rn(sx[b], sx[a]), dy = __fsub_rn(sy[b], sy[a]);
            const float r = __fdiv_rn(__fsqrt_rn(__fmaf_rn(dx, dx, __fmul_rn(dy, dy))), (float)c.H);
            best[e] = r > best[e] ? r : best[e];
        }
    }
#pragma unroll
    for (int e = 0; e < 3; ++e) out[3 * (size_t)t + e] = best[e];
}

// The child's corners in the parent's barycentrics, doubled (integers).
__device__ __forceinline__ void child_corners(int op, int P[3][3]) {
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int q = 0; q < 3; ++q) P[i][q] = 2 * (i == q);
    if (op == 0) return;
    const int e = (op - 1) >> 1, c = (op - 1) & 1;
    const int a = e, b = (e + 1) % 3, o = (e + 2) % 3;
    int Q[3][3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const int pa = q == a ? 2 : 0, pb = q == b ? 2 : 0, pm = (q == a || q == b) ? 1 : 0, po = q == o ? 2 : 0;
        Q[0][q] = c == 0 ? pa : pm;
        Q[1][q] = c == 0 ? pm : pb;
        Q[2][q] = po;
    }
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int q = 0; q < 3; ++q) P[i][q] = Q[i][q];
}

// Where a texel of a child comes from: one parent texel (k, all ones above
// bit 10), or the decode's interpolation of the three in k's ten-bit fields.
struct RebuildTap {
    unsigned k;
    float wa, wb;
};
constexpr unsigned kOneTexel = 0xfffffc00u;
constexpr int kRebuildItems = 2;   // items in flight per thread

// The source of vertex v of the children with split code op > 0.
__device__ __forceinline__ RebuildTap rebuild_tap(int N, int op, int v) {
    int i, j;
    texel_ij(N, v, i, j);
    int P[3][3];
    child_corners(op, P);
    const int X = (N - i - j) * P[0][1] + i * P[1][1] + j * P[2][1];
    const int Y = (N - i - j) * P[0][2] + i * P[1][2] + j * P[2][2];
    if ((X & 1) == 0 && (Y & 1) == 0)
        return RebuildTap{kOneTexel | (unsigned)texel_index(N, X >> 1, Y >> 1), 0.f, 0.f};
    const Cell cl = find_cell(N, __fdiv_rn((float)X, (float)(2 * N)), __fdiv_rn((float)Y, (float)(2 * N)));
    return RebuildTap{(unsigned)(cl.k0 | (cl.k1 << 10) | (cl.k2 << 20)), cl.wa, cl.wb};
}

__device__ __forceinline__ float rebuild_mix(float a, float b, float d, const RebuildTap& tp) {
    return interp(a, b, d, tp.wa, tp.wb);
}
__device__ __forceinline__ float4 rebuild_mix(float4 a, float4 b, float4 d, const RebuildTap& tp) {
    return make_float4(interp(a.x, b.x, d.x, tp.wa, tp.wb), interp(a.y, b.y, d.y, tp.wa, tp.wb),
                       interp(a.z, b.z, d.z, tp.wa, tp.wb), interp(a.w, b.w, d.w, tp.wa, tp.wb));
}

// One level of few triangles, or of channels that the table below does not
// suit: a thread per texel, which finds the source itself and goes through the
// channels.  Bound by latency (level 5 of 50 triangles: 34 us for the whole
// call, 43 with a table in every CTA).
template <bool kVec>
__global__ void __launch_bounds__(256) k_rebuild_texels(const float* __restrict__ gin, int N, int C,
                                                        const int* __restrict__ plan, int n_out,
                                                        float* __restrict__ gout) {
    using Item = std::conditional_t<kVec, float4, float>;
    const int V = (N + 1) * (N + 2) / 2, per = kVec ? C / 4 : C;
    const long long n = (long long)n_out * V, step = (long long)gridDim.x * blockDim.x;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += step) {
        const int k = (int)(q / V), v = (int)(q - (long long)k * V);
        const int code = __ldg(plan + k), op = code & 7;
        const RebuildTap tp = op > 0 ? rebuild_tap(N, op, v) : RebuildTap{kOneTexel | (unsigned)v, 0.f, 0.f};
        const Item* g = reinterpret_cast<const Item*>(gin) + (size_t)(code >> 3) * (unsigned)(V * per);
        Item* d = reinterpret_cast<Item*>(gout) + (size_t)q * per;
        const Item* a = g + (tp.k & 1023u) * per;
        if (tp.k < kOneTexel) {
            const Item *b = g + ((tp.k >> 10) & 1023u) * per, *e = g + ((tp.k >> 20) & 1023u) * per;
            for (int c = 0; c < per; ++c) d[c] = rebuild_mix(__ldg(a + c), __ldg(b + c), __ldg(e + c), tp);
        } else {
            for (int c = 0; c < per; ++c) d[c] = __ldg(a + c);
        }
    }
}

// One level.  The source of a child's texel depends on its code and vertex
// only: every CTA tabulates the six splits first (shared memory), then the
// items, V texels of C / 4 channel groups per triangle (scalar channels when
// C or the alignment does not allow 16 bytes), stream through it with
// consecutive lanes on consecutive addresses.  Bound by the latency of the
// gathers and by HBM: level 5 of 20,000 triangles (718 MB, 107 us at the copy
// rate) 375 -> 131 us against one thread per texel with an index search and
// scalar channels.  Two items in flight per thread at five CTAs per SM; one:
// 141 us, three: 268 us, four at two CTAs: 255 us.
template <bool kVec>
__global__ void __launch_bounds__(256, 5) k_rebuild_level(const float* __restrict__ gin, int N, int C,
                                                       const int* __restrict__ plan, int n_out,
                                                       float* __restrict__ gout) {
    extern __shared__ RebuildTap taps[];   // [6][V]
    const int V = (N + 1) * (N + 2) / 2;
    for (int q = threadIdx.x; q < 6 * V; q += blockDim.x) {
        const int op = q / V + 1, v = q - (op - 1) * V;
        taps[q] = rebuild_tap(N, op, v);
    }
    __syncthreads();
    // items: channel group c of texel r of output triangle k; a thread keeps
    // its channel group (the grid's threads are a multiple of `per`)
    const int per = kVec ? C / 4 : C;
    const unsigned id = blockIdx.x * blockDim.x + threadIdx.x, threads = gridDim.x * blockDim.x;
    const unsigned c = id % per, step = threads / per;   // in texels
    const int dk = (int)(step / V), dr = (int)(step - (unsigned)dk * V);
    int k = (int)(id / per / V), r = (int)(id / per - (unsigned)k * V);
    using Item = std::conditional_t<kVec, float4, float>;
    const Item* in = reinterpret_cast<const Item*>(gin) + c;
    Item* out = reinterpret_cast<Item*>(gout) + c;
    while (k < n_out) {
        Item a[kRebuildItems], b[kRebuildItems], d[kRebuildItems];
        RebuildTap tp[kRebuildItems];
        size_t dst[kRebuildItems];
        int n = 0;
#pragma unroll
        for (int u = 0; u < kRebuildItems; ++u) {
            if (k < n_out) {
                n = u + 1;
                const int code = __ldg(plan + k), op = code & 7;
                tp[u] = op > 0 ? taps[(op - 1) * V + r] : RebuildTap{kOneTexel | (unsigned)r, 0.f, 0.f};
                const Item* g = in + (size_t)(code >> 3) * (unsigned)(V * per);
                a[u] = __ldg(g + (tp[u].k & 1023u) * per);
                if (tp[u].k < kOneTexel) {
                    b[u] = __ldg(g + ((tp[u].k >> 10) & 1023u) * per);
                    d[u] = __ldg(g + ((tp[u].k >> 20) & 1023u) * per);
                }
                dst[u] = ((size_t)k * V + r) * per;
                k += dk;
                r += dr;
                if (r >= V) {
                    r -= V;
                    ++k;
                }
            }
        }
#pragma unroll
        for (int u = 0; u < kRebuildItems; ++u) {
            if (u >= n) break;
            if (tp[u].k < kOneTexel) a[u] = rebuild_mix(a[u], b[u], d[u], tp[u]);
            __stcs(out + dst[u], a[u]);
        }
    }
}

__global__ void __launch_bounds__(256) k_rebuild_verts(const float* __restrict__ vin, const int* __restrict__ plan,
                                                       int n_out, float* __restrict__ vout) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n_out) return;
    const int code = __ldg(plan + k), parent = code >> 3, op = code & 7;
    const float* s = vin + 9 * (size_t)parent;
    float* d = vout + 9 * (size_t)k;
    if (op == 0) {
#pragma unroll
        for (int q = 0; q < 9; ++q) d[q] = __ldg(s + q);
        return;
    }
    const int e = (op - 1) >> 1, c = (op - 1) & 1;
    const int a = e, b = (e + 1) % 3, o = (e + 2) % 3;
    float m[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) m[q] = __fmul_rn(__fadd_rn(__ldg(s + 3 * a + q), __ldg(s + 3 * b + q)), 0.5f);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        d[q] = c == 0 ? __ldg(s + 3 * a + q) : m[q];
        d[3 + q] = c == 0 ? m[q] : __ldg(s + 3 * b + q);
        d[6 + q] = __ldg(s + 3 * o + q);
    }
}

}  // namespace

cudaError_t launch_coverage(const int4* const* gbufs, const long long* n, int n_views, int T, int* counts,
                            cudaStream_t st) {
    CoverTable ct;
    ct.n_views = n_views;
    ct.T = T;
    long long most = 0;
    for (int v = 0; v < n_views; ++v) {
        ct.v[v].gbuf = gbufs[v];
        ct.v[v].n = n[v];
        most = std::max(most, n[v]);
    }
    if (most == 0) return cudaSuccess;
    const int gx = (int)std::min<long long>((most + 255) / 256, 2048);
    k_coverage<<<dim3(gx, n_views), 256, 0, st>>>(ct, counts);
    note_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_edge_ratios(const float* verts, int T, const ds_camera* cams, int n_views, float* out,
                               cudaStream_t st) {
    RatioTable rt;
    rt.n_views = n_views;
    for (int v = 0; v < n_views; ++v) {
        const ds_camera& c = cams[v];
        RatioCam& r = rt.c[v];
        r.fx = c.fx; r.fy = c.fy; r.cx = c.cx; r.cy = c.cy;
        for (int k = 0; k < 9; ++k) r.R[k] = c.R[k];
        for (int k = 0; k < 3; ++k) r.t[k] = c.t[k];
        r.near_z = c.near_z;
        r.W = c.width;
        r.H = c.height;
    }
    k_edge_ratios<<<(T + 255) / 256, 256, 0, st>>>(rt, verts, T, out);
    note_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_rebuild(const float* verts, const float* tex, int T, const int* grid_ns, int n_levels, int C,
                           const int* plan_dev, int n_out, float* verts_out, float* tex_out, cudaStream_t st) {
    if (n_out == 0) return cudaSuccess;
    k_rebuild_verts<<<(n_out + 255) / 256, 256, 0, st>>>(verts, plan_dev, n_out, verts_out);
    note_launches(1);
    size_t off_in = 0, off_out = 0;
    for (int l = 0; l < n_levels; ++l) {
        const int N = grid_ns[l], V = (N + 1) * (N + 2) / 2;
        const float* in = tex + off_in;
        float* out = tex_out + off_out;
        const bool vec = C % 4 == 0 && (((uintptr_t)in | (uintptr_t)out) & 15) == 0;
        // The table pays when a CTA has many more texels than it tabulates, and
        // only where a texel's items are a power of two (level 5, table / texels:
        // C = 8, 2,000 triangles 65 / 53 us, 8,000 110 / 113, 32,000 273 / 331;
        // C = 16, 1,000 64 / 56, 4,000 103 / 117; C = 12, 32,000 580 / 419).
        // Scalar channels: C = 2, 8,000 92 / 84, 16,000 126 / 136; C = 6, 32,000
        // 819 / 360.
        const int per = vec ? C / 4 : C;
        const bool table = (per & (per - 1)) == 0 && (vec ? (long long)n_out * per >= 6000 : per <= 2 && n_out >= 16000);
        cudaError_t e = cudaSuccess;
        if (!table) {
            const long long texels = (long long)n_out * V;
            const int grid = persistent_grid((int)std::min<long long>((texels + 255) / 256, 1 << 30), 16);
            if (vec) k_rebuild_texels<true><<<grid, 256, 0, st>>>(in, N, C, plan_dev, n_out, out);
            else k_rebuild_texels<false><<<grid, 256, 0, st>>>(in, N, C, plan_dev, n_out, out);
            e = cudaGetLastError();
        } else {
            const size_t smem = sizeof(RebuildTap) * 6 * (size_t)V;
            const auto run = [&](auto kernel) {
                cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
                if (e != cudaSuccess) return e;
                const long long items = (long long)n_out * V * per;
                // at least eight items per thread; a multiple of `per` CTAs
                long long grid = std::min<long long>((items + 2047) / 2048, persistent_grid(1 << 30, 5));
                grid = (grid + per - 1) / per * per;
                kernel<<<(unsigned)grid, 256, smem, st>>>(in, N, C, plan_dev, n_out, out);
                return cudaGetLastError();
            };
            e = vec ? run(k_rebuild_level<true>) : run(k_rebuild_level<false>);
        }
        if (e != cudaSuccess) return e;
        note_launches(1);
        off_in += (size_t)T * V * C;
        off_out += (size_t)n_out * V * C;
    }
    return cudaGetLastError();
}

// One round of adaptive control on the host (the split/prune policy).
int adapt_plan(const int32_t* counts, const float* ratios, int T, float threshold, long long budget, int32_t* plan) {
    std::vector<int8_t> split(T, -1);
    long long n = T;
    for (int t = 0; t < T; ++t) {
        int e = 0;
        for (int k = 1; k < 3; ++k)
            if (ratios[3 * (size_t)t + k] > ratios[3 * (size_t)t + e]) e = k;
        if (ratios[3 * (size_t)t + e] > threshold) {
            split[t] = (int8_t)e;
            ++n;
        }
    }
    std::vector<char> removed(T, 0);
    if (budget >= 0 && n > budget) {
        std::vector<int> order(T);
        std::iota(order.begin(), order.end(), 0);
        std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return counts[a] < counts[b]; });
        for (int t : order) {
            if (n <= budget) break;
            removed[t] = 1;
            n -= split[t] >= 0 ? 2 : 1;
        }
    }
    int k = 0;
    for (int t = 0; t < T; ++t) {
        if (removed[t]) continue;
        if (split[t] < 0) {
            plan[k++] = t << 3;
        } else {
            plan[k++] = (t << 3) | (1 + 2 * split[t]);
            plan[k++] = (t << 3) | (2 + 2 * split[t]);
        }
    }
    return k;
}

// The random-initialisation round (host): remove the triangles no training
// image covers, then split the longest edges of the survivors with the
// largest ratios (each once) until the target count is reached.
int adapt_plan_fill(const int32_t* counts, const float* ratios, int T, long long target, int32_t* plan) {
    std::vector<int> keep;
    std::vector<int8_t> longest(T, 0);
    for (int t = 0; t < T; ++t) {
        if (counts[t] <= 0) continue;
        keep.push_back(t);
        int e = 0;
        for (int k = 1; k < 3; ++k)
            if (ratios[3 * (size_t)t + k] > ratios[3 * (size_t)t + e]) e = k;
        longest[t] = (int8_t)e;
    }
    long long want = target - (long long)keep.size();
    const size_t n_split = want <= 0 ? 0 : (size_t)std::min<long long>(want, (long long)keep.size());
    std::vector<int> order(keep);
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) {
        return ratios[3 * (size_t)a + longest[a]] > ratios[3 * (size_t)b + longest[b]];
    });
    std::vector<char> split(T, 0);
    for (size_t k = 0; k < n_split; ++k) split[order[k]] = 1;
    int k = 0;
    for (int t : keep) {
        if (split[t]) {
            plan[k++] = (t << 3) | (1 + 2 * longest[t]);
            plan[k++] = (t << 3) | (2 + 2 * longest[t]);
        } else {
            plan[k++] = t << 3;
        }
    }
    return k;
}

}  // namespace ds
