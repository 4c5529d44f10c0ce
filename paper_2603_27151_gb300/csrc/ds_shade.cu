// ds_shade.cu -- neural deferred shading (Sec. 3.3 "Neural deferred shading";
// supplementary "MLP Architecture"): per pixel and mask sample, the 7 colour
// features of the rasterised G-buffer and the degree-2 real spherical-
// harmonic encoding of the view direction (9 values) feed a 16 -> 16 -> 16 -> 3
// MLP (ReLU, ReLU, sigmoid); the first four features, read as RGBA, are
// blended with the MLP colour: rgb = A * feat_rgb + (1 - A) * mlp.
//
// Two forwards: on the tensor cores (k_shade_fwd_tc, tcgen05 kind::tf32 with
// a hi/lo split, described further down; the faster one and the default)
// and in FP32 on the CUDA cores (k_shade_fwd); the backward runs on the
// CUDA cores.  On the CUDA cores the MLP is ALU-bound (560 multiply-adds per
// pixel-sample against 40 bytes of traffic), so those kernels are organised
// to issue few instructions besides the FFMAs:
//  - the SH half of the first layer does not depend on the mask sample: it is
//    evaluated once per pixel and reused for all S samples;
//  - the parameters sit in shared memory and are read as float4 broadcasts,
//    each load shared by two samples of a pixel (forward) or by two pixels
//    (backward);
//  - the backward stages each round's activations and deltas in shared memory
//    and reduces the weight gradients as 4x8 outer-product blocks per thread
//    over the CTA's pixels, into one FP32 partial per CTA; a finish kernel
//    sums the partials in FP64 in a fixed order (deterministic gradients).
#include <string>

#include "ds_internal.h"

namespace ds {

namespace {

constexpr int kIn = 16, kHid = 16, kOut = 3, kFeat = 7, kSH = 9;
constexpr int oW1 = 0, oB1 = 256, oW2 = 272, oB2 = 528, oW3 = 544, oB3 = 592;
constexpr int kParams = DS_SHADE_N_PARAMS;   // 256 + 16 + 256 + 16 + 48 + 3
constexpr int kParamsPad = 596;   // shared copy padded to a float4 multiple
constexpr int kThreads = 256;

// Real SH basis of degree <= 2 (closed-form orthonormal harmonics, the usual
// graphics order and signs).
constexpr float kC0 = 0.28209479177387814f, kC1 = 0.4886025119029199f;
constexpr float kC2a = 1.0925484305920792f, kC2b = 0.31539156525252005f, kC2c = 0.5462742152960396f;

struct ShadeTable {
    int n, S, n_blocks, overwrite;
    ShadeView v[DS_MAX_VIEWS];
};

__device__ __forceinline__ int find_view(const ShadeTable& t, int blk) {
    int lo = 0, hi = t.n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (t.v[mid].blk0 <= blk) lo = mid; else hi = mid - 1;
    }
    return lo;
}

__device__ __forceinline__ void load_params(const float* __restrict__ g, float* sp) {
    for (int k = threadIdx.x; k < kParamsPad; k += blockDim.x) sp[k] = k < kParams ? __ldg(g + k) : 0.f;
}

// View direction of pixel (x, y) (unit world-space ray through the pixel
// centre) and its SH encoding.
__device__ __forceinline__ void sh_of_pixel(const ShadeView& V, int x, int y, float sh[kSH]) {
    const float dx = ((float)x + 0.5f - V.cx) / V.fx;
    const float dy = ((float)y + 0.5f - V.cy) / V.fy;
    float wx = fmaf(V.R[0], dx, fmaf(V.R[3], dy, V.R[6]));
    float wy = fmaf(V.R[1], dx, fmaf(V.R[4], dy, V.R[7]));
    float wz = fmaf(V.R[2], dx, fmaf(V.R[5], dy, V.R[8]));
    const float inv = 1.0f / sqrtf(fmaf(wx, wx, fmaf(wy, wy, wz * wz)));
    wx *= inv; wy *= inv; wz *= inv;
    sh[0] = kC0;
    sh[1] = -kC1 * wy;
    sh[2] = kC1 * wz;
    sh[3] = -kC1 * wx;
    sh[4] = kC2a * wx * wy;
    sh[5] = -kC2a * wy * wz;
    sh[6] = kC2b * (2.f * wz * wz - wx * wx - wy * wy);
    sh[7] = -kC2a * wx * wz;
    sh[8] = kC2c * (wx * wx - wy * wy);
}

// u = b1 + W1[:, 7:16] sh: the sample-independent part of the first layer.
__device__ __forceinline__ void first_layer_sh(const float* sp, const float sh[kSH], float u[kHid]) {
#pragma unroll
    for (int i = 0; i < kHid; ++i) {
        const float* w = sp + oW1 + i * kIn;
        float a = sp[oB1 + i];
#pragma unroll
        for (int k = 0; k < kSH; ++k) a = fmaf(w[kFeat + k], sh[k], a);
        u[i] = a;
    }
}

__device__ __forceinline__ float sigmoidf_(float z) { return 1.0f / (1.0f + expf(-z)); }

// Forward of NS samples of one pixel: h1, h2 (post-ReLU) and o (sigmoid).
template <int NS>
__device__ __forceinline__ void mlp(const float* sp, const float u[kHid], const float f[NS][kFeat],
                                    float h1[NS][kHid], float h2[NS][kHid], float o[NS][kOut]) {
#pragma unroll
    for (int i = 0; i < kHid; ++i) {
        const float4 w0 = *reinterpret_cast<const float4*>(sp + oW1 + i * kIn);
        const float4 w1 = *reinterpret_cast<const float4*>(sp + oW1 + i * kIn + 4);
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            float a = u[i];
            a = fmaf(w0.x, f[s][0], a); a = fmaf(w0.y, f[s][1], a);
            a = fmaf(w0.z, f[s][2], a); a = fmaf(w0.w, f[s][3], a);
            a = fmaf(w1.x, f[s][4], a); a = fmaf(w1.y, f[s][5], a);
            a = fmaf(w1.z, f[s][6], a);
            h1[s][i] = fmaxf(a, 0.f);
        }
    }
#pragma unroll
    for (int i = 0; i < kHid; ++i) {
        float a[NS];
#pragma unroll
        for (int s = 0; s < NS; ++s) a[s] = sp[oB2 + i];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float4 w = *reinterpret_cast<const float4*>(sp + oW2 + i * kHid + 4 * q);
#pragma unroll
            for (int s = 0; s < NS; ++s) {
                a[s] = fmaf(w.x, h1[s][4 * q + 0], a[s]); a[s] = fmaf(w.y, h1[s][4 * q + 1], a[s]);
                a[s] = fmaf(w.z, h1[s][4 * q + 2], a[s]); a[s] = fmaf(w.w, h1[s][4 * q + 3], a[s]);
            }
        }
#pragma unroll
        for (int s = 0; s < NS; ++s) h2[s][i] = fmaxf(a[s], 0.f);
    }
#pragma unroll
    for (int c = 0; c < kOut; ++c) {
        float a[NS];
#pragma unroll
        for (int s = 0; s < NS; ++s) a[s] = sp[oB3 + c];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float4 w = *reinterpret_cast<const float4*>(sp + oW3 + c * kHid + 4 * q);
#pragma unroll
            for (int s = 0; s < NS; ++s) {
                a[s] = fmaf(w.x, h2[s][4 * q + 0], a[s]); a[s] = fmaf(w.y, h2[s][4 * q + 1], a[s]);
                a[s] = fmaf(w.z, h2[s][4 * q + 2], a[s]); a[s] = fmaf(w.w, h2[s][4 * q + 3], a[s]);
            }
        }
#pragma unroll
        for (int s = 0; s < NS; ++s) o[s][c] = sigmoidf_(a[s]);
    }
}

template <int NS>
__device__ __forceinline__ void shade_samples(const float* sp, const ShadeView& V, const float u[kHid], int s0,
                                              int p) {
    float f[NS][kFeat], h1[NS][kHid], h2[NS][kHid], o[NS][kOut];
#pragma unroll
    for (int s = 0; s < NS; ++s)
#pragma unroll
        for (int c = 0; c < kFeat; ++c) f[s][c] = __ldcs(V.feat + ((size_t)(s0 + s) * kFeat + c) * V.HW + p);
    mlp<NS>(sp, u, f, h1, h2, o);
#pragma unroll
    for (int s = 0; s < NS; ++s) {
        const float A = f[s][3];
#pragma unroll
        for (int c = 0; c < kOut; ++c)
            __stcs(V.rgb + ((size_t)(s0 + s) * kOut + c) * V.HW + p, fmaf(A, f[s][c], (1.0f - A) * o[s][c]));
    }
}

// One thread per pixel, all S samples; blocks tile the concatenated pixels
// of all views.
__global__ void __launch_bounds__(kThreads) k_shade_fwd(const __grid_constant__ ShadeTable t,
                                                         const float* __restrict__ params) {
    __shared__ __align__(16) float sp[kParamsPad];
    load_params(params, sp);
    __syncthreads();
    const ShadeView& V = t.v[find_view(t, blockIdx.x)];
    const int p = (blockIdx.x - V.blk0) * kThreads + threadIdx.x;
    if (p >= V.HW) return;
    float sh[kSH], u[kHid];
    sh_of_pixel(V, p % V.W, p / V.W, sh);
    first_layer_sh(sp, sh, u);
    int s = 0;
    for (; s + 2 <= t.S; s += 2) shade_samples<2>(sp, V, u, s, p);
    if (s < t.S) shade_samples<1>(sp, V, u, s, p);
}

// ---------------------------------------------------------------------------
// Backward.
//
// A CTA of 128 threads takes 256 pixels, two per thread, one sample a round.
// Staging per round, row-major [p][20]: X (input: features, SH), H1, H2,
// D1 = dL/dz1, D2 = dL/dz2, and D3 = dL/dz3 (padded to 4).  Reduction: 7 pixel
// groups x 16 blocks of 4 x 8 weights; block b < 8 owns gW1[4(b/2)..][8(b%2)..]
// (+ gb1 if b is even), b >= 8 the same of gW2, and each block a column of gW3
// (+ gb3 if b = 0).
//
// Bound by the shared-memory pipe, then by the FMA pipe.  With one pixel per
// thread and 4 x 4 blocks a weight load fed four multiply-adds and a reducer's
// two loads sixteen: 840 shared wavefronts per 32 pixel-samples, 74% of the
// pipe's peak, FMA pipe at 40%.  Here a weight load feeds four outputs of two
// pixels, a reducer's three loads 32 multiply-adds, and two multiply-adds are
// one packed instruction: in the layers the weights of neighbouring outputs
// are pairs (stored transposed for the forward) and the activation is in both
// halves; in a reducer the products (d0, d1) x (a0, a1) and (d1, d0) x (a0, a1)
// give all four.  Every sum keeps its order: the layers that of the forward
// kernel, the weight gradients the rows 7 apart of the CTA's blocks.
// Four 1080p views and one of 1023 x 577, S = 2: 1958 -> 1555 us (shared 60% of
// its peak, FMA pipe's issue 30% at two cycles per packed instruction, issue
// 47%; 8 warps per SM, as 224 registers and 108 KB per CTA allow).  16 pixel
// groups x 8 blocks of 8 x 8 were faster (1440) but sum in another order.
constexpr int kPix = kThreads;           // pixels of a block
constexpr int kBwdThreads = kPix / 2;
constexpr int kGroups = 7, kBlocks = 16;
constexpr int kRow = 20;   // 16 values + 4 pad: conflict-free float4 stores of the rows

// A warp of reducers reads two rows of D1 and D2 (of X and H1) at once: the
// 64-byte pads put those arrays on complementary shared-memory banks.
struct BwdSmem {
    float sp[kParamsPad];
    float W1T[kIn][kHid], W2T[kHid][kHid], W3T[kHid][4];   // [input][output]
    float X[kPix][kRow];
    float pad0[16];
    float H1[kPix][kRow], H2[kPix][kRow], D1[kPix][kRow];
    float pad1[16];
    float D2[kPix][kRow];
    float D3[kPix][4];
};
static_assert(sizeof(float) * kGroups * kParams <= sizeof(float) * (2 * kPix * kRow + 16), "reduction buffer");
static_assert(2 * (sizeof(BwdSmem) + 1024) <= 228 * 1024, "two CTAs per SM");

// The sample-independent part of the first layer (16 values per pixel) kept
// in the 4 pad columns of the pixel's X, H1, H2 and D1 rows (the reducers
// read columns 0..15 only).
__device__ __forceinline__ float4* upad(BwdSmem& sm, int row, int q) {
    return reinterpret_cast<float4*>(q == 0 ? &sm.X[row][16] : q == 1 ? &sm.H1[row][16] : q == 2 ? &sm.H2[row][16] : &sm.D1[row][16]);
}

__device__ __forceinline__ void store4(float* dst, const float* v) {
    *reinterpret_cast<float4*>(dst) = make_float4(v[0], v[1], v[2], v[3]);
}

// acc[i] += (w[2 i], w[2 i + 1]) x for N pairs of weights in shared memory and
// the two pixels' x.
template <int N>
__device__ __forceinline__ void fma_pairs(const float* w, float x0, float x1, float2 (&a0)[N], float2 (&a1)[N]) {
    const float2 xx0 = make_float2(x0, x0), xx1 = make_float2(x1, x1);
#pragma unroll
    for (int i = 0; i < N; i += 2) {
        const float4 v = *reinterpret_cast<const float4*>(w + 2 * i);
        a0[i] = __ffma2_rn(make_float2(v.x, v.y), xx0, a0[i]);
        a1[i] = __ffma2_rn(make_float2(v.x, v.y), xx1, a1[i]);
        a0[i + 1] = __ffma2_rn(make_float2(v.z, v.w), xx0, a0[i + 1]);
        a1[i + 1] = __ffma2_rn(make_float2(v.z, v.w), xx1, a1[i + 1]);
    }
}
__device__ __forceinline__ float elem(const float2* a, int i) { return i & 1 ? a[i >> 1].y : a[i >> 1].x; }
template <int N>
__device__ __forceinline__ void store_pairs(float* dst, const float2 (&a)[N]) {
#pragma unroll
    for (int i = 0; i < N; i += 2)
        reinterpret_cast<float4*>(dst)[i / 2] = make_float4(a[i].x, a[i].y, a[i + 1].x, a[i + 1].y);
}

__global__ void __launch_bounds__(kBwdThreads, 2) k_shade_bwd(const __grid_constant__ ShadeTable t,
                                                               const float* __restrict__ params,
                                                               float* __restrict__ partial) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    BwdSmem& sm = *reinterpret_cast<BwdSmem*>(smem_raw);
    const float* sp = sm.sp;
    load_params(params, sm.sp);

    const int tid = threadIdx.x;
    const int grp = tid / kBlocks, blk = tid % kBlocks;
    const bool reducer = grp < kGroups;
    const int layer = blk >> 3;                             // 0: W1, 1: W2
    const int ib = (blk >> 1) & 3, jb = blk & 1;            // row block, column block
    const float* Dsrc = (layer == 0 ? &sm.D1[0][0] : &sm.D2[0][0]) + 4 * ib;
    const float* Asrc = (layer == 0 ? &sm.X[0][0] : &sm.H1[0][0]) + 8 * jb;
    float2 accP[2][4], accQ[2][4], accb[2];   // (d0 a0, d1 a1); (d1 a0, d0 a1); (d0, d1)
    float2 acc3 = make_float2(0.f, 0.f), accb3 = make_float2(0.f, 0.f);   // gW3[0, 1][blk], gb3[0, 1]
    float acc3z = 0.f, accb3z = 0.f;                                      // the third output's
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        accb[i] = make_float2(0.f, 0.f);
#pragma unroll
        for (int j = 0; j < 4; ++j) accP[i][j] = accQ[i][j] = make_float2(0.f, 0.f);
    }
    __syncthreads();
    for (int k = tid; k < kHid * kIn; k += kBwdThreads) {
        sm.W1T[k % kIn][k / kIn] = sp[oW1 + k];
        sm.W2T[k % kHid][k / kHid] = sp[oW2 + k];
    }
    for (int k = tid; k < 4 * kHid; k += kBwdThreads) sm.W3T[k >> 2][k & 3] = (k & 3) < kOut ? sp[oW3 + (k & 3) * kHid + (k >> 2)] : 0.f;
    __syncthreads();

    // A round's features and gradients are loaded before the reduction of the
    // round before it, where registers are free.
    float f[2][8], g[2][kOut];
    const auto load = [&](int b, int s) {
        const ShadeView& V = t.v[find_view(t, b)];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int p = (b - V.blk0) * kPix + e * kBwdThreads + tid;
            const bool valid = p < V.HW;
#pragma unroll
            for (int c = 0; c < kFeat; ++c) f[e][c] = valid ? __ldg(V.feat + ((size_t)s * kFeat + c) * V.HW + p) : 0.f;
#pragma unroll
            for (int c = 0; c < kOut; ++c) g[e][c] = valid ? __ldcs(V.grad_rgb + ((size_t)s * kOut + c) * V.HW + p) : 0.f;
        }
    };
    load(blockIdx.x, 0);
#pragma unroll 1
    for (int b = blockIdx.x; b < t.n_blocks; b += gridDim.x) {
        const ShadeView& V = t.v[find_view(t, b)];
        int p[2];
        bool valid[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            p[e] = (b - V.blk0) * kPix + e * kBwdThreads + tid;
            valid[e] = p[e] < V.HW;
        }
        {
            // the SH columns 8..15 of the input row are the same for every
            // sample (column 7, the constant band, is stored with the features)
            float sh[2][kSH] = {};
            float2 u[2][kHid / 2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                if (valid[e]) sh_of_pixel(V, p[e] % V.W, p[e] / V.W, sh[e]);
                store4(&sm.X[e * kBwdThreads + tid][8], sh[e] + 1);
                store4(&sm.X[e * kBwdThreads + tid][12], sh[e] + 5);
#pragma unroll
                for (int i = 0; i < kHid / 2; ++i) u[e][i] = make_float2(sp[oB1 + 2 * i], sp[oB1 + 2 * i + 1]);
            }
#pragma unroll
            for (int k = 0; k < kSH; ++k) fma_pairs(sm.W1T[kFeat + k], sh[0][k], sh[1][k], u[0], u[1]);
#pragma unroll
            for (int e = 0; e < 2; ++e)
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    *upad(sm, e * kBwdThreads + tid, q) = make_float4(u[e][2 * q].x, u[e][2 * q].y, u[e][2 * q + 1].x, u[e][2 * q + 1].y);
        }
#pragma unroll 1
        for (int s = 0; s < t.S; ++s) {
            float d3[2][4];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                f[e][7] = kC0;
                store4(&sm.X[e * kBwdThreads + tid][0], f[e]);
                store4(&sm.X[e * kBwdThreads + tid][4], f[e] + 4);
            }
            // forward: rows are staged as soon as they are known
            float2 h1[2][kHid / 2], h2[2][kHid / 2];
#pragma unroll
            for (int e = 0; e < 2; ++e)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float4 v = *upad(sm, e * kBwdThreads + tid, q);
                    h1[e][2 * q] = make_float2(v.x, v.y);
                    h1[e][2 * q + 1] = make_float2(v.z, v.w);
                }
#pragma unroll
            for (int k = 0; k < kFeat; ++k) fma_pairs(sm.W1T[k], f[0][k], f[1][k], h1[0], h1[1]);
#pragma unroll
            for (int e = 0; e < 2; ++e) {
#pragma unroll
                for (int i = 0; i < kHid / 2; ++i) {
                    h1[e][i] = make_float2(fmaxf(h1[e][i].x, 0.f), fmaxf(h1[e][i].y, 0.f));
                    h2[e][i] = *reinterpret_cast<const float2*>(sp + oB2 + 2 * i);
                }
                store_pairs(sm.H1[e * kBwdThreads + tid], h1[e]);
            }
#pragma unroll
            for (int k = 0; k < kHid; ++k) fma_pairs(sm.W2T[k], elem(h1[0], k), elem(h1[1], k), h2[0], h2[1]);
            float o[2][kOut];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
#pragma unroll
                for (int i = 0; i < kHid / 2; ++i) h2[e][i] = make_float2(fmaxf(h2[e][i].x, 0.f), fmaxf(h2[e][i].y, 0.f));
                store_pairs(sm.H2[e * kBwdThreads + tid], h2[e]);
#pragma unroll
                for (int c = 0; c < kOut; ++c) o[e][c] = sp[oB3 + c];
            }
#pragma unroll
            for (int i = 0; i < kHid; ++i) {
                const float4 w = *reinterpret_cast<const float4*>(sm.W3T[i]);
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const float h = elem(h2[e], i);
                    o[e][0] = fmaf(w.x, h, o[e][0]);
                    o[e][1] = fmaf(w.y, h, o[e][1]);
                    o[e][2] = fmaf(w.z, h, o[e][2]);
                }
            }
            float gA[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const float A = f[e][3];
                gA[e] = 0.f;
#pragma unroll
                for (int c = 0; c < kOut; ++c) {
                    const float oc = sigmoidf_(o[e][c]);
                    gA[e] = fmaf(g[e][c], f[e][c] - oc, gA[e]);
                    const float go = (1.0f - A) * g[e][c];
                    d3[e][c] = valid[e] ? go * oc * (1.0f - oc) : 0.f;
                }
                d3[e][3] = 0.f;
                store4(sm.D3[e * kBwdThreads + tid], d3[e]);
            }
            // d2_j = (W3^T d3)_j [z2_j > 0]
            float2 d2[2][kHid / 2] = {}, d1[2][kHid / 2] = {};
#pragma unroll
            for (int c = 0; c < kOut; ++c) fma_pairs(sp + oW3 + c * kHid, d3[0][c], d3[1][c], d2[0], d2[1]);
#pragma unroll
            for (int e = 0; e < 2; ++e) {
#pragma unroll
                for (int i = 0; i < kHid / 2; ++i)
                    d2[e][i] = make_float2(h2[e][i].x > 0.f ? d2[e][i].x : 0.f, h2[e][i].y > 0.f ? d2[e][i].y : 0.f);
                store_pairs(sm.D2[e * kBwdThreads + tid], d2[e]);
            }
            // d1 = (W2^T d2) [z1 > 0]
#pragma unroll
            for (int j = 0; j < kHid; ++j) fma_pairs(sp + oW2 + j * kHid, elem(d2[0], j), elem(d2[1], j), d1[0], d1[1]);
#pragma unroll
            for (int e = 0; e < 2; ++e) {
#pragma unroll
                for (int i = 0; i < kHid / 2; ++i)
                    d1[e][i] = make_float2(h1[e][i].x > 0.f ? d1[e][i].x : 0.f, h1[e][i].y > 0.f ? d1[e][i].y : 0.f);
                store_pairs(sm.D1[e * kBwdThreads + tid], d1[e]);
            }
            // feature gradient: blend terms + (W1^T d1)[0:7]
            if (V.grad_feat) {
                float2 gf[2][4] = {};
#pragma unroll
                for (int k = 0; k < kHid; ++k) fma_pairs(sp + oW1 + k * kIn, elem(d1[0], k), elem(d1[1], k), gf[0], gf[1]);
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    if (!valid[e]) continue;
                    float* dst = V.grad_feat + (size_t)s * kFeat * V.HW + p[e];
#pragma unroll
                    for (int c = 0; c < kFeat; ++c) {
                        float v = elem(gf[e], c);
                        if (c < kOut) v = fmaf(f[e][3], g[e][c], v);
                        if (c == 3) v += gA[e];
                        if (t.overwrite) dst[(size_t)c * V.HW] = v;
                        else dst[(size_t)c * V.HW] += v;
                    }
                }
            }
            // a pixel past the view's end adds nothing, whatever the weights are
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                if (valid[e]) continue;
                const int r = e * kBwdThreads + tid;
                for (int c = 0; c < kHid; ++c) sm.X[r][c] = sm.H1[r][c] = sm.H2[r][c] = sm.D1[r][c] = sm.D2[r][c] = 0.f;
            }
            if (s + 1 < t.S) load(b, s + 1);
            else if (b + gridDim.x < t.n_blocks) load(b + gridDim.x, 0);
            __syncthreads();
            if (reducer) {
#pragma unroll 4
                for (int q = grp; q < kPix; q += kGroups) {
                    const float4 dv = *reinterpret_cast<const float4*>(Dsrc + q * kRow);
                    const float4 aa = *reinterpret_cast<const float4*>(Asrc + q * kRow);
                    const float4 ab = *reinterpret_cast<const float4*>(Asrc + q * kRow + 4);
                    const float4 dz = *reinterpret_cast<const float4*>(sm.D3[q]);
                    const float hz = sm.H2[q][blk];
                    const float2 d[2] = {{dv.x, dv.y}, {dv.z, dv.w}}, sw[2] = {{dv.y, dv.x}, {dv.w, dv.z}};
                    const float2 a[4] = {{aa.x, aa.y}, {aa.z, aa.w}, {ab.x, ab.y}, {ab.z, ab.w}};
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            accP[i][j] = __ffma2_rn(d[i], a[j], accP[i][j]);
                            accQ[i][j] = __ffma2_rn(sw[i], a[j], accQ[i][j]);
                        }
                        accb[i] = __fadd2_rn(accb[i], d[i]);
                    }
                    const float2 d01 = make_float2(dz.x, dz.y);
                    acc3 = __ffma2_rn(d01, make_float2(hz, hz), acc3);
                    acc3z = fmaf(dz.z, hz, acc3z);
                    accb3 = __fadd2_rn(accb3, d01);
                    accb3z += dz.z;
                }
            }
            __syncthreads();
        }
    }

    // Reduce the pixel groups in shared memory, then one partial per CTA.
    float* red = &sm.X[0][0];   // [kGroups][kParams]
    if (reducer) {
        float* r = red + grp * kParams;
        const int oW = layer == 0 ? oW1 : oW2, oB = layer == 0 ? oB1 : oB2;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int row = 4 * ib + i;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const float2 v = ((i ^ j) & 1) ? accQ[i >> 1][j >> 1] : accP[i >> 1][j >> 1];
                r[oW + row * kHid + 8 * jb + j] = j & 1 ? v.y : v.x;
            }
            if (jb == 0) r[oB + row] = elem(accb, i);
        }
        r[oW3 + blk] = acc3.x;
        r[oW3 + kHid + blk] = acc3.y;
        r[oW3 + 2 * kHid + blk] = acc3z;
        if (blk == 0) {
            r[oB3] = accb3.x;
            r[oB3 + 1] = accb3.y;
            r[oB3 + 2] = accb3z;
        }
    }
    __syncthreads();
    for (int k = tid; k < kParams; k += kBwdThreads) {
        float a = 0.f;
#pragma unroll
        for (int g = 0; g < kGroups; ++g) a += red[g * kParams + k];
        partial[(size_t)blockIdx.x * kParams + k] = a;
    }
}

// grad_params[k] (+)= sum over CTAs of partial[c][k] in FP64, in a fixed order:
// warp w of the block sums the CTAs w, w + 16, ... for 32 parameters, and the
// 16 sums are added in order.  A thread per parameter over all 304 partials was
// one long chain of loads (49 us; 10 now).
constexpr int kFinWarps = 16;
__global__ void __launch_bounds__(32 * kFinWarps) k_shade_finish(const float* __restrict__ partial, int n_cta,
                                                                 float* __restrict__ out, int overwrite) {
    __shared__ double s_sum[kFinWarps][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, k = blockIdx.x * 32 + lane;
    double a = 0.0;
    if (k < kParams) {
#pragma unroll 4
        for (int c = warp; c < n_cta; c += kFinWarps) a += (double)partial[(size_t)c * kParams + k];
    }
    s_sum[warp][lane] = a;
    __syncthreads();
    if (warp > 0 || k >= kParams) return;
#pragma unroll
    for (int w = 1; w < kFinWarps; ++w) a += s_sum[w][lane];
    out[k] = overwrite ? (float)a : (float)((double)out[k] + a);
}

// ---------------------------------------------------------------------------
// Forward on the tensor cores: the three layers as tcgen05.mma of kind::tf32
// (Blackwell 5th-generation tensor cores).  A tile is 128 pixel-samples, one
// per thread and one tensor-memory lane each (M = 128); N = 16 hidden units
// (the 3 outputs padded to 16); K = 16 inputs in two MMAs of K = 8.  TF32
// keeps 10 mantissa bits, so every operand is split into hi = the TF32
// truncation and lo = the remainder (exact in FP32) and each product is taken
// as x_lo w_hi + x_hi w_lo + x_hi w_hi (the x_lo w_lo term, about 2^-21 of the
// product, is dropped): six MMAs per layer, and a seventh adds the bias (a
// constant K-chunk (1, 1, 0, ...) times the bias tile (b hi, b lo)), issued
// by one thread and completed on an mbarrier.
//
// The layer inputs (operand A) live in tensor memory beside the FP32
// accumulator: each thread writes its row with tcgen05.st and the MMAs read A
// from there, so shared memory carries only the weight and bias tiles (B, 9
// KB).  With A in shared memory every MMA re-read 4 KB of it, and the
// shared-memory bandwidth, not the tensor cores, set the kernel's speed.  Per
// layer the 128 threads read their accumulator row (tcgen05.ld), apply the
// activation and write the next layer's hi/lo row.
namespace tc {

constexpr int kRows = 128;   // pixel-samples per tile = TMEM lanes = M
// Tensor-memory columns of a CTA (one 32-bit value per column and lane): the
// accumulator D in 0..15, A hi in 16..31, A lo in 32..47, and in 48..55 the
// constant K-chunk (1, 1, 0, ..., 0) that adds the bias rows (b hi, b lo) of
// the bias tile.
constexpr uint32_t kTmemCols = 64;
constexpr uint32_t kColD = 0, kColAh = 16, kColAl = 32, kColOne = 48;
constexpr int kMaxCtasPerSm = 512 / (int)kTmemCols;   // the SM's 512 columns, none left waiting
// Instruction descriptor of kind::tf32: D FP32 (bits 4-5 = 1), A and B TF32
// (bits 7-9 and 10-12 = 2), both K-major (bits 15, 16 = 0), N >> 3 in bits
// 17-22, M >> 4 in bits 24-28.
constexpr uint32_t kIdesc = (1u << 4) | (2u << 7) | (2u << 10) | ((16u >> 3) << 17) | ((128u >> 4) << 24);

// Byte offset of element (n, k) of a 16 x 16 K-major TF32 operand in shared
// memory in the canonical layout without swizzle: core matrices of 8 rows x
// 16 bytes (4 values), 128 bytes each; the two core matrices of one MMA's
// K = 8 are 128 bytes apart (leading-dimension offset), the two 8-row groups
// 512 bytes apart (stride-dimension offset).
__device__ __forceinline__ uint32_t op_off(int n, int k) {
    return (uint32_t)(((((n >> 3) << 2) + (k >> 2)) << 7) + ((n & 7) << 4) + ((k & 3) << 2));
}

// Shared-memory matrix descriptor: start address, leading and stride byte
// offsets (all >> 4), descriptor version 1 (bit 46), no swizzle.
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr) {
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(128u >> 4) << 16) | ((uint64_t)(512u >> 4) << 32) |
           (1ull << 46);
}

__device__ __forceinline__ uint32_t saddr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

struct Smem {
    uint8_t w[6][1024];   // W1 hi, W1 lo, W2 hi, W2 lo, W3 hi, W3 lo (N 16 x K 16)
    uint8_t b[3][1024];   // bias tiles of the three layers: K = 0 b hi, K = 1 b lo, else 0
    unsigned long long bar;
    uint32_t tmem;
};

// TF32 hi part (truncation to 10 mantissa bits) and FP32 remainder.
__device__ __forceinline__ void split(float x, uint32_t& h, uint32_t& l) {
    h = __float_as_uint(x) & 0xFFFFE000u;
    l = __float_as_uint(x - __uint_as_float(h));
}

// 16 columns of this thread's lane from column `col` on (warp w owns lanes
// 32w .. 32w + 31, the lane field sits in bits 16-31 of the address).
__device__ __forceinline__ uint32_t lane_addr(uint32_t tmem, uint32_t col) {
    return tmem + ((uint32_t)(threadIdx.x & ~31) << 16) + col;
}

__device__ __forceinline__ void st8(uint32_t ta, const uint32_t (&r)[8]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};\n" ::"r"(ta), "r"(r[0]),
                 "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
                 : "memory");
}

// Write eight values of this thread's operand row, K = 8 half .. 8 half + 7,
// as their hi and lo parts into tensor memory.
__device__ __forceinline__ void store_half(uint32_t tmem, int half, const uint32_t (&h)[8], const uint32_t (&l)[8]) {
    st8(lane_addr(tmem, kColAh + 8 * half), h);
    st8(lane_addr(tmem, kColAl + 8 * half), l);
}

__device__ __forceinline__ void split8(const float* x, uint32_t (&h)[8], uint32_t (&l)[8]) {
#pragma unroll
    for (int i = 0; i < 8; ++i) split(x[i], h[i], l[i]);
}

__device__ __forceinline__ void mma(uint32_t d, uint32_t a_tmem, uint64_t b, uint32_t accumulate) {
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::tf32 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d),
        "r"(a_tmem), "l"(b), "r"(kIdesc), "r"(accumulate));
}

// Layer L: D = A_lo W_hi + A_hi W_lo + A_hi W_hi (small terms first) + the
// bias, then the commit that arrives on the barrier when the MMAs are
// complete.  One thread.
__device__ __forceinline__ void issue_layer(Smem& sm, int L, uint32_t tmem) {
    const uint32_t b0 = saddr(sm.w[2 * L]), b1 = saddr(sm.w[2 * L + 1]);
    const uint32_t d = tmem + kColD;
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        mma(d, tmem + kColAl + 8 * s, smem_desc(b0 + 256 * s), s);
        mma(d, tmem + kColAh + 8 * s, smem_desc(b1 + 256 * s), 1);
    }
#pragma unroll
    for (int s = 0; s < 2; ++s) mma(d, tmem + kColAh + 8 * s, smem_desc(b0 + 256 * s), 1);
    mma(d, tmem + kColOne, smem_desc(saddr(sm.b[L])), 1);
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(saddr(&sm.bar))
                 : "memory");
}

// Wait for phase `parity` of the barrier, for at most about 2^31 SM clocks.
__device__ __forceinline__ bool wait_bar(const Smem& sm, uint32_t parity) {
    const uint32_t b = saddr(&sm.bar);
    const long long t0 = clock64();
    for (;;) {
        uint32_t done;
        asm volatile(
            "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(b), "r"(parity)
            : "memory");
        if (done) return true;
        if (clock64() - t0 > (1ll << 31)) return false;
    }
}

// This thread's accumulator row, 16 columns.
__device__ __forceinline__ void load_row(uint32_t tmem, float (&v)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(lane_addr(tmem, kColD)));
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// This thread's tensor-memory stores complete, and they and its earlier
// tensor-memory loads ordered before the barrier that follows.
__device__ __forceinline__ void before_sync() {
    asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
}

// Logistic function from the hardware exponential and the correctly rounded
// reciprocal (a few 1e-7 from the exact value on [0, 1]).
__device__ __forceinline__ float sigmoid(float z) { return __frcp_rn(1.0f + __expf(-z)); }

}  // namespace tc

// Per round a CTA takes one tile: 128 consecutive pixels of one view (tiles
// never straddle views: view v owns tiles blk0 .. blk0 + ceil(HW / 128) - 1)
// and all S mask samples of them in turn.  The SH encoding of the pixel and
// its hi/lo split are computed once per tile; per sample the thread writes
// its input row (7 features, then the 9 SH values) and the three layers
// run.  The next sample's features are loaded before the current sample's
// MMAs.  Persistent CTAs of 128 threads.  A wait for the MMAs that runs out
// (about a second) sets bit 1 of *status, and the CTA releases its tensor
// memory and returns.  kNoMma: the MMAs are never issued, so that every wait
// runs out (for testing the bounded wait on a GPU).
template <bool kNoMma>
__global__ void __launch_bounds__(tc::kRows, tc::kMaxCtasPerSm) k_shade_fwd_tc(const __grid_constant__ ShadeTable t,
                                                          const float* __restrict__ params, int* __restrict__ status) {
    using namespace tc;
    extern __shared__ uint8_t smem_raw[];
    Smem& sm = *reinterpret_cast<Smem*>(smem_raw + ((1024u - (saddr(smem_raw) & 1023u)) & 1023u));
    const int tid = threadIdx.x, warp = tid >> 5;
    // weights -> TF32 hi/lo operand tiles (W3's 3 rows padded with zeros)
    for (int q = tid; q < 3 * 256; q += kRows) {
        const int L = q >> 8, n = (q >> 4) & 15, k = q & 15;
        const int o = L == 0 ? oW1 : (L == 1 ? oW2 : oW3);
        const float w = (L < 2 || n < kOut) ? __ldg(params + o + n * 16 + k) : 0.f;
        uint32_t h, l;
        split(w, h, l);
        *reinterpret_cast<uint32_t*>(sm.w[2 * L] + op_off(n, k)) = h;
        *reinterpret_cast<uint32_t*>(sm.w[2 * L + 1] + op_off(n, k)) = l;
    }
    for (int q = tid; q < 3 * 256; q += kRows) {
        const int L = q >> 8, n = (q >> 4) & 15, k = q & 15;
        const int o = L == 0 ? oB1 : (L == 1 ? oB2 : oB3);
        const float b = (k < 2 && (L < 2 || n < kOut)) ? __ldg(params + o + n) : 0.f;
        uint32_t h, l;
        split(b, h, l);
        *reinterpret_cast<uint32_t*>(sm.b[L] + op_off(n, k)) = k == 0 ? h : (k == 1 ? l : 0u);
    }
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(saddr(&sm.bar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(saddr(&sm.tmem)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    // the weight tiles (generic-proxy writes) visible to the MMAs
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    before_sync();
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = sm.tmem;
    {
        const uint32_t one = __float_as_uint(1.0f);
        const uint32_t r[8] = {one, one, 0u, 0u, 0u, 0u, 0u, 0u};
        st8(lane_addr(tmem, kColOne), r);
    }
    uint32_t phase = 0;
    bool ok = true;
    for (int tile = blockIdx.x; tile < t.n_blocks && ok; tile += gridDim.x) {
        const ShadeView& V = t.v[find_view(t, tile)];
        const int p = (tile - V.blk0) * kRows + tid;
        const bool valid = p < V.HW;
        const int py = valid ? p / V.W : 0, px = valid ? p - py * V.W : 0;
        // input columns 8..15 (SH bands 1..8), split once for all samples;
        // column 7 is the constant band
        uint32_t shh[8], shl[8];
        {
            float sh[kSH];
            sh_of_pixel(V, px, py, sh);
            split8(sh + 1, shh, shl);
        }
        const float* fp = V.feat + (valid ? p : 0);
        float fn[kFeat];
#pragma unroll
        for (int c = 0; c < kFeat; ++c) fn[c] = valid ? __ldcs(fp + (size_t)c * V.HW) : 0.f;
        for (int s = 0; s < t.S; ++s) {
            float f[kFeat];
#pragma unroll
            for (int c = 0; c < kFeat; ++c) f[c] = fn[c];
            if (s + 1 < t.S) {
#pragma unroll
                for (int c = 0; c < kFeat; ++c)
                    fn[c] = valid ? __ldcs(fp + ((size_t)(s + 1) * kFeat + c) * V.HW) : 0.f;
            }
            {
                const float x[8] = {f[0], f[1], f[2], f[3], f[4], f[5], f[6], kC0};
                uint32_t h[8], l[8];
                split8(x, h, l);
                store_half(tmem, 0, h, l);
                store_half(tmem, 1, shh, shl);
            }
            float o[kOut];
#pragma unroll
            for (int L = 0; L < 3; ++L) {
                // the rows are complete and every thread's reads of the
                // previous accumulator are done: the next MMAs may start
                before_sync();
                __syncthreads();
                if (tid == 0 && !kNoMma) issue_layer(sm, L, tmem);
                ok = __syncthreads_and(wait_bar(sm, phase));
                phase ^= 1u;
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                float d[16];
                load_row(tmem, d);
                if (L < 2) {
#pragma unroll
                    for (int i = 0; i < 16; ++i) d[i] = fmaxf(d[i], 0.f);
#pragma unroll
                    for (int half = 0; half < 2; ++half) {
                        uint32_t h[8], l[8];
                        split8(d + 8 * half, h, l);
                        store_half(tmem, half, h, l);
                    }
                } else {
#pragma unroll
                    for (int c = 0; c < kOut; ++c) o[c] = sigmoid(d[c]);
                }
            }
            if (!ok) break;
            if (valid) {
                const float A = f[3];
#pragma unroll
                for (int c = 0; c < kOut; ++c)
                    __stcs(V.rgb + ((size_t)s * kOut + c) * V.HW + p, fmaf(A, f[c], (1.0f - A) * o[c]));
            }
        }
    }
    if (!ok) {
        // a layer's MMAs did not complete in time: record it, give them one
        // more bounded wait, then release the tensor memory and return
        if (tid == 0) atomicOr(status, 2);
        wait_bar(sm, phase ^ 1u);
    }
    before_sync();
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(kTmemCols) : "memory");
    }
}

void fill_table(ShadeTable& t, const ShadeView* views, int n, int S, bool overwrite) {
    t.n = n;
    t.S = S;
    t.overwrite = overwrite ? 1 : 0;
    int blk = 0;
    for (int i = 0; i < n; ++i) {
        t.v[i] = views[i];
        t.v[i].HW = views[i].W * views[i].H;
        t.v[i].blk0 = blk;
        blk += (t.v[i].HW + kThreads - 1) / kThreads;
    }
    t.n_blocks = blk;
}

}  // namespace

int shade_bwd_grid() {
    static int cached = 0;
    if (cached > 0) return cached;
    int blocks = 0;
    const size_t smem = sizeof(BwdSmem);
    if (cudaFuncSetAttribute(k_shade_bwd, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, k_shade_bwd, kBwdThreads, smem) != cudaSuccess ||
        blocks < 1) {
        cudaGetLastError();
        blocks = 1;
    }
    cached = persistent_grid(1 << 30, blocks);
    return cached;
}

size_t shade_partial_floats(int grid) { return (size_t)grid * kParams; }

cudaError_t launch_shade_fwd(const ShadeView* views, int n, int S, const float* params, cudaStream_t st) {
    ShadeTable t;
    fill_table(t, views, n, S, false);
    if (t.n_blocks == 0 || S == 0) return cudaSuccess;
    k_shade_fwd<<<t.n_blocks, kThreads, 0, st>>>(t, params);
    note_launches(1);
    return cudaGetLastError();
}

// Launch shape of k_shade_fwd_tc: dynamic shared memory and CTAs per SM.
// Each CTA holds kTmemCols of the SM's 512 tensor-memory columns, so at most
// kMaxCtasPerSm may be resident at once (a further CTA's allocation would
// wait for a CTA to finish); the shared-memory request is padded so that no
// more fit, and the residency is the least of what shared memory, registers
// and threads allow.  Computed here from the kernel's attributes: the
// runtime's occupancy query answers 1 for this kernel although more CTAs fit.
bool tc_launch_shape(size_t* dyn_smem, int* per_sm) {
    static size_t c_smem = 0;
    static int c_per_sm = 0;
    if (c_per_sm > 0) {
        *dyn_smem = c_smem;
        *per_sm = c_per_sm;
        return true;
    }
    cudaFuncAttributes fa;
    int dev = 0, smem_sm = 0, reserved = 0, regs_sm = 0, thr_sm = 0;
    if (cudaFuncGetAttributes(&fa, k_shade_fwd_tc<false>) != cudaSuccess || cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&regs_sm, cudaDevAttrMaxRegistersPerMultiprocessor, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&thr_sm, cudaDevAttrMaxThreadsPerMultiProcessor, dev) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    const size_t fixed = fa.sharedSizeBytes + (size_t)reserved;
    size_t smem = sizeof(tc::Smem) + 1024;   // + room to align the weight tiles to 1 KB
    const size_t at_least = (size_t)smem_sm / (tc::kMaxCtasPerSm + 1) + 1;   // kMaxCtasPerSm + 1 do not fit
    if (smem + fixed < at_least) smem = at_least - fixed;
    const int by_smem = (int)((size_t)smem_sm / (smem + fixed));
    const int regs_warp = ((fa.numRegs * 32 + 255) / 256) * 256;   // allocated per warp in units of 256
    const int by_regs = regs_warp > 0 ? regs_sm / (regs_warp * (tc::kRows / 32)) : tc::kMaxCtasPerSm;
    const int by_thr = thr_sm / tc::kRows;
    int n = by_smem < by_regs ? by_smem : by_regs;
    n = n < by_thr ? n : by_thr;
    if (n < 1 || n > tc::kMaxCtasPerSm) return false;
    c_smem = smem;
    c_per_sm = n;
    *dyn_smem = smem;
    *per_sm = n;
    return true;
}

cudaError_t launch_shade_fwd_tc(const ShadeView* views, int n, int S, const float* params, int* status,
                                cudaStream_t st, bool no_mma) {
    ShadeTable t;
    t.n = n;
    t.S = S;
    t.overwrite = 0;
    int blk = 0;
    for (int i = 0; i < n; ++i) {
        t.v[i] = views[i];
        t.v[i].HW = views[i].W * views[i].H;
        t.v[i].blk0 = blk;
        blk += (t.v[i].HW + tc::kRows - 1) / tc::kRows;
    }
    t.n_blocks = blk;
    if (t.n_blocks == 0) return cudaSuccess;
    size_t smem = 0;
    int per_sm = 0;
    if (!tc_launch_shape(&smem, &per_sm)) return cudaErrorInvalidConfiguration;
    // the diagnostic instantiation is launched with the production one's
    // shape (its shared-memory padding keeps the same residency cap)
    auto kernel = no_mma ? k_shade_fwd_tc<true> : k_shade_fwd_tc<false>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kernel<<<persistent_grid(t.n_blocks, per_sm), tc::kRows, smem, st>>>(t, params, status);
    note_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_shade_bwd(const ShadeView* views, int n, int S, const float* params, bool overwrite,
                             float* partial, int grid, float* grad_params, cudaStream_t st) {
    ShadeTable t;
    fill_table(t, views, n, S, overwrite);
    if (t.n_blocks > 0 && S > 0) {
        const size_t smem = sizeof(BwdSmem);
        cudaError_t e = cudaFuncSetAttribute(k_shade_bwd, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        const int g = grid < t.n_blocks ? grid : t.n_blocks;
        k_shade_bwd<<<g, kBwdThreads, smem, st>>>(t, params, partial);
        note_launches(1);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        if (grad_params) {
            k_shade_finish<<<(kParams + 31) / 32, 32 * kFinWarps, 0, st>>>(partial, g, grad_params, overwrite ? 1 : 0);
            note_launches(1);
        }
    } else if (grad_params && overwrite) {
        return cudaMemsetAsync(grad_params, 0, sizeof(float) * kParams, st);
    }
    return cudaGetLastError();
}

}  // namespace ds
