// ds_common.cuh -- internal definitions of the CUDA library (not installed).
//
// Pinned arithmetic: every floating-point step that decides an integer
// (coverage, the depth order, alpha > tau) uses explicit round-to-nearest
// intrinsics (__fmul_rn, __fadd_rn, __fmaf_rn, __fdiv_rn) so that neither the
// compiler's FMA contraction nor approximate division can change a result
// bit.  Gradient arithmetic is free-form FP32.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/diffsoup.h"

namespace ds {

constexpr int kTilePix = 256;        // pixels per tile (one thread each); the
                                     // tile is tile_w x (256 / tile_w) pixels
constexpr int kChunk = 256;          // staging capacity of the tile kernels (triangles per round)
constexpr int kSampleGroup = 4;      // samples sharing one Philox block
constexpr float kGuard = 16384.0f;   // screen-space guard band (pixels)

// Camera as the kernels see it.
struct DevCam {
    float fx, fy, cx, cy;
    float R[9];
    float t[3];
    float near_z;
};

// Background colour (C-1 channels) of samples where no fragment survives.
struct Bg {
    float c[DS_MAX_CHANNELS];
};

// Per-view parameters, passed by value in the kernel parameter space.
struct ViewDesc {
    DevCam cam;
    int W, H, tiles_x, tiles_y;
    int tile_base;   // global index of this view's first tile
    int item_base;   // first work item (tiles x sample groups)
    uint32_t seed_lo, seed_hi;
    ds_gbuf* gbuf;
    float* color;
    int32_t* n_front;
    const float* grad_color;
    const float* score_w;
    const float* target;   // fused training pass: [C-1][H][W] target image
    // The view's soup and the index of its first set-up record: the call's
    // soup and v * T in a single-soup call; one soup per view in a
    // multi-soup forward (ds_raster_forward_multi), records concatenated.
    const float* s_verts;
    float* s_act;
    float* s_act_a;
    int s_T;
    long long rec_base;
};

struct ViewTable {
    int n;          // views
    int S;          // samples per pixel
    int n_groups;   // ceil(S / 4)
    int n_items;    // total work items
    int tile_w, tile_h;   // tile shape in pixels (8x32, 16x16 or 32x8)
    int chunk;      // triangles staged per round in the tile kernels (<= 256)
    // Optional device-resident cameras (ds_camera[n]) and seeds (uint64[n]):
    // when set they replace v[i].cam and v[i].seed_*, so that a captured
    // CUDA graph can render views chosen after capture.
    const ds_camera* dcam;
    const unsigned long long* dseed;
    ViewDesc v[DS_MAX_VIEWS];
};

// Camera and seed of view v (device table if present, else the parameters).
__device__ __forceinline__ const DevCam& view_cam(const ViewTable& vt, int v) {
    if (vt.dcam) return *reinterpret_cast<const DevCam*>(reinterpret_cast<const char*>(vt.dcam + v) + 8);
    return vt.v[v].cam;
}
__device__ __forceinline__ uint2 view_seed(const ViewTable& vt, int v) {
    if (vt.dseed) {
        const unsigned long long s = vt.dseed[v];
        return make_uint2((uint32_t)s, (uint32_t)(s >> 32));
    }
    return make_uint2(vt.v[v].seed_lo, vt.v[v].seed_hi);
}

// Triangle set-up of one (view, triangle), 64 bytes.  Edge i runs from vertex
// i+1 to vertex i+2; E_i(X, Y) = A_i X + B_i Y + C_i in 1/256-pixel units is
// oriented positive inside, with the fill-rule bias folded into C (a pixel
// centre is covered iff every biased E_i >= 0).  k_i = (1/w_i) / |2 area|.
struct __align__(16) SetupRec {
    int32_t A[3];
    int32_t B[3];
    long long C[3];
    float k[3];
    uint32_t bias;   // bit i set: edge i is not owned (bias 1 folded into C_i); bits 3..19: kSmallTri
};
// Bit 3: no edge is longer than 63 pixels in x or y; bits 4..11 and 12..19 are
// then 1 + the cell of 64 x 64 pixels of vertex 0.  Within that cell and the
// eight around it, which hold every pixel that the triangle covers, the edge
// values fit int32: |2 area| + 256 * 2 * 128 * max(|A|, |B|) < 2^31.
constexpr uint32_t kSmallTri = 8u;
constexpr int kSmallEdge = 63 * 256, kCellBits = 14;
static_assert(2LL * kSmallEdge * kSmallEdge + 256LL * 2 * 128 * kSmallEdge + 1 < 1LL << 31, "int32 edge values");
static_assert(sizeof(SetupRec) == 64, "SetupRec must be 64 bytes");

// Continuous (unsnapped) geometry of one (view, triangle) for the vertex
// gradients.  Computed once per backward pass in double-float arithmetic
// (about 2^-46 relative); quantities from which the per-pixel code later
// takes small differences of large values are kept as (hi, lo) float pairs,
// so that the per-pixel arithmetic stays FP32 with compensated steps.
// 208 bytes.
struct __align__(16) GeomRec {
    float2 sx[3], sy[3];   // screen position of each vertex (hi + lo)
    float jx[3][2];        // d sx / d(x_c, z_c): fx / z, -fx x / z^2
    float jy[3][2];        // d sy / d(y_c, z_c): fy / z, -fy y / z^2
    float2 n[3];           // e1 x e2 in camera space (hi + lo)
    float2 m1[3];          // e2 x V0
    float2 m2[3];          // V0 x e1
    float e1[3], e2[3], v0[3];
    float pad;
};
static_assert(sizeof(GeomRec) == 208, "GeomRec must be 208 bytes");

// Soup as the kernels see it.
struct SoupDev {
    const float* verts;   // [T][3][3]
    const float* tex;     // [T][V][C] logits
    float* act;           // [T][V][C] sigmoid(tex)
    float* act_a;         // [T][V]    opacity plane of act
    int T, N, C, V;
};

// ----------------------------------------------------------------- pinned math

// exp(x): Cody-Waite reduction x = k ln2 + r (ln2 = 16-bit head + float
// tail), degree-7 Taylor polynomial of e^r (coefficients 1/n! rounded to
// float) by Horner with fused multiply-adds, scaling by 2^k in two exact
// power-of-two factors.
__device__ __forceinline__ float pow2i(int k) { return __int_as_float((k + 127) << 23); }

__device__ __forceinline__ float exp_poly(float r) {
    float p = 0x1.a01a02p-13f;
    p = __fmaf_rn(p, r, 0x1.6c16c2p-10f);
    p = __fmaf_rn(p, r, 0x1.111112p-7f);
    p = __fmaf_rn(p, r, 0x1.555556p-5f);
    p = __fmaf_rn(p, r, 0x1.555556p-3f);
    p = __fmaf_rn(p, r, 0.5f);
    p = __fmaf_rn(p, r, 1.0f);
    return __fmaf_rn(p, r, 1.0f);
}

__device__ __forceinline__ float pinned_exp(float x) {
    const float t = __fmul_rn(x, 0x1.715476p+0f);
    if (fabsf(x) < 80.0f) {
        // The same value without the conversions of rintf and int (both on the
        // quarter-rate pipe of the special functions): adding and taking off
        // 1.5 * 2^23 rounds t to an integer (to even), whose two's complement
        // then sits in the low bits; e^r 2^k stays normal here, so that one
        // scaling is exact like the two of the general form.
        const float m = __fadd_rn(t, 0x1.8p+23f);
        const float kf = __fsub_rn(m, 0x1.8p+23f);
        const float r = __fmaf_rn(-kf, 0x1.7f7d1cp-20f, __fmaf_rn(-kf, 0x1.62e400p-1f, x));
        return __fmul_rn(exp_poly(r), __int_as_float((__float_as_int(m) + 127) << 23));
    }
    if (x != x) return x;
    if (x >= 0x1.62e430p+6f) return __int_as_float(0x7f800000);
    if (x < -0x1.9fe368p+6f) return 0.0f;
    const float kf = rintf(t);
    const float r = __fmaf_rn(-kf, 0x1.7f7d1cp-20f, __fmaf_rn(-kf, 0x1.62e400p-1f, x));
    const int k = (int)kf;
    const int k1 = k / 2, k2 = k - k1;
    return __fmul_rn(__fmul_rn(exp_poly(r), pow2i(k1)), pow2i(k2));
}

// Sigmoid of Sec. 3.3, applied per feature vertex before rasterisation.  The
// correctly rounded reciprocal is the IEEE division 1 / (1 + e^-x).
__device__ __forceinline__ float pinned_sigmoid(float th) { return __frcp_rn(__fadd_rn(1.0f, pinned_exp(-th))); }

// Four of them, the same bits: the range test and its branch once, e^-x as
// packed pairs (the reduction and the polynomial of pinned_exp, each operation
// with the same rounding).
__device__ __forceinline__ float2 splat(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 exp_neg_near(float2 th) {   // e^-th, |th| < 80
    const float2 x = make_float2(-th.x, -th.y);
    const float2 m = __fadd2_rn(__fmul2_rn(x, splat(0x1.715476p+0f)), splat(0x1.8p+23f));
    const float2 kf = __fadd2_rn(m, splat(-0x1.8p+23f));
    const float2 r = __ffma2_rn(kf, splat(-0x1.7f7d1cp-20f), __ffma2_rn(kf, splat(-0x1.62e400p-1f), x));
    float2 p = splat(0x1.a01a02p-13f);
    p = __ffma2_rn(p, r, splat(0x1.6c16c2p-10f));
    p = __ffma2_rn(p, r, splat(0x1.111112p-7f));
    p = __ffma2_rn(p, r, splat(0x1.555556p-5f));
    p = __ffma2_rn(p, r, splat(0x1.555556p-3f));
    p = __ffma2_rn(p, r, splat(0.5f));
    p = __ffma2_rn(p, r, splat(1.0f));
    p = __ffma2_rn(p, r, splat(1.0f));
    return __fmul2_rn(p, make_float2(__int_as_float((__float_as_int(m.x) + 127) << 23),
                                     __int_as_float((__float_as_int(m.y) + 127) << 23)));
}
__device__ __forceinline__ float4 pinned_sigmoid4(float4 th) {
    if (!(fabsf(th.x) < 80.0f && fabsf(th.y) < 80.0f && fabsf(th.z) < 80.0f && fabsf(th.w) < 80.0f))
        return make_float4(pinned_sigmoid(th.x), pinned_sigmoid(th.y), pinned_sigmoid(th.z), pinned_sigmoid(th.w));
    const float2 a = __fadd2_rn(splat(1.0f), exp_neg_near(make_float2(th.x, th.y)));
    const float2 b = __fadd2_rn(splat(1.0f), exp_neg_near(make_float2(th.z, th.w)));
    return make_float4(__frcp_rn(a.x), __frcp_rn(a.y), __frcp_rn(b.x), __frcp_rn(b.y));
}

// Philox4x32-10 block (Salmon et al., SC'11).
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint32_t lo0 = 0xD2511F53u * c.x, hi0 = __umulhi(0xD2511F53u, c.x);
        const uint32_t lo1 = 0xCD9E8D57u * c.z, hi1 = __umulhi(0xCD9E8D57u, c.z);
        c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    return c;
}

// Mesh-colour cell: the micro-triangle of the N-subdivided triangle that
// holds barycentrics (b1, b2).  Grid vertex (i, j), i + j <= N, sits at
// barycentrics (1 - (i+j)/N, i/N, j/N) and has index j(N+1) - j(j-1)/2 + i.
struct Cell {
    int k0, k1, k2;   // corner texel indices
    float wa, wb;     // value = a0 + wa (a1 - a0) + wb (a2 - a0)
    bool lower;       // lower (i,j),(i+1,j),(i,j+1) or upper micro-triangle
};

__device__ __forceinline__ int texel_index(int N, int i, int j) {
    return ((j * (2 * N + 3 - j)) >> 1) + i;   // j (N + 1) - j (j - 1) / 2 + i
}

// (i, j) of vertex v of the N-subdivided grid (rows of constant j).
__device__ __forceinline__ void texel_ij(int N, int v, int& i, int& j) {
    const float b = (float)(2 * N + 3);
    int jj = (int)floorf(0.5f * (b - sqrtf(b * b - 8.0f * (float)v)));
    jj = jj < 0 ? 0 : (jj > N ? N : jj);
    while (jj > 0 && texel_index(N, 0, jj) > v) --jj;
    while (jj < N && texel_index(N, 0, jj + 1) <= v) ++jj;
    j = jj;
    i = v - texel_index(N, 0, jj);
}

// Rounding towards minus infinity into int32 saturates (NaN gives 0), so the
// clamps also hold for barycentrics outside the triangle; the corner
// indices follow from the cell's first one: row j + 1 starts N + 1 - j
// texels after the same column of row j.
__device__ __forceinline__ Cell find_cell(int N, float b1, float b2) {
    const float Nf = (float)N;
    const float u = __fmul_rn(Nf, b1), v = __fmul_rn(Nf, b2);
    const int i = max(0, min(__float2int_rd(u), N - 1));
    const int j = max(0, min(__float2int_rd(v), N - 1 - i));
    const float fu = __fsub_rn(u, (float)i), fv = __fsub_rn(v, (float)j);
    Cell c;
    c.lower = (__fadd_rn(fu, fv) <= 1.0f) || (i + j == N - 1);
    const int k = texel_index(N, i, j), row = N + 1 - j;
    c.k0 = c.lower ? k : k + row + 1;
    c.k1 = k + (c.lower ? 1 : row);
    c.k2 = k + (c.lower ? row : 1);
    c.wa = c.lower ? fu : __fsub_rn(1.0f, fu);
    c.wb = c.lower ? fv : __fsub_rn(1.0f, fv);
    return c;
}

__device__ __forceinline__ float interp(float a0, float a1, float a2, float wa, float wb) {
    return __fmaf_rn(wb, __fsub_rn(a2, a0), __fmaf_rn(wa, __fsub_rn(a1, a0), a0));
}

// The same for two channels, packed (a - b as fma(b, -1, a): one rounding).
__device__ __forceinline__ float2 interp2(float2 a0, float2 a1, float2 a2, float2 wa, float2 wb) {
    return __ffma2_rn(wb, __ffma2_rn(a0, splat(-1.0f), a2), __ffma2_rn(wa, __ffma2_rn(a0, splat(-1.0f), a1), a0));
}

// Pinned perspective-correct fragment from the three oriented (unbiased)
// edge values: q_i = E_i k_i, rho = (q0 + q1) + q2 (inverse depth).
struct Frag {
    float q1, q2, rho;
};

__device__ __forceinline__ Frag edge_frag(float e0, float e1, float e2, float k0, float k1, float k2) {
    Frag f;
    const float q0 = __fmul_rn(e0, k0);
    f.q1 = __fmul_rn(e1, k1);
    f.q2 = __fmul_rn(e2, k2);
    f.rho = __fadd_rn(__fadd_rn(q0, f.q1), f.q2);
    return f;
}

// (rho, t) is in front of (rho2, t2): larger inverse depth, then lower index.
__device__ __forceinline__ bool in_front(float rho, int t, float rho2, int t2) {
    return rho > rho2 || (rho == rho2 && t < t2);
}

// Exact covered test and oriented edge values of one set-up record at a
// pixel (int64 arithmetic).
__device__ __forceinline__ bool cover_exact(const SetupRec& r, int px, int py, long long E[3]) {
    const long long X = 256LL * px + 128, Y = 256LL * py + 128;
    bool cov = true;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const long long eb = (long long)r.A[i] * X + (long long)r.B[i] * Y + r.C[i];
        cov = cov && (eb >= 0);
        E[i] = eb + ((r.bias >> i) & 1u);
    }
    return cov;
}

// The same with the values rounded once, in int32 where the record and the
// pixel allow it.
__device__ __forceinline__ bool cover_near(const SetupRec& r, int px, int py, float e[3]) {
    const unsigned dx = (unsigned)((px >> 6) + 2) - ((r.bias >> 4) & 255u);
    const unsigned dy = (unsigned)((py >> 6) + 2) - ((r.bias >> 12) & 255u);
    if ((r.bias & kSmallTri) && dx <= 2u && dy <= 2u) {
        const uint32_t X = 256u * px + 128u, Y = 256u * py + 128u;
        int low = 0;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const int eb = (int)((uint32_t)r.A[i] * X + ((uint32_t)r.B[i] * Y + (uint32_t)r.C[i]));
            low |= eb;
            e[i] = __int2float_rn(eb + (int)((r.bias >> i) & 1u));
        }
        return low >= 0;
    }
    long long E[3];
    const bool cov = cover_exact(r, px, py, E);
#pragma unroll
    for (int i = 0; i < 3; ++i) e[i] = __ll2float_rn(E[i]);
    return cov;
}

// ------------------------------------------------------------ compensated FP32
// TwoSum (Knuth): s + err == a + b exactly.
__device__ __forceinline__ float two_sum(float a, float b, float& err) {
    const float s = __fadd_rn(a, b);
    const float bp = __fsub_rn(s, a);
    const float ap = __fsub_rn(s, bp);
    err = __fadd_rn(__fsub_rn(a, ap), __fsub_rn(b, bp));
    return s;
}

// a*b - c*d with one rounding error (Kahan's algorithm with fused multiply-add).
__device__ __forceinline__ float diff_prod(float a, float b, float c, float d) {
    const float w = __fmul_rn(c, d);
    const float e = __fmaf_rn(-c, d, w);
    const float f = __fmaf_rn(a, b, -w);
    return __fadd_rn(f, e);
}

// Dot product of an exact FP32 vector with a (hi, lo) vector, evaluated as if
// in twice the working precision (Ogita, Rump, Oishi, "Accurate sum and dot
// product", SIAM J. Sci. Comput. 26(6), 2005: Dot2 with TwoProduct by FMA).
__device__ __forceinline__ float dot2(float x0, float x1, float x2, const float2* y) {
    float p = __fmul_rn(x0, y[0].x);
    float c = __fadd_rn(__fmaf_rn(x0, y[0].x, -p), __fmul_rn(x0, y[0].y));
    float s = p, t;
    p = __fmul_rn(x1, y[1].x);
    s = two_sum(s, p, t);
    c = __fadd_rn(c, __fadd_rn(t, __fadd_rn(__fmaf_rn(x1, y[1].x, -p), __fmul_rn(x1, y[1].y))));
    p = __fmul_rn(x2, y[2].x);
    s = two_sum(s, p, t);
    c = __fadd_rn(c, __fadd_rn(t, __fadd_rn(__fmaf_rn(x2, y[2].x, -p), __fmul_rn(x2, y[2].y))));
    return __fadd_rn(s, c);
}

// Pinned direction (z = 1) of the camera ray through screen point (x, y)
// (a pixel centre or the midpoint of two; both exact in FP32).
__device__ __forceinline__ void pinned_ray(const DevCam& c, float x, float y, float& dx, float& dy) {
    dx = __fdiv_rn(__fsub_rn(x, c.cx), c.fx);
    dy = __fdiv_rn(__fsub_rn(y, c.cy), c.fy);
}

__device__ __forceinline__ SetupRec load_rec(const SetupRec* p) {
    const int4* q = reinterpret_cast<const int4*>(p);
    SetupRec r;
    int4* d = reinterpret_cast<int4*>(&r);
    d[0] = __ldg(q);
    d[1] = __ldg(q + 1);
    d[2] = __ldg(q + 2);
    d[3] = __ldg(q + 3);
    return r;
}

// Adam (Sec. 3.4; supplementary "Hyperparameters"): the step's scalars, with
// the bias corrections c1 = 1/(1 - b1^t), c2 = 1/(1 - b2^t) formed on the host.
struct AdamDev {
    float lr, b1, b2, eps, c1, c2;
};

// One value's Adam step:
//   m <- b1 m + (1 - b1) g,  v <- b2 v + (1 - b2) g^2,
//   x <- x - lr (m c1) / (sqrt(v c2) + eps),
// every rounding fixed by an explicit intrinsic, so that each kernel that
// applies it (the optimiser step, the fused gradient finishes) gives the
// same bits for the same gradient.
__device__ __forceinline__ void adam_apply(float& x, float& m, float& v, float g, const AdamDev& a) {
    m = __fmaf_rn(a.b1, m, __fmul_rn(1.0f - a.b1, g));
    v = __fmaf_rn(a.b2, v, __fmul_rn(1.0f - a.b2, __fmul_rn(g, g)));
    const float u = __fdiv_rn(__fmul_rn(a.lr, __fmul_rn(m, a.c1)), __fadd_rn(__fsqrt_rn(__fmul_rn(v, a.c2)), a.eps));
    x = __fsub_rn(x, u);
}

}  // namespace ds
