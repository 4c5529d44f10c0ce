// ds_ssim.cu -- the photometric loss lambda L1 + (1 - lambda) L_SSIM (Eq. 10,
// Sec. 3.4) per pixel, fused with its upstream gradients for the backward
// pass.  Per channel, SSIM uses an 11 x 11 Gaussian window (sigma 1.5,
// normalised), zero padding outside the image, C1 = 0.01^2, C2 = 0.03^2.  The
// per-pixel loss
//     ell_p = lambda mean_c |x - y| + (1 - lambda)(1 - mean_c ssim_c(p))
// is written as the score weight (scale * ell_p) and the colour gradient is
// that of scale * sum_p ell_p:
//     d/dx(q) = lambda sign(x - y)/C - (1 - lambda)/C [w*G1 + 2 x w*G2 + y w*G3](q),
// G1..G3 the derivatives of ssim with respect to the raw moments w*x, w*x^2,
// w*(xy) at each p (zero outside the image).
//
// One CTA marches down a strip of 118 columns, 16 rows a step, one channel
// after the other.  The five moments (separable blur) need rows 5 above and
// below, the blur of G1..G3 back onto the image 5 more: the horizontally
// blurred rows that the next step needs again (10 of 26) stay in shared
// memory, so that no row of a segment is blurred twice.  118 + 10 moment
// columns are 128: with 512 threads every stage is one task per thread -- four
// neighbouring outputs of a row (horizontal) or of a column (vertical) that
// share their window.  No intermediate map reaches HBM.
//
// Tiles of 64 x 16 pixels on their own blur 2.6 rows per row horizontally and
// 1.9 vertically (549 M against 310 M warp instructions on four 1080p images
// of three channels).  There 735 -> 527 us; issue active 55%, FMA pipe 31% (a
// packed FMA takes two of its cycles), shared-memory wavefronts 50% of their
// peak, one CTA of 16 warps per SM.
//
// The blurs are issue-bound, so their operands are interleaved in shared
// memory as pairs that take the same weight -- (x, y), (x^2, y^2), (G1, G2)
// -- and each tap of a pair is one packed FP32 multiply-add (fma.rn.f32x2,
// the weight duplicated in both halves); x y and G3 stay scalar.
#include <cmath>
#include <new>

#include "ds_internal.h"

namespace ds {

namespace {

constexpr int kR = 5, kTaps = 2 * kR + 1;
constexpr int kThreads = 512;
constexpr int kStep = 16;                 // rows per step
constexpr int kKeep = kStep + 2 * kR;     // rows of a vertical pass's input
constexpr int kTX = 118;                  // output columns of a strip
constexpr int kMX = kTX + 2 * kR;         // moment columns (128)
constexpr int kIX = kTX + 4 * kR;         // input columns (138)
constexpr int kGX = 132;                  // G row stride: the last task of a row reads two columns past the strip's
constexpr int kHX = 120;                  // row stride of the blurred G
constexpr int kMaxSteps = 9;              // steps of the longest segment
constexpr int kMaxRows = kStep * kMaxSteps - 4 * kR;   // its output rows (124)
constexpr float kC1 = 0.01f * 0.01f, kC2 = 0.03f * 0.03f;

struct SsimView {
    const float* color;    // [S][Co][H][W]
    const float* target;   // [Co][H][W]
    float* grad_color;     // [S][Co][H][W] or null
    float* score_w;        // [S][H][W] or null
    int W, H, strips, cta0;   // strips or tiles per row, first CTA of this view (all samples)
};

struct SsimTable {
    int n, S, Co, rows;   // output rows of a segment
    float lambda, scale;
    float w[kR + 1];   // half of the symmetric window, centre last
    SsimView v[DS_MAX_VIEWS];
};

struct SsimSmem {
    float2 XY[2][kStep][kIX];    // (x, y) of this step's and the next step's rows
    float2 ha[kKeep][kMX];       // horizontal pass of (x, y): 10 rows kept, 16 new
    float2 hb[kKeep][kMX];       // of (x^2, y^2)
    float hc[kKeep][kMX];        // of x y
    float2 Ga[kStep][kGX];       // (G1, G2)
    float Gb[kStep][kGX];        // G3
    float2 ga[kKeep][kHX];       // horizontal pass of (G1, G2): 10 rows kept, 16 new
    float gb[kKeep][kHX];        // of G3
    float P[kMaxRows][kTX];      // ssim, summed over channels
};
static_assert(sizeof(SsimSmem) <= 227 * 1024, "shared memory of one CTA");
static_assert(kMX == 128 && kThreads == 4 * kMX && kThreads == 32 * kStep, "one task per thread");

// Columns of the pair arrays are stored with bit 1 flipped where bit 4 is set:
// the horizontal passes read and write 16 bytes per lane at a stride of 32,
// which would meet each bank twice.
__device__ __forceinline__ int swz(int col) { return col ^ ((col >> 3) & 2); }

__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

// Step s of a channel (rows relative to the segment's first output row y0):
// input rows y0 - 10 + 16 s + i; moments, ssim and G of rows y0 - 15 + 16 s + i;
// outputs of rows y0 - 20 + 16 s + i, i = 0..15.  Rows of a vertical pass that
// reach back before the channel's first step hold leftovers; what comes of
// them is never read.
__global__ void __launch_bounds__(kThreads, 1) k_loss_l1_ssim(const __grid_constant__ SsimTable t, float* __restrict__ loss) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SsimSmem& sm = *reinterpret_cast<SsimSmem*>(smem_raw);
    // view, sample, segment, strip of this CTA
    int item = blockIdx.x, vi = 0;
    while (vi + 1 < t.n && t.v[vi + 1].cta0 <= item) ++vi;
    const SsimView& V = t.v[vi];
    item -= V.cta0;
    const int per = V.strips * ((V.H + t.rows - 1) / t.rows);
    const int s = item / per, sl = item - s * per;
    const int x0 = (sl % V.strips) * kTX, y0 = (sl / V.strips) * t.rows;
    const int rows = min(t.rows, V.H - y0), steps = (rows + 4 * kR + kStep - 1) / kStep;
    const size_t HW = (size_t)V.W * V.H;
    const int tid = threadIdx.x;
    const int hr = tid >> 5, hq = 4 * (tid & 31);   // horizontal task: row, first column
    const int vq = tid & (kMX - 1), vr = 4 * (tid >> 7);   // vertical task: column, first row
    const int vs = swz(vq);
    const int flip = (hq >> 4) & 1, lim = 8 - ((hq >> 1) & 7);
    // the m-th 16 bytes of a horizontal task's window
    const auto chunk = [&](const float2* row, int m) {
        const int f = flip ^ (m >= lim ? 1 : 0);
        return reinterpret_cast<const float4*>(row)[(hq >> 1) + m + (m & 1 ? -f : f)];
    };

    for (int k = tid; k < rows * kTX; k += kThreads) (&sm.P[0][0])[k] = 0.f;
    // The window is symmetric: six weights, in both halves of a pair.
    float2 wd[kR + 1];
#pragma unroll
    for (int j = 0; j <= kR; ++j) wd[j] = make_float2(t.w[j], t.w[j]);
    const auto w2 = [&](int tap) { return wd[tap <= kR ? tap : 2 * kR - tap]; };
    // A step's input rows are loaded into registers a step ahead: a warp per row.
    constexpr int kLoads = (kIX + 31) / 32;
    const int lane = tid & 31, lx = x0 - 2 * kR + lane;
    float px[kLoads], py[kLoads];
    const auto load_regs = [&](int c, int step) {
        const int gy = y0 - 2 * kR + kStep * step + hr;
        const bool row = gy >= 0 && gy < V.H;
        const float* xs = V.color + ((size_t)s * t.Co + c) * HW + (size_t)(row ? gy : 0) * V.W + lx;
        const float* ys = V.target + (size_t)c * HW + (size_t)(row ? gy : 0) * V.W + lx;
#pragma unroll
        for (int i = 0; i < kLoads; ++i) {
            const bool in = row && (unsigned)(lx + 32 * i) < (unsigned)V.W && (32 * i + 32 <= kIX || lane < kIX - 32 * i);
            px[i] = in ? __ldg(xs + 32 * i) : 0.f;
            py[i] = in ? __ldg(ys + 32 * i) : 0.f;
        }
    };
    const auto store_regs = [&](int buf) {
#pragma unroll
        for (int i = 0; i < kLoads; ++i)
            if (32 * i + 32 <= kIX || lane < kIX - 32 * i) sm.XY[buf][hr][swz(lane) + 32 * i] = make_float2(px[i], py[i]);
    };
    load_regs(0, 0);
    store_regs(0);
    __syncthreads();
    int buf = 0;
#pragma unroll 1
    for (int it = 0, c = 0, st = 0; it < t.Co * steps; ++it) {
        const bool last_step = st + 1 == steps;
        const int nc = last_step ? c + 1 : c, ns = last_step ? 0 : st + 1;
        if (nc < t.Co) load_regs(nc, ns);
        // ---- horizontal pass of the five moments over the new rows
        {
            float2 A[4] = {}, B[4] = {};
            float C[4] = {};
#pragma unroll
            for (int jj = 0; jj < kTaps + 3; jj += 2) {
                const float4 in = chunk(sm.XY[buf][hr], jj / 2);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float2 v = h ? make_float2(in.z, in.w) : make_float2(in.x, in.y);
                    const float2 sq = __fmul2_rn(v, v);
                    const float xy = v.x * v.y;
#pragma unroll
                    for (int o = 0; o < 4; ++o) {
                        const int tap = jj + h - o;
                        if (tap < 0 || tap >= kTaps) continue;
                        A[o] = ffma2(w2(tap), v, A[o]);
                        B[o] = ffma2(w2(tap), sq, B[o]);
                        C[o] = fmaf(w2(tap).x, xy, C[o]);
                    }
                }
            }
            float4* a = reinterpret_cast<float4*>(&sm.ha[2 * kR + hr][hq]);
            float4* b = reinterpret_cast<float4*>(&sm.hb[2 * kR + hr][hq]);
            a[flip] = make_float4(A[0].x, A[0].y, A[1].x, A[1].y);
            a[1 - flip] = make_float4(A[2].x, A[2].y, A[3].x, A[3].y);
            b[flip] = make_float4(B[0].x, B[0].y, B[1].x, B[1].y);
            b[1 - flip] = make_float4(B[2].x, B[2].y, B[3].x, B[3].y);
            *reinterpret_cast<float4*>(&sm.hc[2 * kR + hr][hq]) = make_float4(C[0], C[1], C[2], C[3]);
        }
        __syncthreads();
        // ---- the blurred G's last ten rows are kept
        {
            constexpr int n2 = 2 * kR * kHX / 2, n1 = 2 * kR * kHX / 4;   // float4 of the pair array, of the scalar one
            float4* a = reinterpret_cast<float4*>(&sm.ga[0][0]) + tid;
            float4* b = reinterpret_cast<float4*>(&sm.gb[0][0]) + tid;
            a[0] = a[kStep * kHX / 2];
            if (tid < n1) b[0] = b[kStep * kHX / 4];
            if (tid < n2 - kThreads) a[kThreads] = a[kThreads + kStep * kHX / 2];
        }
        // ---- vertical pass, ssim and its derivatives w.r.t. the raw moments
        if (st > 0 || vr + 3 >= 2 * kR) {
            float2 A[4] = {}, B[4] = {};
            float C[4] = {};
#pragma unroll
            for (int j = 0; j < kTaps + 3; ++j) {
                const float2 ha = sm.ha[vr + j][vs], hb = sm.hb[vr + j][vs];
                const float hc = sm.hc[vr + j][vq];
#pragma unroll
                for (int o = 0; o < 4; ++o) {
                    const int tap = j - o;
                    if (tap < 0 || tap >= kTaps) continue;
                    A[o] = ffma2(w2(tap), ha, A[o]);
                    B[o] = ffma2(w2(tap), hb, B[o]);
                    C[o] = fmaf(w2(tap).x, hc, C[o]);
                }
            }
#pragma unroll
            for (int o = 0; o < 4; ++o) {
                const int r = vr + o, ry = kStep * st - 3 * kR + r;   // row within the segment
                float g1 = 0.f, g2 = 0.f, g3 = 0.f;
                if ((unsigned)(x0 - kR + vq) < (unsigned)V.W && (unsigned)(y0 + ry) < (unsigned)V.H) {
                    const float mx = A[o].x, my = A[o].y;
                    const float A_ = 2.f * mx * my + kC1;
                    const float B_ = 2.f * (C[o] - mx * my) + kC2;
                    const float Cc = mx * mx + my * my + kC1;
                    const float D = (B[o].x - mx * mx) + (B[o].y - my * my) + kC2;
                    // one reciprocal, 1/(Cc D)^2, gives ssim and its quotients by A, B, Cc, D
                    const float ab = A_ * B_, cd = Cc * D;
                    const float inv = 1.0f / (cd * cd);
                    const float ssim = ab * cd * inv;
                    const float sA = B_ * cd * inv, sB = A_ * cd * inv;   // ssim / A, ssim / B
                    const float sCc = ab * D * inv, sD = ab * Cc * inv;    // ssim / Cc, ssim / D
                    const float dmu = 2.f * my * sA - 2.f * mx * sCc;
                    const float dvar = -sD;
                    const float dcov = 2.f * sB;
                    g1 = dmu - 2.f * mx * dvar - my * dcov;
                    g2 = dvar;
                    g3 = dcov;
                    if ((unsigned)ry < (unsigned)rows && (unsigned)(vq - kR) < (unsigned)kTX)
                        sm.P[ry][vq - kR] += ssim;
                }
                sm.Ga[r][vs] = make_float2(g1, g2);
                sm.Gb[r][vq] = g3;
            }
        }
        __syncthreads();
        // ---- horizontal pass of G1..G3; the moments' last ten rows are kept;
        // the next step's input
        if (hq < kHX && (st > 0 || hr >= 2 * kR)) {
            float2 A[4] = {};
            float B[4] = {};
#pragma unroll
            for (int j4 = 0; j4 < kTaps + 3; j4 += 4) {
                const float4 gb = *reinterpret_cast<const float4*>(&sm.Gb[hr][hq + j4]);
                const float b4[4] = {gb.x, gb.y, gb.z, gb.w};
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    if (j4 + 2 * h >= kTaps + 3) continue;
                    const float4 ga = chunk(sm.Ga[hr], j4 / 2 + h);
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const float2 va = e ? make_float2(ga.z, ga.w) : make_float2(ga.x, ga.y);
#pragma unroll
                        for (int o = 0; o < 4; ++o) {
                            const int tap = j4 + 2 * h + e - o;
                            if (tap < 0 || tap >= kTaps) continue;
                            A[o] = ffma2(w2(tap), va, A[o]);
                            B[o] = fmaf(w2(tap).x, b4[2 * h + e], B[o]);
                        }
                    }
                }
            }
            float4* a = reinterpret_cast<float4*>(&sm.ga[2 * kR + hr][hq]);
            a[flip] = make_float4(A[0].x, A[0].y, A[1].x, A[1].y);
            a[1 - flip] = make_float4(A[2].x, A[2].y, A[3].x, A[3].y);
            *reinterpret_cast<float4*>(&sm.gb[2 * kR + hr][hq]) = make_float4(B[0], B[1], B[2], B[3]);
        }
        {
            constexpr int n2 = 2 * kR * kMX / 2, n1 = 2 * kR * kMX / 4;
            float4* a = reinterpret_cast<float4*>(&sm.ha[0][0]) + tid;
            float4* b = reinterpret_cast<float4*>(&sm.hb[0][0]) + tid;
            float4* c4 = reinterpret_cast<float4*>(&sm.hc[0][0]) + tid;
            a[0] = a[kStep * kMX / 2];
            b[0] = b[kStep * kMX / 2];
            if (tid < n1) c4[0] = c4[kStep * kMX / 4];
            if (tid < n2 - kThreads) {
                a[kThreads] = a[kThreads + kStep * kMX / 2];
                b[kThreads] = b[kThreads + kStep * kMX / 2];
            }
        }
        if (nc < t.Co) store_regs(buf ^ 1);
        __syncthreads();
        // ---- vertical pass onto the image: the gradient (the pixels' colours
        // once more, from L2)
        if (V.grad_color && st > 0 && vq < kTX) {
            const int ry0 = kStep * st - 4 * kR + vr;
            const bool col_in = x0 + vq < V.W;
            const long long pix = (long long)(y0 + ry0) * V.W + (x0 + vq);
            const float* xs = V.color + ((size_t)s * t.Co + c) * HW + pix;
            const float* ys = V.target + (size_t)c * HW + pix;
            float X[4], Y[4];
#pragma unroll
            for (int o = 0; o < 4; ++o) {
                const bool in = (unsigned)(ry0 + o) < (unsigned)rows && col_in;
                X[o] = in ? __ldg(xs + (size_t)o * V.W) : 0.f;
                Y[o] = in ? __ldg(ys + (size_t)o * V.W) : 0.f;
            }
            float2 A[4] = {};
            float B[4] = {};
#pragma unroll
            for (int j = 0; j < kTaps + 3; ++j) {
                const float2 ga = sm.ga[vr + j][vs];
                const float gb = sm.gb[vr + j][vq];
#pragma unroll
                for (int o = 0; o < 4; ++o) {
                    const int tap = j - o;
                    if (tap < 0 || tap >= kTaps) continue;
                    A[o] = ffma2(w2(tap), ga, A[o]);
                    B[o] = fmaf(w2(tap).x, gb, B[o]);
                }
            }
            float* gout = V.grad_color + (((size_t)s * t.Co + c) * HW + pix);
#pragma unroll
            for (int o = 0; o < 4; ++o) {
                const int ry = ry0 + o;
                if ((unsigned)ry >= (unsigned)rows || !col_in) continue;
                const float x = X[o], y = Y[o];
                const float d = x - y;
                const float dsum = A[o].x + 2.f * x * A[o].y + y * B[o];
                const float sg = d > 0.f ? 1.f : (d < 0.f ? -1.f : 0.f);
                const float gval = (t.lambda * sg - (1.f - t.lambda) * dsum) / (float)t.Co;
                gout[(size_t)o * V.W] = t.scale * gval;
            }
        }
        // no barrier here: the next horizontal pass touches nothing that the
        // vertical one reads
        buf ^= 1;
        c = nc;
        st = ns;
    }
    __syncthreads();   // P complete
    // per-pixel loss, score weight, total
    float acc = 0.f;
    if (vq < kTX && x0 + vq < V.W) {
        // the L1 sum from the colours again (L2): folding it into P channel by
        // channel saves this read (505 us) but rounds the sum another way.
        // Eight pixels per thread at a time for the loads' latency (one at a
        // time: 565 us)
        constexpr int kBatch = 8;
        const float* xs = V.color + (size_t)s * t.Co * HW + (size_t)y0 * V.W + x0 + vq;
        const float* ys = V.target + (size_t)y0 * V.W + x0 + vq;
        for (int r0 = tid / kMX; r0 < rows; r0 += 4 * kBatch) {
            float l1[kBatch] = {};
            for (int ch = 0; ch < t.Co; ++ch)
#pragma unroll
                for (int u = 0; u < kBatch; ++u) {
                    const size_t o = ch * HW + (size_t)min(r0 + 4 * u, rows - 1) * V.W;
                    l1[u] += fabsf(__ldg(xs + o) - __ldg(ys + o));
                }
#pragma unroll
            for (int u = 0; u < kBatch; ++u) {
                const int r = r0 + 4 * u;
                if (r >= rows) break;
                const float ell = t.lambda * l1[u] / (float)t.Co + (1.f - t.lambda) * (1.f - sm.P[r][vq] / (float)t.Co);
                if (V.score_w) V.score_w[(size_t)s * HW + (size_t)(y0 + r) * V.W + x0 + vq] = t.scale * ell;
                acc += ell;
            }
        }
    }
    if (loss) {
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, d);
        __shared__ float wsum[kThreads / 32];
        if ((tid & 31) == 0) wsum[tid >> 5] = acc;
        __syncthreads();
        if (tid == 0) {
            float tot = 0.f;
            for (int u = 0; u < kThreads / 32; ++u) tot += wsum[u];
            atomicAdd(loss, t.scale * tot);
        }
    }
}

// ---------------------------------------------------------------- small calls
// Calls of few tiles, and images whose strips or segments are mostly empty: one
// CTA per 64 x 16 tile, the whole halo blurred on its own.  More arithmetic per
// pixel than the march, but no chain of steps (4 views of 256 x 200: 34 against
// 40 us), and less of it past the image's edges (64 images of 512 x 16: 56
// against 101).
constexpr int kTileX = 64, kTileY = 16;
constexpr int kTileIX = kTileX + 4 * kR, kTileIY = kTileY + 4 * kR;   // staged input 84 x 36
constexpr int kTileMX = kTileX + 2 * kR, kTileMY = kTileY + 2 * kR;   // moment region 74 x 26

struct TileSmem {
    float2 XY[kTileIY][kTileIX];            // (x, y)
    union {
        struct {
            float2 a[kTileIY][kTileMX];     // horizontal pass of (x, y)
            float2 b[kTileIY][kTileMX];     // of (x^2, y^2)
            float c[kTileIY][kTileMX];      // of x y
        } hm;
        struct {
            float2 a[kTileMY][kTileX];     // horizontal pass of (G1, G2)
            float b[kTileMY][kTileX];      // of G3
        } hg;
    };
    float2 Ga[kTileMY][kTileMX];            // (G1, G2)
    float Gb[kTileMY][kTileMX];             // G3
    float St[kTileY][kTileX];             // ssim of the tile's pixels (this channel)
};

__global__ void __launch_bounds__(256) k_loss_l1_ssim_tile(const __grid_constant__ SsimTable t, float* __restrict__ loss) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TileSmem& sm = *reinterpret_cast<TileSmem*>(smem_raw);
    // view, sample, tile of this CTA
    int item = blockIdx.x, vi = 0;
    while (vi + 1 < t.n && t.v[vi + 1].cta0 <= item) ++vi;
    const SsimView& V = t.v[vi];
    item -= V.cta0;
    const int tiles = V.strips * ((V.H + kTileY - 1) / kTileY);
    const int s = item / tiles, tl = item - s * tiles;
    const int x0 = (tl % V.strips) * kTileX, y0 = (tl / V.strips) * kTileY;
    const size_t HW = (size_t)V.W * V.H;
    const int tid = threadIdx.x;

    // The window is symmetric: six weights, in both halves of a pair.
    float2 wd[kR + 1];
#pragma unroll
    for (int j = 0; j <= kR; ++j) wd[j] = make_float2(t.w[j], t.w[j]);
    const auto w2 = [&](int tap) { return wd[tap <= kR ? tap : 2 * kR - tap]; };
    float l1[4] = {0.f, 0.f, 0.f, 0.f}, ss[4] = {0.f, 0.f, 0.f, 0.f};
    // The staged inputs of channel c + 1 are loaded into registers while
    // channel c is processed (the loads' latency overlaps the blur passes).
    constexpr int kLoads = (kTileIX * kTileIY + 255) / 256;
    float px[kLoads], py[kLoads];
    auto load_regs = [&](int c) {
        const float* xs = V.color + ((size_t)s * t.Co + c) * HW;
        const float* ys = V.target + (size_t)c * HW;
#pragma unroll
        for (int i = 0; i < kLoads; ++i) {
            const int k = tid + 256 * i;
            const int r = k / kTileIX, q = k - r * kTileIX;
            const int gy = y0 - 2 * kR + r, gx = x0 - 2 * kR + q;
            const bool in = k < kTileIX * kTileIY && gx >= 0 && gx < V.W && gy >= 0 && gy < V.H;
            px[i] = in ? __ldg(xs + (size_t)gy * V.W + gx) : 0.f;
            py[i] = in ? __ldg(ys + (size_t)gy * V.W + gx) : 0.f;
        }
    };
    auto store_regs = [&]() {
#pragma unroll
        for (int i = 0; i < kLoads; ++i) {
            const int k = tid + 256 * i;
            if (k < kTileIX * kTileIY) {
                const int r = k / kTileIX, q = k - r * kTileIX;
                sm.XY[r][q] = make_float2(px[i], py[i]);
            }
        }
    };
    load_regs(0);
    store_regs();
    __syncthreads();
    for (int c = 0; c < t.Co; ++c) {
        if (c + 1 < t.Co) load_regs(c + 1);
        // 2. horizontal pass of the five moments, two neighbouring outputs
        //    per thread sharing their window (the pair starts at an even
        //    column: two input pairs per 16-byte read)
        for (int k = tid; k < kTileIY * (kTileMX / 2); k += 256) {
            const int r = k / (kTileMX / 2), q = 2 * (k - r * (kTileMX / 2));
            float2 A[2] = {}, B[2] = {};
            float Cxy[2] = {0.f, 0.f};
#pragma unroll
            for (int jj = 0; jj <= kTaps; jj += 2) {
                const float4 in = *reinterpret_cast<const float4*>(&sm.XY[r][q + jj]);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int j = jj + h;
                    const float2 v = h ? make_float2(in.z, in.w) : make_float2(in.x, in.y);
                    const float2 sq = __fmul2_rn(v, v);
                    const float xy = v.x * v.y;
#pragma unroll
                    for (int o = 0; o < 2; ++o) {
                        const int tap = j - o;
                        if (tap < 0 || tap >= kTaps) continue;
                        A[o] = ffma2(w2(tap), v, A[o]);
                        B[o] = ffma2(w2(tap), sq, B[o]);
                        Cxy[o] = fmaf(w2(tap).x, xy, Cxy[o]);
                    }
                }
            }
            *reinterpret_cast<float4*>(&sm.hm.a[r][q]) = make_float4(A[0].x, A[0].y, A[1].x, A[1].y);
            *reinterpret_cast<float4*>(&sm.hm.b[r][q]) = make_float4(B[0].x, B[0].y, B[1].x, B[1].y);
            *reinterpret_cast<float2*>(&sm.hm.c[r][q]) = make_float2(Cxy[0], Cxy[1]);
        }
        __syncthreads();
        // 3. vertical pass (two rows per thread), ssim and its derivatives
        //    w.r.t. the raw moments
        for (int k = tid; k < (kTileMY / 2) * kTileMX; k += 256) {
            const int rp = k / kTileMX, q = k - rp * kTileMX, r0 = 2 * rp;
            float2 A[2] = {}, B[2] = {};
            float Cxy[2] = {0.f, 0.f};
#pragma unroll
            for (int j = 0; j <= kTaps; ++j) {
                const float2 ha = sm.hm.a[r0 + j][q], hb = sm.hm.b[r0 + j][q];
                const float hc = sm.hm.c[r0 + j][q];
#pragma unroll
                for (int o = 0; o < 2; ++o) {
                    const int tap = j - o;
                    if (tap < 0 || tap >= kTaps) continue;
                    A[o] = ffma2(w2(tap), ha, A[o]);
                    B[o] = ffma2(w2(tap), hb, B[o]);
                    Cxy[o] = fmaf(w2(tap).x, hc, Cxy[o]);
                }
            }
#pragma unroll
            for (int o = 0; o < 2; ++o) {
                const int r = r0 + o;
                const int gy = y0 - kR + r, gx = x0 - kR + q;
                float g1 = 0.f, g2 = 0.f, g3 = 0.f;
                if (gx >= 0 && gx < V.W && gy >= 0 && gy < V.H) {
                    const float mx = A[o].x, my = A[o].y;
                    const float A_ = 2.f * mx * my + kC1;
                    const float B_ = 2.f * (Cxy[o] - mx * my) + kC2;
                    const float Cc = mx * mx + my * my + kC1;
                    const float D = (B[o].x - mx * mx) + (B[o].y - my * my) + kC2;
                    // one reciprocal, 1/(Cc D)^2, gives ssim and its quotients by A, B, Cc, D
                    const float ab = A_ * B_, cd = Cc * D;
                    const float inv = 1.0f / (cd * cd);
                    const float ssim = ab * cd * inv;
                    const float sA = B_ * cd * inv, sB = A_ * cd * inv;   // ssim / A, ssim / B
                    const float sCc = ab * D * inv, sD = ab * Cc * inv;    // ssim / Cc, ssim / D
                    const float dmu = 2.f * my * sA - 2.f * mx * sCc;
                    const float dvar = -sD;
                    const float dcov = 2.f * sB;
                    g1 = dmu - 2.f * mx * dvar - my * dcov;
                    g2 = dvar;
                    g3 = dcov;
                    if (r >= kR && r < kR + kTileY && q >= kR && q < kR + kTileX) sm.St[r - kR][q - kR] = ssim;
                }
                sm.Ga[r][q] = make_float2(g1, g2);
                sm.Gb[r][q] = g3;
            }
        }
        __syncthreads();
        // 4. horizontal pass of G1..G3 (over the moments' buffer), two
        //    outputs per thread
        for (int k = tid; k < kTileMY * (kTileX / 2); k += 256) {
            const int r = k / (kTileX / 2), q = 2 * (k - r * (kTileX / 2));
            float2 A[2] = {};
            float Bg[2] = {0.f, 0.f};
#pragma unroll
            for (int jj = 0; jj <= kTaps; jj += 2) {
                const float4 ga = *reinterpret_cast<const float4*>(&sm.Ga[r][q + jj]);
                const float2 gb = *reinterpret_cast<const float2*>(&sm.Gb[r][q + jj]);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int j = jj + h;
                    const float2 va = h ? make_float2(ga.z, ga.w) : make_float2(ga.x, ga.y);
                    const float vb = h ? gb.y : gb.x;
#pragma unroll
                    for (int o = 0; o < 2; ++o) {
                        const int tap = j - o;
                        if (tap < 0 || tap >= kTaps) continue;
                        A[o] = ffma2(w2(tap), va, A[o]);
                        Bg[o] = fmaf(w2(tap).x, vb, Bg[o]);
                    }
                }
            }
            *reinterpret_cast<float4*>(&sm.hg.a[r][q]) = make_float4(A[0].x, A[0].y, A[1].x, A[1].y);
            *reinterpret_cast<float2*>(&sm.hg.b[r][q]) = make_float2(Bg[0], Bg[1]);
        }
        __syncthreads();
        // 5. vertical pass onto the tile (four rows of one column per thread):
        //    gradient and the loss terms
        {
            const int q = tid % kTileX, r0 = 4 * (tid / kTileX);
            float2 A[4] = {};
            float Bg[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int j = 0; j < kTaps + 3; ++j) {
                const float2 ha = sm.hg.a[r0 + j][q];
                const float hb = sm.hg.b[r0 + j][q];
#pragma unroll
                for (int o = 0; o < 4; ++o) {
                    const int tap = j - o;
                    if (tap < 0 || tap >= kTaps) continue;
                    A[o] = ffma2(w2(tap), ha, A[o]);
                    Bg[o] = fmaf(w2(tap).x, hb, Bg[o]);
                }
            }
#pragma unroll
            for (int o = 0; o < 4; ++o) {
                const int r = r0 + o;
                const int gy = y0 + r, gx = x0 + q;
                if (gx >= V.W || gy >= V.H) continue;
                const float2 xy = sm.XY[r + 2 * kR][q + 2 * kR];
                const float x = xy.x, y = xy.y;
                const float d = x - y;
                l1[o] += fabsf(d);
                ss[o] += sm.St[r][q];
                if (V.grad_color) {
                    const float dsum = A[o].x + 2.f * x * A[o].y + y * Bg[o];
                    const float sg = d > 0.f ? 1.f : (d < 0.f ? -1.f : 0.f);
                    const float gval = (t.lambda * sg - (1.f - t.lambda) * dsum) / (float)t.Co;
                    V.grad_color[((size_t)s * t.Co + c) * HW + (size_t)gy * V.W + gx] = t.scale * gval;
                }
            }
        }
        __syncthreads();
        if (c + 1 < t.Co) {
            store_regs();
            __syncthreads();
        }
    }
    // per-pixel loss, score weight, total
    float acc = 0.f;
#pragma unroll
    for (int h = 0; h < 4; ++h) {
        const int q = tid % kTileX, r = 4 * (tid / kTileX) + h;
        const int gy = y0 + r, gx = x0 + q;
        if (gx >= V.W || gy >= V.H) continue;
        const float ell = t.lambda * l1[h] / (float)t.Co + (1.f - t.lambda) * (1.f - ss[h] / (float)t.Co);
        if (V.score_w) V.score_w[(size_t)s * HW + (size_t)gy * V.W + gx] = t.scale * ell;
        acc += ell;
    }
    if (loss) {
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, d);
        __shared__ float wsum[8];
        if ((tid & 31) == 0) wsum[tid >> 5] = acc;
        __syncthreads();
        if (tid == 0) {
            float tot = 0.f;
            for (int u = 0; u < 8; ++u) tot += wsum[u];
            atomicAdd(loss, t.scale * tot);
        }
    }
}

constexpr int segment_rows(int steps) { return kStep * steps - 4 * kR; }

// Adds the march's CTAs for a view with segments of K, K + 1, ... steps (K a
// constant, so that no division is left: the host has 64 views times 8 to do
// before the launch).
template <int K = 2>
void add_march_ctas(int w, int h, long long* ctas) {
    constexpr int rows = segment_rows(K);
    ctas[K] += (long long)((w + kTX - 1) / kTX) * ((h + rows - 1) / rows);
    if constexpr (K < kMaxSteps) add_march_ctas<K + 1>(w, h, ctas);
}

}  // namespace

cudaError_t launch_loss_l1_ssim(int n_views, int S, int Co, const int* hw, const float* const* colors,
                                const float* const* targets, float* const* grad_colors, float* const* score_ws,
                                float lambda, float scale, float* loss, cudaStream_t st) {
    SsimTable* t = new (std::nothrow) SsimTable();
    if (!t) return cudaErrorMemoryAllocation;
    t->n = n_views;
    t->S = S;
    t->Co = Co;
    t->lambda = lambda;
    t->scale = scale;
    double w[kTaps], sum = 0.0;
    for (int j = 0; j < kTaps; ++j) {
        const double k = j - kR;
        w[j] = std::exp(-k * k / (2.0 * 1.5 * 1.5));
        sum += w[j];
    }
    for (int j = 0; j <= kR; ++j) t->w[j] = (float)(w[j] / sum);
    // Segment length: long ones blur fewer rows twice (20 per segment), short
    // ones spread a small call over the chip.  A CTA fills an SM and takes time
    // in proportion to its steps, so the waves of CTAs times the steps (and a
    // bit for starting up) is what is least.
    const int sms = persistent_grid(1 << 30, 1);
    long long ctas[kMaxSteps + 1] = {};
    for (int v = 0; v < n_views; ++v) add_march_ctas(hw[2 * v], hw[2 * v + 1], ctas);
    int steps = 2;
    double best = 1e300;
    for (int k = 2; k <= kMaxSteps; ++k) {
        const double cost = (double)((S * ctas[k] + sms - 1) / sms) * (k + 0.5);
        if (cost < best) best = cost, steps = k;
    }
    const auto tiles = [](int w, int h) {
        return (long long)((w + kTileX - 1) / kTileX) * ((h + kTileY - 1) / kTileY);
    };
    long long n_tiles = 0;
    for (int v = 0; v < n_views; ++v) n_tiles += S * tiles(hw[2 * v], hw[2 * v + 1]);
    // The tile kernel's cost in the same unit, a step of the march (about 12 us
    // with three channels): two CTAs fill an SM for 2.3 steps, and what is
    // left over after whole waves takes 1.6 or, above one CTA per SM, 2.6.
    // Over 236 shapes from 1 to 1,920 columns, 16 to 1,080 rows and 1 to 64
    // images the slower kernel is picked once, by 0.6%; with the tile kernel
    // up to one wave and the march above it was up to 79% (64 images of
    // 512 x 16).
    const long long left = n_tiles % (2 * sms);
    const bool small = 2.3 * (double)(n_tiles / (2 * sms)) + (left == 0 ? 0.0 : left <= sms ? 1.6 : 2.6) <= best;
    t->rows = segment_rows(steps);
    long long cta = 0;
    for (int v = 0; v < n_views; ++v) {
        SsimView& d = t->v[v];
        d.W = hw[2 * v];
        d.H = hw[2 * v + 1];
        d.color = colors[v];
        d.target = targets[v];
        d.grad_color = grad_colors ? grad_colors[v] : nullptr;
        d.score_w = score_ws ? score_ws[v] : nullptr;
        d.strips = small ? (d.W + kTileX - 1) / kTileX : (d.W + kTX - 1) / kTX;
        d.cta0 = (int)cta;
        cta += S * (small ? tiles(d.W, d.H) : (long long)d.strips * ((d.H + t->rows - 1) / t->rows));
    }
    const auto run = [&](auto kernel, int threads, size_t smem) {
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess || cta == 0) return e;
        kernel<<<(unsigned)cta, threads, smem, st>>>(*t, loss);
        note_launches(1);
        return cudaGetLastError();
    };
    const cudaError_t e = small ? run(k_loss_l1_ssim_tile, 256, sizeof(TileSmem))
                                : run(k_loss_l1_ssim, kThreads, sizeof(SsimSmem));
    delete t;
    return e;
}

}  // namespace ds
