// ds_activate.cu -- texture activation.
#include "ds_internal.h"

namespace ds {

// ---------------------------------------------------------------- activation
// a = sigmoid(theta) on every feature-vertex channel (Sec. 3.3, applied to the
// finest grid before rasterisation); the opacity channel is also written to a
// planar [T][V] copy so that the per-fragment opacity lookups of the masked
// depth test touch 4 bytes per corner.
__global__ void k_activate(const float* __restrict__ tex, float* __restrict__ act,
                           float* __restrict__ act_a, long long n, int C) {
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += stride) {
        const float a = pinned_sigmoid(__ldg(tex + i));
        act[i] = a;
        const long long q = i / C;
        if (i - q * C == C - 1) act_a[q] = a;
    }
}

// Same with 16-byte vectors when C % 4 == 0 (the opacity channel is the last
// lane of every C/4-th vector).
__global__ void k_activate4(const float4* __restrict__ tex, float4* __restrict__ act,
                            float* __restrict__ act_a, long long n4, int C4) {
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n4; i += stride) {
        const float4 x = __ldg(tex + i);
        const float4 a = pinned_sigmoid4(x);
        act[i] = a;
        const long long q = i / C4;
        if (i - q * C4 == C4 - 1) act_a[q] = a.w;
    }
}

cudaError_t launch_activate(const SoupDev& s, cudaStream_t st) {
    const long long n = (long long)s.T * s.V * s.C;
    const bool vec = (s.C % 4 == 0) && ((uintptr_t)s.tex % 16 == 0) && ((uintptr_t)s.act % 16 == 0);
    const long long work = vec ? n / 4 : n;
    int grid = (int)((work + 255) / 256);
    if (grid > 152 * 16) grid = 152 * 16;
    if (grid < 1) grid = 1;
    if (vec)
        k_activate4<<<grid, 256, 0, st>>>(reinterpret_cast<const float4*>(s.tex),
                                          reinterpret_cast<float4*>(s.act), s.act_a, n / 4, s.C / 4);
    else
        k_activate<<<grid, 256, 0, st>>>(s.tex, s.act, s.act_a, n, s.C);
    note_launches(1);
    return cudaGetLastError();
}

}  // namespace ds
