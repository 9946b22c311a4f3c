// Normals of a patch's blended maps by finite differences (Sec. 4.2: the
// normals are derived from the height maps by finite differences).  The
// paper gives no formula; with choppy displacement the surface is the
// displaced grid p(i, j) = (i c + Dx, j c + Dy, h) (c the cell size), and its
// normal is the normalised cross product of the two finite-difference
// tangents: central differences inside the patch, one-sided at its edges.
#include <cuda_runtime.h>

#include "internal.h"

namespace scwp {
namespace {

__global__ void __launch_bounds__(256) k_normals(const float* maps, int W, int H, float cell, float* dst) {
    const size_t plane = (size_t)W * H;
    const float* h = maps;
    const float* dx = maps + plane;
    const float* dy = maps + 2 * plane;
    for (size_t o = (size_t)blockIdx.x * blockDim.x + threadIdx.x; o < plane; o += (size_t)gridDim.x * blockDim.x) {
        const int j = (int)(o / W), i = (int)(o - (size_t)j * W);
        const int il = i > 0 ? i - 1 : i, ir = i < W - 1 ? i + 1 : i;
        const int jl = j > 0 ? j - 1 : j, jr = j < H - 1 ? j + 1 : j;
        const size_t a = (size_t)j * W + il, b = (size_t)j * W + ir;
        const size_t c = (size_t)jl * W + i, d = (size_t)jr * W + i;
        // tangents along i and j (each scaled by its own step count, which
        // does not change the normal's direction)
        float tx0 = (float)(ir - il) * cell + dx[b] - dx[a], tx1 = dy[b] - dy[a], tx2 = h[b] - h[a];
        float ty0 = dx[d] - dx[c], ty1 = (float)(jr - jl) * cell + dy[d] - dy[c], ty2 = h[d] - h[c];
        if (ir == il) { tx0 = cell; tx1 = tx2 = 0.f; }   // one-texel-wide patch
        if (jr == jl) { ty1 = cell; ty0 = ty2 = 0.f; }
        const float nx = tx1 * ty2 - tx2 * ty1;
        const float ny = tx2 * ty0 - tx0 * ty2;
        const float nz = tx0 * ty1 - tx1 * ty0;
        const float inv = rsqrtf(nx * nx + ny * ny + nz * nz);
        dst[o] = nx * inv;
        dst[plane + o] = ny * inv;
        dst[2 * plane + o] = nz * inv;
    }
}

}  // namespace

cudaError_t launch_normals(const float* maps, int W, int H, float cell, float* dst, cudaStream_t st) {
    const size_t n = (size_t)W * H;
    int blocks = (int)((n + 255) / 256);
    if (blocks > 152 * 16) blocks = 152 * 16;
    k_normals<<<blocks, 256, 0, st>>>(maps, W, H, cell, dst);
    count_launches(1);
    return cudaGetLastError();
}

namespace {

// Maps to a caller's device buffer.  A small map is latency: a copy enqueued
// through the copy API took 5 us each, one after the other (33 of them 169 us
// of a 1.5 ms frame of 32 patches); this kernel's launch overlaps its
// predecessor's end.  Four 16-byte loads in flight per thread where both
// ends are aligned.
constexpr int kCopyTpb = 256, kCopyItems = 4;

template <typename T>
__global__ void __launch_bounds__(kCopyTpb) k_copy(const T* __restrict__ src, T* __restrict__ dst, size_t n) {
    pdl_enter();
    const size_t stride = (size_t)gridDim.x * kCopyTpb;
    size_t i = (size_t)blockIdx.x * kCopyTpb + threadIdx.x;
    for (; i + (kCopyItems - 1) * stride < n; i += kCopyItems * stride) {
        T v[kCopyItems];
#pragma unroll
        for (int k = 0; k < kCopyItems; ++k) v[k] = src[i + k * stride];
#pragma unroll
        for (int k = 0; k < kCopyItems; ++k) dst[i + k * stride] = v[k];
    }
    for (; i < n; i += stride) dst[i] = src[i];
}

template <typename T>
cudaError_t copy_of(const float* src, float* dst, size_t n, cudaStream_t st) {
    const size_t m = n * sizeof(float) / sizeof(T);
    const size_t want = (m + kCopyTpb * kCopyItems - 1) / (kCopyTpb * kCopyItems);
    const int blocks = (int)(want < 1 ? 1 : want > 152 * 8 ? 152 * 8 : want);
    count_launches(1);
    return launch_pdl(k_copy<T>, blocks, kCopyTpb, 0, st, reinterpret_cast<const T*>(src), reinterpret_cast<T*>(dst), m);
}

}  // namespace

cudaError_t launch_copy(const float* src, float* dst, size_t n, cudaStream_t st) {
    return (((uintptr_t)src | (uintptr_t)dst) & 15u) == 0 && n % 4 == 0 ? copy_of<uint4>(src, dst, n, st)
                                                                       : copy_of<float>(src, dst, n, st);
}

}  // namespace scwp
