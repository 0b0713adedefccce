// compams_collect: one worker's gradient, which a backward pass leaves as one tensor per parameter, gathered into
// that worker's packed row of G.
//
// Bound by the launch for small models and by memory beyond: 4 bytes read and 4 written per coordinate, one launch
// for up to kCollectMax tensors instead of one copy each (ResNet-18 shapes, 62 tensors: the copies cost the host
// 0.5 ms per worker: four workers' gradients collected and one Top-k step 2.21 ms, now 0.287). The tensors' addresses and the tiles' starts travel as the kernel's argument; a CTA finds its
// tensor by bisection in the constant bank.
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/compams.h"
#include "common.cuh"

namespace {

using namespace compams;

constexpr int kCollectMax = 160;    // tensors of one launch: their list (3.8 KB) fits the classic argument space
constexpr int kCollectTile = 4096;  // coordinates per CTA: 4 groups of 4 per thread

struct CollectList {
    const float* src[kCollectMax];  // null: the tensor got no gradient, its coordinates are 0
    int64_t dst[kCollectMax];       // first coordinate in the row
    int32_t tile0[kCollectMax + 1]; // first tile of each tensor
    int32_t len_mod[kCollectMax];   // elements of its last tile
    int32_t count;
};
static_assert(sizeof(CollectList) <= 4000, "kernel argument space");

// A tile's coordinates in groups of four that start on 16-byte boundaries of the row (the first and the last group
// may be partial), so that the stores are 128 bits wide; the loads take the width that the tensor's phase allows.
__global__ void __launch_bounds__(kThreads) collect_kernel(float* __restrict__ row, const __grid_constant__ CollectList c) {
    int lo = 0, hi = c.count - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (c.tile0[mid] <= (int)blockIdx.x) lo = mid; else hi = mid - 1;
    }
    const int local = (int)blockIdx.x - c.tile0[lo];
    const bool last = (int)blockIdx.x + 1 == c.tile0[lo + 1];
    const int len = last ? c.len_mod[lo] : kCollectTile;
    const size_t r0 = (size_t)local * kCollectTile;
    float* out = row + c.dst[lo] + r0;
    const float* in = c.src[lo] ? c.src[lo] + r0 : nullptr;
    const int phase = align_class(out);  // elements past a 16-byte boundary of the row
    const int cls = in ? align_class(in - phase) : 0;
    constexpr int kGroups = kCollectTile / 4 / kThreads;
    float4 x[kGroups];
#pragma unroll
    for (int u = 0; u < kGroups; ++u) {
        const int r = (u * kThreads + (int)threadIdx.x) * 4 - phase;
        x[u] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (in && r >= 0 && r + 3 < len) x[u] = load4_stream(in + r, cls);
    }
#pragma unroll
    for (int u = 0; u < kGroups; ++u) {
        const int r = (u * kThreads + (int)threadIdx.x) * 4 - phase;
        if (r >= 0 && r + 3 < len) {
            *reinterpret_cast<float4*>(out + r) = x[u];
        } else {
            for (int k = 0; k < 4; ++k)
                if (r + k >= 0 && r + k < len) out[r + k] = in ? in[r + k] : 0.0f;
        }
    }
    // a row that starts past a boundary leaves up to 3 coordinates of a full tile beyond the groups above
    const int tail = kCollectTile - phase + (int)threadIdx.x;
    if (tail < len) out[tail] = in ? in[tail] : 0.0f;
}

}  // namespace

extern "C" int compams_collect(float* row, const float* const* tensors, const int64_t* offsets, int32_t count,
                               void* cuda_stream) {
    if (!row || !tensors || !offsets || count < 1 || (reinterpret_cast<uintptr_t>(row) & 3u) || offsets[0] < 0)
        return COMPAMS_ERR_INVALID_ARG;
    for (int32_t k = 0; k < count; ++k) {
        const int64_t len = offsets[k + 1] - offsets[k];
        if (len < 1 || len > ((int64_t)1 << 40) || (reinterpret_cast<uintptr_t>(tensors[k]) & 3u)) return COMPAMS_ERR_INVALID_ARG;
    }
    CollectList c;
    for (int32_t k0 = 0; k0 < count;) {
        int64_t tiles = 0;
        c.count = 0;
        for (; k0 < count && c.count < kCollectMax; ++k0, ++c.count) {
            const int64_t len = offsets[k0 + 1] - offsets[k0], nt = (len + kCollectTile - 1) / kCollectTile;
            if (tiles + nt > (int64_t)0x7fffffff) break;
            c.src[c.count] = tensors[k0];
            c.dst[c.count] = offsets[k0];
            c.tile0[c.count] = (int32_t)tiles;
            c.len_mod[c.count] = (int32_t)(len - (nt - 1) * kCollectTile);
            tiles += nt;
        }
        c.tile0[c.count] = (int32_t)tiles;
        collect_kernel<<<(unsigned)tiles, kThreads, 0, (cudaStream_t)cuda_stream>>>(row, c);
        if (cudaGetLastError() != cudaSuccess) return COMPAMS_ERR_CUDA;
    }
    return COMPAMS_OK;
}
