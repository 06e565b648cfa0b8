// Copy-in of the host-buffer entry point: up to four arrays in pinned host memory, read over PCIe by the
// SMs into device memory by ONE kernel.  A copy command costs 3.7 us of its stream besides its
// bytes (6.5 us the first), and a step has four arrays of which three are small; this kernel takes
// them together, at 48 GB/s against the copy engine's 52.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace omni {

constexpr int kGatherThreads = 512, kGatherAhead = 4;
struct GatherPart {
    const void *src;      // host, 16-byte aligned
    void *dst;            // device, 16-byte aligned
    size_t bytes;         // a multiple of 4
};
struct GatherParts {
    GatherPart part[4];   // an unused one has bytes = 0
};

__global__ void __launch_bounds__(kGatherThreads) host_gather_kernel(const __grid_constant__ GatherParts parts)
{
    // the staging area may still be in use by the previous kernels of the stream, and they may have
    // produced the host buffers
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const size_t first = (size_t)blockIdx.x * kGatherThreads + threadIdx.x, step = (size_t)gridDim.x * kGatherThreads;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        const GatherPart &g = parts.part[a];
        const uint4 *src = static_cast<const uint4 *>(g.src);
        uint4 *dst = static_cast<uint4 *>(g.dst);
        const size_t n = g.bytes / 16;
        for (size_t i = first; i < n; i += kGatherAhead * step) {
            uint4 v[kGatherAhead];
#pragma unroll
            for (int k = 0; k < kGatherAhead; ++k)
                if (i + k * step < n) v[k] = __ldcv(src + i + k * step);
#pragma unroll
            for (int k = 0; k < kGatherAhead; ++k)
                if (i + k * step < n) dst[i + k * step] = v[k];
        }
        const size_t words = (g.bytes % 16) / 4;
        if (first < words) static_cast<uint32_t *>(g.dst)[4 * n + first] = __ldcv(static_cast<const uint32_t *>(g.src) + 4 * n + first);
    }
}

}  // namespace omni
