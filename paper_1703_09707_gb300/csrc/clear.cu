// clear.cu -- the clears before a shooting or binning call (the source map, the ray
// counters, the work queue) in one launch.  The kernel that follows may be launched with
// programmatic stream serialisation: it then starts at once, does everything that touches
// neither, and waits for the clears (pdl_wait) before its first increment.  Two or
// four cudaMemsetAsync, each a node of its own before the kernel could start, took 3 us of
// a 49 us map (100 stars, 1000^2 rays) and 4 us of binning 8192^2 records (163 -> 159 us).
// The clear takes the shared-memory carveout of the kernel behind it although it uses no
// shared memory: an SM takes no CTA that needs another carveout before it has drained, so that
// kernel's first CTAs would crowd on the few SMs that drain first.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "mlens_dev.cuh"

namespace mlens {

__global__ void __launch_bounds__(256) k_clear(ClearArgs a)
{
    pdl_launch_next();
    const size_t tid = (size_t)blockIdx.x * blockDim.x + threadIdx.x, step = (size_t)gridDim.x * blockDim.x;
    // the map from its first 16-byte boundary in vectors, the rest in words
    const size_t head = min(a.n, (size_t)((16u - ((uintptr_t)a.map & 15u)) & 15u) / 4u), vec = (a.n - head) / 4;
    uint4 *v = reinterpret_cast<uint4 *>(a.map + head);
    for (size_t k = tid; k < vec; k += step) v[k] = make_uint4(0u, 0u, 0u, 0u);
    const size_t rest = a.n - 4 * vec;  // below 8: `head` words in front, the others behind
    if (tid < rest) a.map[tid < head ? tid : 4 * vec + tid] = 0u;
#pragma unroll
    for (int w = 0; w < 3; ++w)
        if (tid < (size_t)a.nwords[w]) a.words[w][tid] = 0u;
}

cudaError_t launch_clear(const ClearArgs &a, cudaStream_t s)
{
    const size_t blocks = std::min<size_t>((a.n / 4 + 255) / 256 + 1, 2048);
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
    attr[0].val.sharedMemCarveout = (unsigned)a.carveout;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(256);
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = a.carveout < 0 ? 0 : 1;
    return cudaLaunchKernelEx(&cfg, k_clear, a);
}

}  // namespace mlens
