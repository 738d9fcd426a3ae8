// clear.cu -- the clears before a shooting or binning call (the source map, the ray
// counters, the work queue) in one launch.  The kernel that follows may be launched with
// programmatic stream serialisation: it then starts at once, does everything that touches
// neither, and waits for the clears (pdl_wait) before its first increment.  Two or
// four cudaMemsetAsync, each a node of its own before the kernel could start, took 3 us of
// a 49 us map (100 stars, 1000^2 rays) and 4 us of binning 8192^2 records (163 -> 159 us).
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
    k_clear<<<(unsigned)blocks, 256, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace mlens
