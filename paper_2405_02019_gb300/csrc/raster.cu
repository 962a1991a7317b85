// Orders a stretch of the device raster by (step, neuron) on the GPU, for reads that
// find the device idle (drain() in abi.cu).
//
// The engines append spikes in no order inside a step; circuit groups append whole runs
// of steps one group after another, and the resident engine's blocks run up to two steps
// apart.  The order is that of a counting sort by step followed by a sort of each step's
// few hundred neurons:
//   k_raster_count   spikes per step (one atomic per warp and distinct step);
//   k_raster_scan    their exclusive prefix sums, in one CTA;
//   k_raster_scatter every spike into its step's bucket;
//   k_raster_rank    one CTA per step: a neuron's place is the number of smaller neurons
//                    in its bucket (a neuron spikes at most once per step).
// The host then fills the step numbers from the prefix sums, so only neurons and one
// offset per step cross the link.  What bounds it: four launches and about m compares per
// spike in a step of m spikes (m is 3 to 500 here), both far below the host's sort.
// snn_read_spikes through the Python binding, host sort -> this: 435,183 spikes of a
// 16-circuit batch in two groups 12.8 -> 1.14 ms, 512,358 spikes of the 4x circuit
// 11.6 -> 1.36 ms, 29,493 spikes of a full-scale call 0.56 (resident engine) and 0.40
// (pipelined) -> 0.17 and 0.19 ms.
#include <cuda_runtime.h>

#include "internal.hpp"

namespace snn {

namespace {

constexpr int kRasterThreads = 256;

// Adds 1 to counter[s] for every lane with ok and returns the lane's place before the
// add; lanes of a warp with the same s share one atomic.
__device__ __forceinline__ uint32_t bucket_add(uint32_t *counter, uint32_t s, bool ok)
{
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t same = __match_any_sync(0xFFFFFFFFu, ok ? s : 0xFFFFFFFFu);
    const int leader = __ffs(same) - 1;
    uint32_t base = 0;
    if (ok && static_cast<int>(lane) == leader) base = atomicAdd(counter + s, static_cast<uint32_t>(__popc(same)));
    base = __shfl_sync(0xFFFFFFFFu, base, leader);
    return base + __popc(same & ((1u << lane) - 1u));
}

// Spikes whose step is not in [t0, t0 + n_steps) are counted in off[n_steps] (none are
// expected; the host then falls back to its own sort).
__global__ void __launch_bounds__(kRasterThreads) k_raster_count(const RasterSort a)
{
    const int64_t e = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    const bool in = e < a.count;
    const uint32_t s = in ? static_cast<uint32_t>(a.t[e]) - static_cast<uint32_t>(a.t0) : 0u;
    bucket_add(a.cur, min(s, static_cast<uint32_t>(a.n_steps)), in);
}

// off[0 .. n_steps + 1]: exclusive prefix sums of cur[0 .. n_steps], which they replace.
__global__ void __launch_bounds__(1024) k_raster_scan(const RasterSort a)
{
    __shared__ uint32_t warp_sum[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t carry = 0;
    for (int64_t b = 0; b <= a.n_steps; b += 1024) {
        const int64_t j = b + threadIdx.x;
        const uint32_t v = j <= a.n_steps ? a.cur[j] : 0u;
        uint32_t x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) warp_sum[warp] = x;
        __syncthreads();
        uint32_t before = 0, total = 0;
        for (int w = 0; w < 32; ++w) {
            before += w < warp ? warp_sum[w] : 0u;
            total += warp_sum[w];
        }
        if (j <= a.n_steps) {
            const uint32_t at = carry + before + x - v;
            a.off[j] = at;
            a.cur[j] = at;
        }
        carry += total;
        __syncthreads();
    }
    if (threadIdx.x == 0) a.off[a.n_steps + 1] = carry;
}

__global__ void __launch_bounds__(kRasterThreads) k_raster_scatter(const RasterSort a)
{
    const int64_t e = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    const bool in = e < a.count;
    const uint32_t s = in ? static_cast<uint32_t>(a.t[e]) - static_cast<uint32_t>(a.t0) : 0u;
    const uint32_t pos = bucket_add(a.cur, min(s, static_cast<uint32_t>(a.n_steps)), in);
    if (in) a.out[pos] = a.nrn[e];
}

// Buckets above kRasterMaxBucket spikes stay as they are; the host orders those.
__global__ void __launch_bounds__(kRasterThreads) k_raster_rank(const RasterSort a)
{
    __shared__ __align__(16) int32_t ids[kRasterMaxBucket + 4];
    for (int64_t s = blockIdx.x; s < a.n_steps; s += gridDim.x) {
        const uint32_t lo = a.off[s];
        const int m = static_cast<int>(a.off[s + 1] - lo);
        if (m < 2 || m > kRasterMaxBucket) continue;  // the whole CTA
        for (int j = threadIdx.x; j < m + 4; j += kRasterThreads) ids[j] = j < m ? a.out[lo + j] : INT32_MAX;
        __syncthreads();
        for (int j = threadIdx.x; j < m; j += kRasterThreads) {
            const int32_t id = ids[j];
            int rank = 0;
            for (int k = 0; k < m; k += 4) {
                const int4 v = *reinterpret_cast<const int4 *>(ids + k);
                rank += (v.x < id) + (v.y < id) + (v.z < id) + (v.w < id);
            }
            a.out[lo + rank] = id;
        }
        __syncthreads();  // the ids are rewritten for the next step
    }
}

}  // namespace

int launch_raster_sort(const RasterSort &a, int num_sms, void *stream)
{
    const cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int grid = static_cast<int>((a.count + kRasterThreads - 1) / kRasterThreads);
    cudaError_t e = cudaMemsetAsync(a.cur, 0, sizeof(uint32_t) * (a.n_steps + 1), st);
    if (e != cudaSuccess) return static_cast<int>(e);
    k_raster_count<<<grid, kRasterThreads, 0, st>>>(a);
    k_raster_scan<<<1, 1024, 0, st>>>(a);
    k_raster_scatter<<<grid, kRasterThreads, 0, st>>>(a);
    k_raster_rank<<<static_cast<int>(std::min<int64_t>(a.n_steps, int64_t{num_sms} * 6)), kRasterThreads, 0, st>>>(a);
    return static_cast<int>(cudaGetLastError());
}

}  // namespace snn
