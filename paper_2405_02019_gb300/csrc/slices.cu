// Phase 2 alone (Listing push2, §3.1) for long sender lists on rows: plain and packed
// records, delivered one slice of delays at a time.
//
// A row is sorted by delay, so the synapses of one delay (about 120 of a full row) are one
// run of it, and all of a list's events with delay d land in one ring row.  A CTA therefore
// takes a group of delays and a run of senders, sums the events per target in shared
// memory, and adds each nonzero sum to the ring once.  The row-by-row kernel
// (k_deliver_list) issues one L2 reduction per event, at random addresses; their rate, 1.6e11
// to 1.75e11 events per second, is what bounds it, at a fifth of the memory's rate.  Here the
// reductions are one per nonzero sum and on consecutive addresses.  The delays of a PLAIN9
// slice of one delay need not be read at all.
//   - Shared memory holds kSliceCells sums.  Networks with more neurons are cut into
//     `parts` target ranges: the CTAs of the parts read the same records side by side (the
//     second reads them from L2) and each adds its own targets.  Networks with fewer take
//     several delays per group.
//   - The groups' events, in delay order, form one line, cut into equal pieces, one per
//     CTA, from the network's own counts per delay: a CTA's piece is a sender range of one
//     group, or ends in one group and starts the next.
//   - The rare longest delays form a last group whose events are reduced directly: summing
//     them would cost more in clearing and adding the sums than it saves.
// The records are streamed by independent warps (stream.cuh); a unit is a quad of four
// records, whose ends outside the slice are masked.
// Measured (CUDA events, back to back, one box, row by row -> slices): 8,192 senders (3.0e7
// events) of the half-scale circuit 191 -> 68 us, of the full one (two parts) 187 -> 110; 20,480
// (7.6e7 events) 443 -> 141 and 435 -> 227 us.
#include <cuda_runtime.h>

#include "internal.hpp"
#include "stream.cuh"

namespace snn {

namespace {

constexpr int kSliceThreads = 768;
// (the stream counts units in 32 bits: a plan has at most kSliceMaxParts kSliceCells rows of at
// most 65,535 synapses, padded to quads)
static_assert(int64_t{kSliceMaxParts} * kSliceCells * 65536 / 4 < int64_t{1} << 32, "units of a sliced network");
constexpr int kSliceWarps = kSliceThreads / 32;
constexpr int kSliceRounds = 2;
constexpr size_t kSliceSmem = sizeof(int32_t) * kSliceCells + sizeof(uint2) * 32 * kSliceRounds * kSliceWarps;

__device__ __forceinline__ void red_add_s32(int32_t *addr, int32_t v)
{
    asm volatile("red.relaxed.gpu.global.add.s32 [%0], %1;" ::"l"(addr), "r"(v) : "memory");
}

// One group's delays d0 .. d1 - 1.  (The two kinds of group share one instance of the
// stream: with an instance each the kernel spilled up to 600 bytes a thread.)
template <int FMT>
struct SliceSource {
    static constexpr int kRounds = kSliceRounds;
    static constexpr bool kFlags = true;
    struct Raw {
        int64_t row;
        uint32_t begin, end;  // in the row
        uint32_t pop;
    };
    struct Set {
        int4 tgt[kRounds], w[kRounds];
        uint32_t d[kRounds];
        uint32_t mask[kRounds];  // records of the quad in the slice; the sender's population above
    };

    const StepArgs &a;
    const int32_t *list;
    uint32_t bins;  // shared address
    int64_t t;
    int d0, d1;
    int32_t lo, width;  // targets lo .. lo + width - 1
    bool direct;        // reduced into the ring, not summed

    __device__ __forceinline__ int32_t sender(int64_t j) const { return __ldcg(list + j); }
    __device__ __forceinline__ Raw raw(int64_t, int32_t s) const
    {
        Raw r;
        const uint16_t *off = a.row_delay + static_cast<int64_t>(s) * kDMax;
        r.row = __ldg(a.row_ptr + s);
        r.begin = __ldg(off + d0);
        r.end = __ldg(off + (d1 & kDMask));  // entry 0 is the row's end
        r.pop = FMT == SNN_RECORD_PACKED_I8 ? __ldg(a.pop_id + s) : 0u;
        return r;
    }
    __device__ __forceinline__ Segment segment(const Raw &r) const
    {
        // rows start on quads
        return Segment{static_cast<uint32_t>(r.row / 4) + r.begin / 4,
                       r.end > r.begin ? static_cast<int32_t>((r.end + 3) / 4 - r.begin / 4) : 0,
                       (r.begin & 3u) | ((r.end & 3u) << 2) | (r.pop << 4)};
    }
    __device__ __forceinline__ void load(const StreamUnit (&u)[kRounds], Set &s) const
    {
#pragma unroll
        for (int k = 0; k < kRounds; ++k) {
            uint32_t m = 0;
            if (u[k].ok) {
                const int64_t q = u[k].index;
                s.tgt[k] = __ldcs(reinterpret_cast<const int4 *>(a.syn_tgt) + q);
                if (FMT == SNN_RECORD_PLAIN9) {
                    s.w[k] = __ldcs(reinterpret_cast<const int4 *>(a.syn_w) + q);
                    if (d1 - d0 > 1 || direct) s.d[k] = __ldcs(reinterpret_cast<const uint32_t *>(a.syn_d) + q);
                } else if (FMT == SNN_RECORD_PACKED_I8) {
                    s.w[k].x = __ldcs(a.syn_w + q);
                } else {
                    const int2 h = __ldcs(reinterpret_cast<const int2 *>(a.syn_w) + q);
                    s.w[k].x = h.x;
                    s.w[k].y = h.y;
                }
                m = 0xFu;
                if (u[k].starts) m &= 0xFu << (u[k].flags & 3u);
                const uint32_t tail = (u[k].flags >> 2) & 3u;
                if (u[k].ends && tail != 0u) m &= 0xFu >> (4u - tail);
                m |= (u[k].flags >> 4) << 4;
            }
            s.mask[k] = m;
        }
    }
    __device__ __forceinline__ int32_t weight(const Set &s, int k, int e) const
    {
        const int32_t wq[4] = {s.w[k].x, s.w[k].y, s.w[k].z, s.w[k].w};
        if (FMT == SNN_RECORD_PLAIN9) return wq[e];
        if (FMT == SNN_RECORD_PACKED_I8) {
            const int32_t tt[4] = {s.tgt[k].x, s.tgt[k].y, s.tgt[k].z, s.tgt[k].w};
            const int b = static_cast<int>((static_cast<uint32_t>(tt[e]) >> kWordPopShift) & 7u);
            const int2 pq = __ldg(reinterpret_cast<const int2 *>(&a.tables->i8_pair[s.mask[k] >> 4][b]));
            return pq.x + static_cast<int32_t>(static_cast<int8_t>((s.w[k].x >> (8 * e)) & 0xFF)) * pq.y;
        }
        const uint32_t h = static_cast<uint32_t>(e < 2 ? s.w[k].x : s.w[k].y) >> (16 * (e & 1));
        return __float2int_rn(__fmul_rn(__uint_as_float((h & 0xFFFFu) << 16), 4096.0f));
    }
    __device__ __forceinline__ uint32_t target(const Set &s, int k, int e) const
    {
        const int32_t tt[4] = {s.tgt[k].x, s.tgt[k].y, s.tgt[k].z, s.tgt[k].w};
        return static_cast<uint32_t>(tt[e]) & (FMT == SNN_RECORD_PLAIN9 ? 0xFFFFFFFFu : kWordTargetMask);
    }
    __device__ __forceinline__ int delay(const Set &s, int k, int e) const
    {
        const int32_t tt[4] = {s.tgt[k].x, s.tgt[k].y, s.tgt[k].z, s.tgt[k].w};
        return static_cast<int>(FMT == SNN_RECORD_PLAIN9 ? (s.d[k] >> (8 * e)) & 0xFFu
                                                         : (static_cast<uint32_t>(tt[e]) >> kWordDelayShift) & 63u);
    }
    // kOne: the slice is one delay, so a record's bin is its target's
    template <bool kOne>
    __device__ __forceinline__ void sum(const Set &s) const
    {
#pragma unroll
        for (int k = 0; k < kRounds; ++k)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const uint32_t c = target(s, k, e) - static_cast<uint32_t>(lo);
                const uint32_t i = kOne ? c : static_cast<uint32_t>((delay(s, k, e) - d0) * width) + c;
                add_shared_masked(bins + 4 * i, weight(s, k, e), c, static_cast<uint32_t>(width), s.mask[k], 1u << e);
            }
    }
    __device__ __forceinline__ void reduce(const Set &s) const
    {
#pragma unroll
        for (int k = 0; k < kRounds; ++k)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const uint32_t g = target(s, k, e);
                if (((s.mask[k] >> e) & 1u) && g - static_cast<uint32_t>(lo) < static_cast<uint32_t>(width))
                    red_add_s32(a.ring + ((t + delay(s, k, e)) & kDMask) * a.npad + g, weight(s, k, e));
            }
    }
    __device__ __forceinline__ void add(const Set &s) const
    {
        if (direct) reduce(s);
        else if (d1 - d0 == 1) sum<true>(s);
        else sum<false>(s);
    }
};

template <int FMT>
__global__ void __launch_bounds__(kSliceThreads, 1)
    k_deliver_slices(const StepArgs a, const SlicePlan plan, const int32_t *list, const int64_t n, const int64_t t)
{
    extern __shared__ int4 slice_smem4[];
    int32_t *bins = reinterpret_cast<int32_t *>(slice_smem4);
    const int tid = threadIdx.x, warp = tid >> 5;
    uint2 *scratch = reinterpret_cast<uint2 *>(bins + kSliceCells) + 32 * kSliceRounds * warp;
    const int part = blockIdx.x % plan.parts;
    const int64_t c = blockIdx.x / plan.parts, C = gridDim.x / plan.parts;
    const int32_t lo = part * plan.width;
    const int64_t W = plan.cum[plan.groups];
    const int64_t x0 = W * c / C, x1 = W * (c + 1) / C;  // this CTA's piece of the line
    for (int g = 0; g < plan.groups; ++g) {
        const int64_t g0 = plan.cum[g], g1 = plan.cum[g + 1];
        if (g1 <= x0 || g0 >= x1 || g0 == g1) continue;
        // the piece's senders of the group: a cut of the line is the same sender for both sides
        const int64_t s0 = x0 > g0 ? (x0 - g0) * n / (g1 - g0) : 0;
        const int64_t s1 = x1 < g1 ? (x1 - g0) * n / (g1 - g0) : n;
        if (s0 >= s1) continue;
        const int d0 = 1 + g * plan.delays;
        const bool direct = d0 >= plan.tail;
        const int d1 = direct ? kDMax : min(d0 + plan.delays, plan.tail);
        const SliceSource<FMT> src{a, list + s0, shared_address(bins), t, d0, d1, lo, plan.width, direct};
        WarpStream<SliceSource<FMT>> stream(src, s1 - s0, warp, kSliceWarps, scratch);
        if (!direct) {
            const int cells = (d1 - d0) * plan.width;  // a multiple of 4
            __syncthreads();                           // the previous group's sums are read
            for (int j = tid; j < cells / 4; j += kSliceThreads) slice_smem4[j] = make_int4(0, 0, 0, 0);
            __syncthreads();
        }
        stream.run();
        if (direct) continue;
        __syncthreads();
        for (int d = d0; d < d1; ++d) {
            const int32_t *row = bins + (d - d0) * plan.width;
            int32_t *dst = a.ring + ((t + d) & kDMask) * a.npad + lo;
            constexpr int kFlush = 8;  // sums read together: one at a time their latencies added up to 10 us
            for (int j0 = tid; j0 < plan.width; j0 += kSliceThreads * kFlush) {
                int32_t v[kFlush];
#pragma unroll
                for (int q = 0; q < kFlush; ++q)
                    v[q] = j0 + q * kSliceThreads < plan.width ? row[j0 + q * kSliceThreads] : 0;
#pragma unroll
                for (int q = 0; q < kFlush; ++q)
                    if (v[q] != 0) red_add_s32(dst + j0 + q * kSliceThreads, v[q]);
            }
        }
    }
}

}  // namespace

// Whether a list of n_senders with about `events` synapses is faster by slices than row by
// row.  Fitted to both kernels from 64 to 20,480 senders on seven networks: rows take about
// 3 us + 5.8 us per million events; slices 15 us (clearing and adding the sums) + 1.42 us,
// for each part, per million of events plus 20 for every run of a sender in a group.  So a
// full-scale row list pays from about 2,000 senders, a half-scale one from 1,000, and short
// rows later (740 synapses in two parts: never at 20,480).
bool slices_pay(const SlicePlan &plan, int64_t n_senders, int64_t events)
{
    if (plan.parts == 0) return false;
    const double rows_us = 3.0 + 5.8e-6 * static_cast<double>(events);
    const double runs = 20.0 * static_cast<double>(plan.groups) * static_cast<double>(n_senders);
    return 15.0 + 1.42e-6 * plan.parts * (static_cast<double>(events) + runs) < rows_us;
}

SlicePlan make_slice_plan(const int64_t (&events)[kDMax], int64_t n, int64_t npad)
{
    SlicePlan p{};
    int64_t total = 0;
    for (int d = 1; d < kDMax; ++d) total += events[d];
    const int64_t parts = (npad + kSliceCells - 1) / kSliceCells;
    if (total == 0 || parts > kSliceMaxParts) return p;
    const int64_t width = (npad / 4 + parts - 1) / parts * 4;
    p.width = static_cast<int32_t>(width);
    p.delays = static_cast<int32_t>(std::min<int64_t>(kDMax - 1, kSliceCells / width));
    // the longest delays, at most 3 % of the events, in whole groups
    int tail = kDMax;
    for (int64_t run = 0; tail > 2 && (run + events[tail - 1]) * 100 <= total * 3; --tail) run += events[tail - 1];
    tail = std::min(kDMax, 1 + (tail - 1 + p.delays - 1) / p.delays * p.delays);
    p.tail = tail;
    p.groups = (tail - 1 + p.delays - 1) / p.delays + (tail < kDMax ? 1 : 0);
    for (int g = 0; g < p.groups; ++g) {
        const int d0 = 1 + g * p.delays, d1 = d0 >= tail ? kDMax : std::min(d0 + p.delays, tail);
        int64_t ev = 0;
        for (int d = d0; d < d1; ++d) ev += events[d];
        // what the group costs, in summed events: its events per sender, the start of a
        // sender's run (measured 20), and 3 for an event that is reduced directly
        const double per_sender = static_cast<double>(ev) / static_cast<double>(n);
        p.cum[g + 1] = p.cum[g] + (ev > 0 ? 1 + static_cast<uint32_t>((d0 >= tail ? 3.0 : 1.0) * per_sender * 4096.0 + 20.0 * 4096.0) : 0);
    }
    p.parts = static_cast<int32_t>(parts);
    return p;
}

int launch_deliver_slices(const StepArgs &a, const SlicePlan &plan, const int32_t *list, int64_t n, int64_t t, int num_sms,
                          void *stream)
{
    const cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int grid = std::max(1, num_sms / plan.parts) * plan.parts;
    const auto kernel = a.format == SNN_RECORD_PACKED_I8     ? k_deliver_slices<SNN_RECORD_PACKED_I8>
                        : a.format == SNN_RECORD_PACKED_BF16 ? k_deliver_slices<SNN_RECORD_PACKED_BF16>
                                                             : k_deliver_slices<SNN_RECORD_PLAIN9>;
    kernel<<<grid, kSliceThreads, kSliceSmem, st>>>(a, plan, list, n, t);
    return static_cast<int>(cudaGetLastError());
}

int prepare_slices_kernel(int format)
{
    const auto kernel = format == SNN_RECORD_PACKED_I8     ? k_deliver_slices<SNN_RECORD_PACKED_I8>
                        : format == SNN_RECORD_PACKED_BF16 ? k_deliver_slices<SNN_RECORD_PACKED_BF16>
                                                           : k_deliver_slices<SNN_RECORD_PLAIN9>;
    return static_cast<int>(
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kSliceSmem)));
}

}  // namespace snn
