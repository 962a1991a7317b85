// A warp's stream over the segments of a list of senders.
//
// Delivery reads, for every sender of a list, short segments of the record store (about 25
// records each).  A warp takes its senders 32 at a time, one segment per lane,
// and concatenates the segments: the batch becomes one run of `units` (the 16- or 32-byte
// pieces that a lane loads at once), dealt to the lanes in order.  Everything that locates
// a unit stays in the warp: a prefix sum by shuffles, and a scratch line in shared memory
// where each segment leaves its offset at its first unit.  The next batch's list entries
// and segment bounds are loaded while the current batch's units are read, and a set of
// units is in flight while the set before it is added, across batches too.  The warps of a
// CTA never wait for one another until the list is done, so the record reads, which bound
// these kernels, do not drain.
#pragma once

#include <cstdint>

namespace snn {

// One lane's segment: its first unit in the record store, its units, and what the source
// wants back with each of them.
struct Segment {
    uint32_t first;
    int32_t units;
    uint32_t flags;
};

// One unit of the stream, per lane.
struct StreamUnit {
    uint32_t index;         // in the record store
    uint32_t flags;         // of its segment
    bool ok, starts, ends;  // inside the batch; the first, the last of its segment
};

struct StreamBatch {
    Segment seg;
    int32_t pfx;    // the lane's first unit in the batch
    int32_t total;  // units of the batch
};

__device__ __forceinline__ StreamBatch stream_batch(const Segment &seg)
{
    const int lane = threadIdx.x & 31;
    int32_t x = seg.units;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
        if (lane >= o) x += y;
    }
    return StreamBatch{seg, x - seg.units, __shfl_sync(0xFFFFFFFFu, x, 31)};
}

// 1 << s, 0 for s outside [0, 32)
__device__ __forceinline__ uint32_t bit_or_none(int32_t s)
{
    uint32_t v;
    asm("shl.b32 %0, %1, %2;" : "=r"(v) : "r"(1u), "r"(static_cast<uint32_t>(s)));
    return v;
}

__device__ __forceinline__ uint32_t shared_address(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// Adds w to the shared word at `addr` if key < limit and w != 0.
__device__ __forceinline__ void add_shared_if(uint32_t addr, int32_t w, uint32_t key, uint32_t limit)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.lt.u32 p, %2, %3;\n\tsetp.ne.and.s32 p, %1, 0, p;\n\t"
        "@p red.relaxed.cta.shared.add.s32 [%0], %1;\n\t}" ::"r"(addr),
        "r"(w), "r"(key), "r"(limit)
        : "memory");
}

// Adds w to the shared word at `addr` if key < limit and mask has a bit of `bits`.
__device__ __forceinline__ void add_shared_masked(uint32_t addr, int32_t w, uint32_t key, uint32_t limit, uint32_t mask,
                                                  uint32_t bits)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .u32 m;\n\tand.b32 m, %4, %5;\n\tsetp.lt.u32 p, %2, %3;\n\t"
        "setp.ne.and.u32 p, m, 0, p;\n\t@p red.relaxed.cta.shared.add.s32 [%0], %1;\n\t}" ::"r"(addr),
        "r"(w), "r"(key), "r"(limit), "r"(mask), "r"(bits)
        : "memory");
}

// Position of the highest set bit (x != 0)
__device__ __forceinline__ uint32_t highest_bit(uint32_t x)
{
    uint32_t v;
    asm("bfind.u32 %0, %1;" : "=r"(v) : "r"(x));
    return v;
}

// The units e0 .. e0 + 32 kRounds of the batch, unit e0 + 32 k + lane in u[k].  `scratch`:
// the warp's 32 kRounds entries.  `carry`: the segment that holds unit e0 - 1 (anything at
// e0 = 0), updated for the next call.  Flags, starts and ends are told with kFlags only.
template <int kRounds, bool kFlags>
__device__ __forceinline__ void stream_locate(const StreamBatch &b, uint2 *scratch, int32_t e0, uint2 &carry,
                                              StreamUnit (&u)[kRounds])
{
    const int lane = threadIdx.x & 31;
    uint32_t *scratch1 = reinterpret_cast<uint32_t *>(scratch);
    const int32_t st = b.seg.units > 0 ? b.pfx - e0 : -1;  // the lane's segment starts here
    const int32_t en = st + b.seg.units - 1;               // ... and ends here (-2 or -1: none)
    __syncwarp();                                          // the previous set's reads of the scratch are done
    if (static_cast<uint32_t>(st) < 32u * kRounds) {
        if (kFlags) scratch[st] = make_uint2(b.seg.first - b.pfx, b.seg.flags);
        else scratch1[st] = b.seg.first - b.pfx;
    }
    __syncwarp();
    const uint32_t upto_lane = 0xFFFFFFFFu >> (31 - lane);
#pragma unroll
    for (int k = 0; k < kRounds; ++k) {
        const uint32_t starts = __reduce_or_sync(0xFFFFFFFFu, bit_or_none(st - 32 * k));
        uint2 own = carry;
        if (starts & upto_lane) {
            const uint32_t at = 32 * k + highest_bit(starts & upto_lane);
            if (kFlags) own = scratch[at];
            else own.x = scratch1[at];
        }
        carry.x = __shfl_sync(0xFFFFFFFFu, own.x, 31);
        const int32_t e = e0 + 32 * k + lane;
        u[k].index = own.x + static_cast<uint32_t>(e);
        u[k].ok = e < b.total;
        if (kFlags) {
            const uint32_t ends = __reduce_or_sync(0xFFFFFFFFu, bit_or_none(en - 32 * k));
            carry.y = __shfl_sync(0xFFFFFFFFu, own.y, 31);
            u[k].flags = own.y;
            u[k].starts = (starts >> lane) & 1u;
            u[k].ends = (ends >> lane) & 1u;
        }
    }
}

// Streams segments 0 .. n - 1 of a source: warp `warp` of `warps` takes batches of equal
// size.  A source gives
//   int32_t sender(int64_t j)          segment j's sender, from the list (>= 0)
//   Raw raw(int64_t j, int32_t sender) the loads that bound the segment, issued early
//   Segment segment(const Raw &)       the segment
//   void load(const StreamUnit (&)[kRounds], Set &)   issues a set's record loads
//   void add(const Set &)              adds the set's records
// Once the reads keep flowing, what these loops cost is instructions, so sources add a
// record by predicated instructions (add_shared_if below): as branches, the adds and the
// tests around them took 37 warp instructions per warp-wide add.
template <class Source>
struct WarpStream {
    static constexpr int kRounds = Source::kRounds;
    const Source &src;
    int64_t n;
    uint2 *scratch;
    int64_t at, step;  // the lane's segment of the batch after next, segments per pass of all warps
    int32_t size;      // segments per batch
    int32_t s_next;    // its sender (-1: none)
    typename Source::Raw raw;  // bounds of the next batch
    bool raw_ok;
    StreamBatch batch;
    int32_t e0;
    uint2 carry;

    __device__ __forceinline__ int32_t fetch() const
    {
        return static_cast<int32_t>(threadIdx.x & 31) < size && at < n ? src.sender(at) : -1;
    }
    // The next batch's bounds, and the list entry of the one after it.
    __device__ __forceinline__ void ahead()
    {
        raw_ok = s_next >= 0;
        if (raw_ok) raw = src.raw(at, s_next);
        at += step;
        s_next = fetch();
    }

    __device__ __forceinline__ WarpStream(const Source &source, int64_t count, int warp, int warps, uint2 *scr)
        : src(source), n(count), scratch(scr)
    {
        // passes of all warps over the list, each as even as its batches of at most 32 allow
        const int64_t passes = (n + 32 * warps - 1) / (32 * warps);
        size = static_cast<int32_t>((n + warps * passes - 1) / (warps * passes));
        step = static_cast<int64_t>(size) * warps;
        at = static_cast<int64_t>(size) * warp + (threadIdx.x & 31);
        s_next = fetch();
        ahead();
        batch = StreamBatch{Segment{0, 0, 0}, 0, 0};
        e0 = 0;
        carry = make_uint2(0, 0);
    }

    // Issues the loads of the next set; false when the stream is done (the whole warp).
    __device__ __forceinline__ bool next(typename Source::Set &set)
    {
        while (e0 >= batch.total) {
            if (!__any_sync(0xFFFFFFFFu, raw_ok)) return false;
            batch = stream_batch(raw_ok ? src.segment(raw) : Segment{0, 0, 0});
            e0 = 0;
            ahead();
        }
        StreamUnit u[kRounds];
        stream_locate<kRounds, Source::kFlags>(batch, scratch, e0, carry, u);
        src.load(u, set);
        e0 += 32 * kRounds;
        return true;
    }

    __device__ __forceinline__ void run()
    {
        typename Source::Set a, b;
        bool more = next(a);
        while (more) {
            const bool more_b = next(b);
            src.add(a);
            if (!more_b) break;
            more = next(a);
            src.add(b);
        }
    }
};

}  // namespace snn
