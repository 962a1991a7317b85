// Target-blocked records (SNN_RECORD_BLOCKED6, _BLOCKED4, _BLOCKED8): phase 2 of Listing
// push2 (§3.1) with one CTA per block of consecutive targets.
//
// Each sender's row is grouped by target block, so CTA p reads, for every sender, only
// the segment that lands in its block (row_ptr[s] + seg[s][p] .. + seg[s][p + 1]); a
// segment is a whole number of aligned quads of records (zero-weight padding).  The warps
// stream the segments of the list independently (stream.cuh): a unit is a quad, read as
// 8 bytes of records and 16 of int32 weights (BLOCKED6), one 16-byte unit of records and
// bfloat16 weights (BLOCKED4) or 32 bytes of (weight, record) pairs (BLOCKED8).
// The weights of delays below kBlockedBinRows are summed per (delay, local target) in
// shared memory and each nonzero sum is added to its ring entry once at the end; only this
// CTA writes these ring columns during the launch, so that final add is a plain
// read-modify-write.  Longer delays (one microcircuit event in 1e5) go straight to the ring
// as reductions; they land in other ring rows than the plain adds.  Integer addition makes
// every order give the same ring.
// Few events (kBlockedRowEvents; nearly every step of a simulation) are not worth clearing
// and adding the sums: then all warps of the launch share the (sender, block) segments, a few
// consecutive ones of a row each, and every record is a reduction into the ring.
// Measured (CUDA events, a list of 20,480 full-scale senders, 7.6e7 events): BLOCKED8 186 ->
// 130-134 us, 4.8 TB/s of its own bytes where the measured copy moves 6.8.  Before, the CTA staged
// 2,048 senders at a time between barriers, so the record reads drained two or three times
// per pass.  At 2,048 senders of the half-scale circuit BLOCKED4 stays at 22 us: launch,
// list -> bounds -> records -> ring is one chain of round trips there.
#include <cuda_runtime.h>

#include "internal.hpp"
#include "launch.cuh"
#include "stream.cuh"

namespace snn {

namespace {

// Threads per CTA: all that fit for a given list; in the step loop half, which leaves the
// next update kernel room to start beside this one.
constexpr int kBlockedStepThreads = 512;
constexpr int kBlockedRowBatch = 4;  // segments of a row that a warp takes at least (a round of quads)

// Rounds of 32 quads per set (two sets are in flight), and a record's fields.
template <int FMT>
struct BlockedForm {
    static constexpr bool wide = FMT == SNN_RECORD_BLOCKED8;
    static constexpr int rounds = 2;  // (of 3 BLOCKED4's 64 registers spill: 105 -> 119 us for 7.6e7 events)
    static constexpr int delay_shift = wide ? 16 : kBlockLocalBits;  // local target below
    static constexpr size_t scratch_bytes(int threads) { return sizeof(uint2) * rounds * threads; }
};
constexpr size_t kBlockedBinBytes = sizeof(int32_t) * kBlockedBinRows * kBlockMaxWidth;
static_assert(kBlockedBinBytes + BlockedForm<SNN_RECORD_BLOCKED4>::scratch_bytes(kBlockedThreads) <= 232448,
              "blocked delivery: shared memory above the 227 KB opt-in limit");
static_assert(kBlockedBinRows >= 2 && kBlockedBinRows <= kDMax && kBlockMaxWidth % 4 == 0, "bins");

__device__ __forceinline__ void red_add_s32(int32_t *addr, int32_t v)
{
    asm volatile("red.relaxed.gpu.global.add.s32 [%0], %1;" ::"l"(addr), "r"(v) : "memory");
}

// bfloat16 current (pA) -> 2^-12 pA, as the SNN_RECORD_PACKED_BF16 read-back
__device__ __forceinline__ int32_t bf16_fx(uint32_t h)
{
    return __float2int_rn(__fmul_rn(__uint_as_float((h & 0xFFFFu) << 16), 4096.0f));
}

// A set's loads, kept as read (decoded only when added): per round two 16-byte values,
//   BLOCKED6: va.xy = the quad's four uint16 records, vb = its four int32 weights;
//   BLOCKED4: va = the 16-byte unit (records, then bfloat16 currents);
//   BLOCKED8: va, vb = two 16-byte halves of (int32 weight, uint32 record) pairs.
template <int FMT>
__device__ __forceinline__ void blocked_quad(const uint4 &va, const uint4 &vb, uint32_t (&rec)[4], int32_t (&w)[4])
{
    if (BlockedForm<FMT>::wide) {
        rec[0] = va.y;
        rec[1] = va.w;
        rec[2] = vb.y;
        rec[3] = vb.w;
        w[0] = static_cast<int32_t>(va.x);
        w[1] = static_cast<int32_t>(va.z);
        w[2] = static_cast<int32_t>(vb.x);
        w[3] = static_cast<int32_t>(vb.z);
        return;
    }
    rec[0] = va.x & 0xFFFFu;
    rec[1] = va.x >> 16;
    rec[2] = va.y & 0xFFFFu;
    rec[3] = va.y >> 16;
    if (FMT == SNN_RECORD_BLOCKED4) {
        w[0] = bf16_fx(va.z);
        w[1] = bf16_fx(va.z >> 16);
        w[2] = bf16_fx(va.w);
        w[3] = bf16_fx(va.w >> 16);
    } else {
        w[0] = static_cast<int32_t>(vb.x);
        w[1] = static_cast<int32_t>(vb.y);
        w[2] = static_cast<int32_t>(vb.z);
        w[3] = static_cast<int32_t>(vb.w);
    }
}

template <int FMT>
__device__ __forceinline__ void reduce_record(const StepArgs &a, int64_t t, int32_t base, uint32_t rec, int32_t w)
{
    constexpr int shift = BlockedForm<FMT>::delay_shift;
    const int d = static_cast<int>(rec >> shift);
    red_add_s32(a.ring + ((t + d) & kDMask) * a.npad + base + static_cast<int>(rec & ((1u << shift) - 1)), w);
}

// Block p's segments of a list's senders, summed in the CTA's bins.
template <int FMT>
struct BlockedSource {
    using Form = BlockedForm<FMT>;
    static constexpr int kRounds = Form::rounds;
    static constexpr bool kFlags = false;
    static constexpr uint32_t kLimit = static_cast<uint32_t>(kBlockedBinRows) << Form::delay_shift;
    struct Raw {
        int64_t row;
        uint16_t o0, o1;
    };
    struct Set {
        uint4 va[kRounds], vb[kRounds];
    };

    const StepArgs &a;
    const int32_t *list;
    uint32_t bins;  // shared address
    int64_t t;
    int32_t base;
    int p;

    __device__ __forceinline__ int32_t sender(int64_t j) const { return __ldcg(list + j); }
    __device__ __forceinline__ Raw raw(int64_t, int32_t s) const
    {
        const uint16_t *sg = a.blk_seg + static_cast<int64_t>(s) * (a.n_blocks + 1) + p;
        return Raw{__ldg(a.row_ptr + s), __ldg(sg), __ldg(sg + 1)};
    }
    __device__ __forceinline__ Segment segment(const Raw &r) const
    {
        return Segment{static_cast<uint32_t>((r.row + r.o0) / kBlockQuad), (r.o1 - r.o0) / kBlockQuad, 0u};
    }
    __device__ __forceinline__ void load(const StreamUnit (&u)[kRounds], Set &s) const
    {
        const uint4 *q16 = reinterpret_cast<const uint4 *>(a.blk_rec);
        const int lane = threadIdx.x & 31;
#pragma unroll
        for (int k = 0; k < kRounds; ++k) {
            s.va[k] = make_uint4(0, 0, 0, 0);  // units past the end: zero weights add nothing
            s.vb[k] = make_uint4(0, 0, 0, 0);
            if (FMT == SNN_RECORD_BLOCKED8) {
                // the round's 32 quads as 64 16-byte halves, consecutive halves on
                // consecutive lanes (so one load instruction reads whole lines of a
                // segment): lane l takes halves l and 32 + l, of quads l / 2 and 16 + l / 2
                const uint32_t q = u[k].ok ? u[k].index : 0xFFFFFFFFu;
                const uint32_t q0 = __shfl_sync(0xFFFFFFFFu, q, lane >> 1);
                const uint32_t q1 = __shfl_sync(0xFFFFFFFFu, q, 16 + (lane >> 1));
                if (q0 != 0xFFFFFFFFu) s.va[k] = __ldcs(q16 + 2 * uint64_t(q0) + (lane & 1));
                if (q1 != 0xFFFFFFFFu) s.vb[k] = __ldcs(q16 + 2 * uint64_t(q1) + (lane & 1));
            } else if (u[k].ok) {
                if (FMT == SNN_RECORD_BLOCKED4) {
                    s.va[k] = __ldcs(q16 + u[k].index);
                } else {
                    const uint2 r = __ldcs(reinterpret_cast<const uint2 *>(a.blk_rec) + u[k].index);
                    s.va[k] = make_uint4(r.x, r.y, 0, 0);
                    s.vb[k] = __ldcs(reinterpret_cast<const uint4 *>(a.syn_w) + u[k].index);
                }
            }
        }
    }
    // A record: local target, delay above.  (Padding is passed over, not added: its zeros
    // would all meet in one bin.)
    __device__ __forceinline__ void near(uint32_t rec, int32_t w) const
    {
        const uint32_t d = rec >> Form::delay_shift;
        const uint32_t i = rec - d * ((1u << Form::delay_shift) - kBlockMaxWidth);
        add_shared_if(bins + 4 * i, w, rec, kLimit);
    }
    __device__ __forceinline__ void add(const Set &s) const
    {
        uint32_t longest = 0;
#pragma unroll
        for (int k = 0; k < kRounds; ++k) {
            uint32_t rec[4];
            int32_t w[4];
            blocked_quad<FMT>(s.va[k], s.vb[k], rec, w);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                near(rec[e], w[e]);
                longest = max(longest, rec[e]);
            }
        }
        if (longest < kLimit) return;
#pragma unroll
        for (int k = 0; k < kRounds; ++k) {
            uint32_t rec[4];
            int32_t w[4];
            blocked_quad<FMT>(s.va[k], s.vb[k], rec, w);
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (w[e] != 0 && rec[e] >= kLimit) reduce_record<FMT>(a, t, base, rec[e], w[e]);
        }
    }
};

// All blocks' segments of a list's senders: segment j is block j mod n_blocks of sender
// j div n_blocks, so that consecutive lanes hold consecutive segments of one row.
template <int FMT>
struct BlockedRowSource {
    static constexpr int kRounds = 1;
    static constexpr bool kFlags = true;  // a unit's flags: the first target of its block
    struct Raw {
        int64_t row;
        int32_t base;
        uint16_t o0, o1;
    };
    struct Set {
        uint4 va, vb;
        int32_t base;
    };

    const StepArgs &a;
    const int32_t *list;
    int64_t t;

    __device__ __forceinline__ int32_t sender(int64_t j) const
    {
        return __ldcg(list + static_cast<uint32_t>(j) / static_cast<uint32_t>(a.n_blocks));
    }
    __device__ __forceinline__ Raw raw(int64_t j, int32_t s) const
    {
        const uint32_t p = static_cast<uint32_t>(j) % static_cast<uint32_t>(a.n_blocks);
        const uint16_t *sg = a.blk_seg + static_cast<int64_t>(s) * (a.n_blocks + 1) + p;
        return Raw{__ldg(a.row_ptr + s), __ldg(a.blk_off + p), __ldg(sg), __ldg(sg + 1)};
    }
    __device__ __forceinline__ Segment segment(const Raw &r) const
    {
        return Segment{static_cast<uint32_t>((r.row + r.o0) / kBlockQuad), (r.o1 - r.o0) / kBlockQuad,
                       static_cast<uint32_t>(r.base)};
    }
    __device__ __forceinline__ void load(const StreamUnit (&u)[1], Set &s) const
    {
        s.va = make_uint4(0, 0, 0, 0);
        s.vb = make_uint4(0, 0, 0, 0);
        s.base = static_cast<int32_t>(u[0].flags);
        if (!u[0].ok) return;
        const uint4 *q16 = reinterpret_cast<const uint4 *>(a.blk_rec);
        const uint64_t q = u[0].index;
        if (FMT == SNN_RECORD_BLOCKED8) {
            s.va = __ldcs(q16 + 2 * q);
            s.vb = __ldcs(q16 + 2 * q + 1);
        } else if (FMT == SNN_RECORD_BLOCKED4) {
            s.va = __ldcs(q16 + q);
        } else {
            const uint2 r = __ldcs(reinterpret_cast<const uint2 *>(a.blk_rec) + q);
            s.va = make_uint4(r.x, r.y, 0, 0);
            s.vb = __ldcs(reinterpret_cast<const uint4 *>(a.syn_w) + q);
        }
    }
    __device__ __forceinline__ void add(const Set &s) const
    {
        uint32_t rec[4];
        int32_t w[4];
        blocked_quad<FMT>(s.va, s.vb, rec, w);
#pragma unroll
        for (int e = 0; e < 4; ++e)
            if (w[e] != 0) reduce_record<FMT>(a, t, s.base, rec[e], w[e]);
    }
};

template <int FMT, int kThreads>
__global__ void __launch_bounds__(kThreads, 1024 / kThreads)
    k_deliver_blocked(const StepArgs a, const int32_t *list, int64_t n_list, int64_t t_list, int k)
{
    using Form = BlockedForm<FMT>;
    extern __shared__ int4 smem4[];
    const uint32_t bins = shared_address(smem4);
    const int tid = threadIdx.x, warp = tid >> 5;
    uint2 *scratch = reinterpret_cast<uint2 *>(reinterpret_cast<uint8_t *>(smem4) + kBlockedBinBytes) + 32 * Form::rounds * warp;

    int64_t t;
    const int32_t *spk;
    int64_t nspk;
    if (list != nullptr) {
        t = t_list;
        spk = list;
        nspk = n_list;
    } else {
        // graph engine: the spikes step t appended to the raster (t_base as in k_step)
        allow_next_grid();
        t = a.ctl->t_base + k;
        wait_previous_grid();
        const uint32_t cur = __ldcg(&a.ctl->cursor);
        const uint32_t begin = __ldcg(&a.ctl->step_begin[t & 1]);
        if (blockIdx.x == 0 && threadIdx.x == 0) a.ctl->step_begin[(t + 1) & 1] = cur;
        const uint32_t end = cur < a.rast_cap ? cur : a.rast_cap;
        spk = a.rast_nrn + begin;
        nspk = end > begin ? static_cast<int64_t>(end - begin) : 0;
    }
    if (nspk == 0) return;
    if (nspk * a.mean_row < kBlockedRowEvents && nspk * a.n_blocks < (int64_t{1} << 31)) {
        // consecutive warps on consecutive CTAs, so that few segments spread over all SMs
        const BlockedRowSource<FMT> src{a, spk, t};
        WarpStream<BlockedRowSource<FMT>>(src, nspk * a.n_blocks, warp * gridDim.x + blockIdx.x,
                                          kThreads / 32 * gridDim.x, scratch, kBlockedRowBatch).run();
        return;
    }

    const int p = blockIdx.x;
    const int32_t base = a.blk_off[p];
    const int32_t width = a.blk_off[p + 1] - base;
    const BlockedSource<FMT> src{a, spk, bins, t, base, p};
    WarpStream<BlockedSource<FMT>> stream(src, nspk, warp, kThreads / 32, scratch);
    for (int j = tid; j < kBlockedBinRows * kBlockMaxWidth / 4; j += kThreads) smem4[j] = make_int4(0, 0, 0, 0);
    __syncthreads();
    stream.run();
    __syncthreads();
    // add the sums of the binned delays to their ring rows; width is a multiple
    // of 4 except for the last block, whose extra columns lie inside the padded ring row
    const int w4 = (width + 3) >> 2;
    for (int q = tid; q < (kBlockedBinRows - 1) * w4; q += kThreads) {
        const int d = 1 + q / w4;
        const int c4 = q - (d - 1) * w4;
        const int4 v = smem4[(d * kBlockMaxWidth) / 4 + c4];
        if ((v.x | v.y | v.z | v.w) == 0) continue;
        int4 *dst = reinterpret_cast<int4 *>(a.ring + ((t + d) & kDMask) * a.npad + base) + c4;
        int4 o = __ldcg(dst);
        o.x = static_cast<int32_t>(static_cast<uint32_t>(o.x) + static_cast<uint32_t>(v.x));
        o.y = static_cast<int32_t>(static_cast<uint32_t>(o.y) + static_cast<uint32_t>(v.y));
        o.z = static_cast<int32_t>(static_cast<uint32_t>(o.z) + static_cast<uint32_t>(v.z));
        o.w = static_cast<int32_t>(static_cast<uint32_t>(o.w) + static_cast<uint32_t>(v.w));
        __stcg(dst, o);
    }
}

template <int FMT, int kThreads>
constexpr size_t blocked_smem() { return kBlockedBinBytes + BlockedForm<FMT>::scratch_bytes(kThreads); }

template <int FMT, int kThreads>
cudaError_t opt_in()
{
    return cudaFuncSetAttribute(k_deliver_blocked<FMT, kThreads>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                static_cast<int>(blocked_smem<FMT, kThreads>()));
}

template <int FMT>
void launch_blocked(const StepArgs &a, const int32_t *list, int64_t n, int64_t t, int k, void *stream, bool programmatic)
{
    if (list)
        launch_after(k_deliver_blocked<FMT, kBlockedThreads>, a.n_blocks, kBlockedThreads,
                     blocked_smem<FMT, kBlockedThreads>(), stream, false, a, list, n, t, k);
    else
        launch_after(k_deliver_blocked<FMT, kBlockedStepThreads>, a.n_blocks, kBlockedStepThreads,
                     blocked_smem<FMT, kBlockedStepThreads>(), stream, programmatic, a, list, n, t, k);
}

}  // namespace

int prepare_blocked_kernel()
{
    cudaError_t e = opt_in<SNN_RECORD_BLOCKED6, kBlockedThreads>();
    if (e == cudaSuccess) e = opt_in<SNN_RECORD_BLOCKED4, kBlockedThreads>();
    if (e == cudaSuccess) e = opt_in<SNN_RECORD_BLOCKED8, kBlockedThreads>();
    if (e == cudaSuccess) e = opt_in<SNN_RECORD_BLOCKED6, kBlockedStepThreads>();
    if (e == cudaSuccess) e = opt_in<SNN_RECORD_BLOCKED4, kBlockedStepThreads>();
    if (e == cudaSuccess) e = opt_in<SNN_RECORD_BLOCKED8, kBlockedStepThreads>();
    return static_cast<int>(e);
}

void launch_deliver_blocked(const StepArgs &a, const int32_t *list, int64_t n, int64_t t, int k, void *stream,
                            bool programmatic)
{
    if (a.format == SNN_RECORD_BLOCKED4) launch_blocked<SNN_RECORD_BLOCKED4>(a, list, n, t, k, stream, programmatic);
    else if (a.format == SNN_RECORD_BLOCKED8) launch_blocked<SNN_RECORD_BLOCKED8>(a, list, n, t, k, stream, programmatic);
    else launch_blocked<SNN_RECORD_BLOCKED6>(a, list, n, t, k, stream, programmatic);
}

}  // namespace snn
