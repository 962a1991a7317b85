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
// Few events (nearly every step of a simulation) are not worth clearing and adding the sums:
// below kBlockedRowEvents, and while no warp gets more than two windows, all warps of the
// launch share the rows, a window of 32 consecutive quads at a time, and every record is a
// reduction into the ring.
// Measured, 20,480 senders (7.6e7 events): BLOCKED8 at full scale 181 -> 128 us, 4.8 TB/s of
// its own bytes where a copy moves 6.8; BLOCKED4 and 6 of the half-scale circuit 162 -> 107
// and 192 -> 169 us.  Before, the CTA staged 2,048 senders at a time between barriers, so the
// record reads drained two or three times per pass.  Short lists are one chain of round trips,
// list -> bounds -> records -> ring, as long as it was (kernel time, BLOCKED4 of the half-scale
// circuit: 2,048 senders 20.6 -> 20.4 us, 512 10.85 -> 10.8; BLOCKED8 at 512 12.85 -> 11.95).  On
// few blocks it is longer for BLOCKED4: 52 blocks, 256 to 1,024 senders, 0.3 to 0.6 us of 10 to 20.
#include <cuda_runtime.h>

#include "internal.hpp"
#include "launch.cuh"
#include "stream.cuh"

namespace snn {

namespace {

// Threads per CTA: all that fit for a given list; in the step loop half, which leaves the
// next update kernel room to start beside this one.
constexpr int kBlockedStepThreads = 512;
// Clearing and adding the bins is what a short list pays for: fewer delays are binned below
// kBlockedLongList senders (512 full-scale senders with BLOCKED8: 14.3 us with 48 rows, 13.5 with
// 33; at 2,048 both take 23.5).
constexpr int64_t kBlockedLongList = 2048;
constexpr int kBlockedShortRows = 33;

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
    int32_t stride;  // of the bins
    uint32_t limit;  // records from here on have a delay that is not binned
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
        const uint32_t i = rec - d * ((1u << Form::delay_shift) - static_cast<uint32_t>(stride));
        add_shared_if(bins + 4 * i, w, rec, limit);
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
        if (longest < limit) return;
#pragma unroll
        for (int k = 0; k < kRounds; ++k) {
            uint32_t rec[4];
            int32_t w[4];
            blocked_quad<FMT>(s.va[k], s.vb[k], rec, w);
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (w[e] != 0 && rec[e] >= limit) reduce_record<FMT>(a, t, base, rec[e], w[e]);
        }
    }
};

// Few events: a warp takes 32 consecutive quads of one row.  Which block a quad belongs to
// comes from the row's block table, read alongside the quads: each block that starts inside
// the window marks its first quad, and a lane's block is the last one at or before it.
// `offs`: the block boundaries, in shared memory; `scratch`: the warp's 32 words.
template <int FMT>
__device__ __forceinline__ void blocked_row_window(const StepArgs &a, int64_t t, int64_t row_quad, uint32_t len,
                                                   int32_t s, uint32_t w0, const int32_t *offs, int32_t *scratch)
{
    constexpr int kPer = 5;  // the table of up to 160 blocks in one round trip
    const int lane = threadIdx.x & 31;
    const bool ok = w0 + lane < len;
    uint4 va = make_uint4(0, 0, 0, 0), vb = va;
    if (ok) {
        const int64_t q = row_quad + w0 + lane;
        const uint4 *q16 = reinterpret_cast<const uint4 *>(a.blk_rec);
        if (FMT == SNN_RECORD_BLOCKED8) {
            va = __ldcs(q16 + 2 * q);
            vb = __ldcs(q16 + 2 * q + 1);
        } else if (FMT == SNN_RECORD_BLOCKED4) {
            va = __ldcs(q16 + q);
        } else {
            const uint2 r = __ldcs(reinterpret_cast<const uint2 *>(a.blk_rec) + q);
            va = make_uint4(r.x, r.y, 0, 0);
            vb = __ldcs(reinterpret_cast<const uint4 *>(a.syn_w) + q);
        }
    }
    const uint16_t *sg = a.blk_seg + static_cast<int64_t>(s) * (a.n_blocks + 1);
    __syncwarp();
    scratch[lane] = -1;
    __syncwarp();
    int before = 0;  // blocks that start at or before the window
    for (int b0 = 0; b0 < a.n_blocks; b0 += 32 * kPer) {
        uint32_t st[kPer];
#pragma unroll
        for (int i = 0; i < kPer; ++i)
            st[i] = b0 + lane + 32 * i < a.n_blocks ? __ldg(sg + b0 + lane + 32 * i) / kBlockQuad : 0xFFFFFFFFu;
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            before += __popc(__ballot_sync(0xFFFFFFFFu, st[i] <= w0));
            if (st[i] > w0 && st[i] < w0 + 32) atomicMax(scratch + (st[i] - w0), b0 + lane + 32 * i);
        }
    }
    __syncwarp();
    int b = max(scratch[lane], before - 1);  // empty blocks start where the next one does: the last wins
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xFFFFFFFFu, b, o);
        if (lane >= o) b = max(b, y);
    }
    if (!ok) return;
    uint32_t rec[4];
    int32_t w[4];
    blocked_quad<FMT>(va, vb, rec, w);
    const int32_t base = offs[b];
#pragma unroll
    for (int e = 0; e < 4; ++e)
        if (w[e] != 0) reduce_record<FMT>(a, t, base, rec[e], w[e]);
}

template <int FMT, int kThreads>
__global__ void __launch_bounds__(kThreads, 1024 / kThreads)
    k_deliver_blocked(const StepArgs a, const int32_t *list, int64_t n_list, int64_t t_list, int k)
{
    using Form = BlockedForm<FMT>;
    extern __shared__ int4 smem4[];
    const uint32_t bins = shared_address(smem4);
    int32_t *bins_i = reinterpret_cast<int32_t *>(smem4);  // with few events: the block boundaries
    const int tid = threadIdx.x, warp = tid >> 5;
    uint2 *scratch = reinterpret_cast<uint2 *>(reinterpret_cast<uint8_t *>(smem4) + kBlockedBinBytes) + 32 * Form::rounds * warp;

    int64_t t;
    const int32_t *spk;
    int64_t nspk;
    // consecutive warps on consecutive CTAs, so that few windows spread over all SMs
    const int64_t gw = static_cast<int64_t>(warp) * gridDim.x + blockIdx.x;
    const int64_t warps = static_cast<int64_t>(kThreads / 32) * gridDim.x;
    int4 first = make_int4(0, 0, 0, -1);
    // (the block boundaries of the row by row path fit the bins' memory)
    bool rows = a.n_blocks <= kBlockedBinRows * kBlockMaxWidth;
    if (rows && list == nullptr)
        for (int j = tid; j < a.n_blocks; j += kThreads) bins_i[j] = __ldg(a.blk_off + j);
    if (list != nullptr) {
        t = t_list;
        spk = list;
        nspk = n_list;
    } else {
        // graph engine: the spikes step t appended to the raster (t_base as in k_step), and the
        // entry of this warp's first window in the same round trip
        allow_next_grid();
        t = a.ctl->t_base + k;
        const int64_t j0 = gw / a.row_windows;
        wait_previous_grid();
        const uint32_t cur = __ldcg(&a.ctl->cursor);
        const uint32_t begin = __ldcg(&a.ctl->step_begin[t & 1]);
        if (j0 < a.queue_cap) first = __ldcg(reinterpret_cast<const int4 *>(a.queue + (t & 1) * a.npad + j0));
        if (blockIdx.x == 0 && threadIdx.x == 0) a.ctl->step_begin[(t + 1) & 1] = cur;
        const uint32_t end = cur < a.rast_cap ? cur : a.rast_cap;
        spk = a.rast_nrn + begin;
        nspk = end > begin ? static_cast<int64_t>(end - begin) : 0;
    }
    if (nspk == 0) return;
    rows = rows && nspk * a.mean_row < kBlockedRowEvents && nspk * a.row_windows <= 2 * warps;
    if (rows) {
        if (list != nullptr)
            for (int j = tid; j < a.n_blocks; j += kThreads) bins_i[j] = __ldg(a.blk_off + j);
        __syncthreads();
        for (int64_t it = gw; it < nspk * a.row_windows; it += warps) {
            const int64_t j = it / a.row_windows;
            const uint32_t w0 = static_cast<uint32_t>(it - j * a.row_windows) * 32;
            int64_t row_quad;
            uint32_t len;
            int32_t s;
            if (list != nullptr) {
                s = __ldcg(spk + j);
                const int64_t rs = __ldg(a.row_ptr + s);
                row_quad = rs / kBlockQuad;
                len = static_cast<uint32_t>((__ldg(a.row_ptr + s + 1) - rs) / kBlockQuad);
            } else {
                const int4 e = it == gw ? first : __ldcg(reinterpret_cast<const int4 *>(a.queue + (t & 1) * a.npad + j));
                row_quad = entry_first_quad(e.x, e.y);
                len = entry_quads(e.y);
                s = e.z;
            }
            if (w0 < len)
                blocked_row_window<FMT>(a, t, row_quad, len, s, w0, bins_i, reinterpret_cast<int32_t *>(scratch));
        }
        return;
    }

    const int p = blockIdx.x;
    const int32_t base = a.blk_off[p];
    const int32_t stride = BlockedForm<FMT>::wide ? kBlockMaxWidth : (a.blk_off[p + 1] - base + 3) & ~3;
    // fewer bins to clear and add for a short list
    const int bin_rows = nspk < kBlockedLongList ? kBlockedShortRows : kBlockedBinRows;
    const uint32_t limit = static_cast<uint32_t>(bin_rows) << BlockedForm<FMT>::delay_shift;
    const BlockedSource<FMT> src{a, spk, bins, t, base, stride, limit, p};
    WarpStream<BlockedSource<FMT>> stream(src, nspk, warp, kThreads / 32, scratch);
    if (list == nullptr) __syncthreads();  // the block boundaries are written before they are cleared
    for (int j = tid; j < bin_rows * stride / 4; j += kThreads) smem4[j] = make_int4(0, 0, 0, 0);
    __syncthreads();
    stream.run();
    __syncthreads();
    // add the sums of the binned delays to their ring rows; width is a multiple
    // of 4 except for the last block, whose extra columns lie inside the padded ring row
    const int w4 = (a.blk_off[p + 1] - base + 3) >> 2;
    for (int q = tid; q < (bin_rows - 1) * w4; q += kThreads) {
        const int d = 1 + q / w4;
        const int c4 = q - (d - 1) * w4;
        const int4 v = smem4[(d * stride) / 4 + c4];
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
