// Device side of the simulation step (sm_103a).
//
// Phase 1 (Listing push of §3.1, fused with the ring read of §3.2 and the spike queue
// of Listing push2), for every neuron:
//     in   = W[t mod 64][i] + T(t, i) * w_ext      (int32, 2^-12 pA units)
//     W[t mod 64][i] = 0
//     if R == 0: x = p22 U + p21 I; spike if x >= theta (then x = reset, R = t_ref); U = x
//     else:      U = reset; R -= 1
//     I = p11 I + in * 2^-12
// T is Poisson(nu_th K dt) by CDF inversion of one Philox word (§2.2).  Spikers are
// compacted warp by warp (one atomic per warp with spikes) into the raster, which is
// also the step's spike queue.
// Phase 2 (Listing push2 of §3.1): every queued spiker's row (sorted by delay, §3.5)
// is cut into runs of 256-synapse chunks; a warp streams a chunk with 16-byte loads and
// adds each weight into W[(t + d) mod 64][target] with a fire-and-forget int32
// reduction, so the order of delivery cannot change the result.
//
// Three engines run these phases (every one gives the same raster):
//   k_step               -- pipelined (default): one kernel per step delivers step t's
//                           spikes while it finishes step t's update and decides step
//                           t+1's spikes (a spike at s depends only on spikes <= s-2);
//                           replayed from a CUDA graph with programmatic launch
//                           (batches may run in circuit groups);
//   k_update + k_deliver -- one kernel per phase, replayed from a CUDA graph (batches
//                           may run in circuit groups: k_update takes a neuron range);
//   k_persistent         -- the pipelined schedule in one cooperative launch for a
//                           batch of steps, one grid-wide barrier per step whose
//                           spin-wait is bounded (on timeout the kernel records an
//                           error and exits).
// k_deliver_list delivers a given sender list (measurement and tests); blocked records
// (target-blocked rows) have their own phase 2, k_deliver_blocked (blocked.cu).
//
// No FMA in the neuron arithmetic: __fmul_rn / __fadd_rn round every product and sum
// on its own, which is what makes the raster reproducible bit for bit.
#include <cuda_runtime.h>

#include "internal.hpp"
#include "launch.cuh"
#include "philox.cuh"

namespace snn {

namespace {

__device__ __forceinline__ void red_add_s32(int32_t *addr, int32_t v)
{
    asm volatile("red.relaxed.gpu.global.add.s32 [%0], %1;" ::"l"(addr), "r"(v) : "memory");
}

__device__ __forceinline__ uint32_t ld_acquire_u32(const uint32_t *p)
{
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ uint64_t global_ns()
{
    uint64_t v;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(v));
    return v;
}

// Streaming 16-byte load of read-once data (evict-first in L1/L2).
__device__ __forceinline__ int4 ld_stream4(const int32_t *p) { return __ldcs(reinterpret_cast<const int4 *>(p)); }
__device__ __forceinline__ uint32_t ld_stream_u32(const uint8_t *p)
{
    return __ldcs(reinterpret_cast<const unsigned int *>(p));
}

// Global warp number with consecutive numbers on consecutive CTAs, so that a short
// list of work items spreads over all SMs instead of filling the first CTAs.
__device__ __forceinline__ int64_t spread_warp()
{
    return static_cast<int64_t>(threadIdx.x >> 5) * gridDim.x + blockIdx.x;
}

__device__ __forceinline__ void red_release_add_u32(uint32_t *addr, uint32_t v)
{
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(addr), "r"(v) : "memory");
}

__device__ __forceinline__ int32_t neuron_step(const StepArgs &a, float &u, float &cur, uint32_t &r, int32_t in)
{
    int32_t spike = 0;
    if (r == 0u) {
        float x = __fadd_rn(__fmul_rn(a.p22, u), __fmul_rn(a.p21, cur));
        if (x >= a.theta) {
            spike = 1;
            x = a.u_reset;
            r = static_cast<uint32_t>(a.t_ref);
        }
        u = x;
    } else {
        u = a.u_reset;
        r -= 1u;
    }
    cur = __fadd_rn(__fmul_rn(a.p11, cur), __fmul_rn(__int2float_rn(in), 0x1p-12f));
    return spike;
}

__device__ __forceinline__ void prefetch_l2(const void *p, uint32_t bytes)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// Bytes [lo, hi) of an array of records, in whole 16-byte units.
__device__ __forceinline__ void prefetch_bytes(const void *p, int64_t lo, int64_t hi)
{
    lo &= ~int64_t{15};
    hi = (hi + 15) & ~int64_t{15};
    prefetch_l2(reinterpret_cast<const uint8_t *>(p) + lo, static_cast<uint32_t>(hi - lo));
}

// Row [rs, re) of the record store into L2 (of every array the format keeps).
__device__ __forceinline__ void prefetch_row(const StepArgs &a, int64_t rs, int64_t re)
{
    if (re <= rs) return;
    const int tb = a.format == SNN_RECORD_BLOCKED6 ? 2 : a.format == SNN_RECORD_BLOCKED8 ? 8 : 4;
    const int wb = a.format == SNN_RECORD_PLAIN9 || a.format == SNN_RECORD_BLOCKED6 ? 4
                   : a.format == SNN_RECORD_PACKED_BF16                             ? 2
                   : a.format == SNN_RECORD_PACKED_I8                               ? 1
                                                                                    : 0;
    prefetch_bytes(a.syn_tgt, rs * tb, re * tb);
    if (wb) prefetch_bytes(a.syn_w, rs * wb, re * wb);
    if (a.format == SNN_RECORD_PLAIN9) prefetch_bytes(a.syn_d, rs, re);
}


// The thalamic counts of four neurons, one byte each, from Philox counter (t, ctr): the
// first eight thresholds of the first neuron's population are read once and compared with
// all four words; a count of eight and more goes on from there, and a quad that spans two
// populations looks each neuron's up.  Not inlined: the step kernel draws in two places.
__device__ __noinline__ uint32_t draw_quad(uint64_t t, uint64_t ctr, uint64_t seed, uint32_t pops,
                                           const uint64_t *thresholds)
{
    const Block4 rnd = philox4x64_10(t, ctr, 0, 0, seed, kStreamThalamic);
    const uint64_t *thr = thresholds + (pops & 0xFFu) * kPK;
    uint32_t T[4] = {0, 0, 0, 0};
#pragma unroll
    for (int k = 0; k < 8; k += 2) {
        const ulonglong2 v2 = __ldg(reinterpret_cast<const ulonglong2 *>(thr + k));
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint64_t v = rnd.w[j] >> 1;
            T[j] += (v >= v2.x ? 1u : 0u) + (v >= v2.y ? 1u : 0u);
        }
    }
    const bool mixed = pops != (pops & 0xFFu) * 0x01010101u;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if (!mixed && T[j] < 8u) continue;
        const uint64_t v = rnd.w[j] >> 1;
        const uint64_t *own = thresholds + ((pops >> (8 * j)) & 0xFFu) * kPK;
        uint32_t c = mixed ? 0u : 8u;
        while (c < static_cast<uint32_t>(kPK) && v >= __ldg(own + c)) ++c;
        T[j] = c;
    }
    return T[0] | (T[1] << 8) | (T[2] << 16) | (T[3] << 24);
}

// The draws of step t for quad q = 32 g + lane (g: group of 128 neurons), one byte per neuron:
// the thalamic count, and kDrawValid for a neuron of a circuit (the others are inert).
// Independent of the dynamics, so a step kernel draws before it waits for the kernel before it.
constexpr uint32_t kDrawValid = 0x80u;
__device__ __forceinline__ uint32_t pipe_draws(const StepArgs &a, int64_t t, int64_t g, bool draw)
{
    const int64_t i0 = (g * 32 + (threadIdx.x & 31)) * 4;
    if (g >= a.quad_warps || i0 >= a.n) return 0u;
    CircuitInfo ci{0, a.n_all, a.seed, 0};
    if (a.n_circuits > 1) ci = a.circuits[__ldg(a.group_circuit + g)];
    uint32_t packed = 0;
    if (draw)
        packed = draw_quad(static_cast<uint64_t>(t), static_cast<uint64_t>((i0 - ci.base) >> 2), ci.seed,
                           __ldg(reinterpret_cast<const unsigned int *>(a.pop_id + i0)), a.tables->thresholds[0]);
    const int64_t left = ci.base + ci.n - i0;  // neurons of the circuit from the quad on
    return left >= 4 ? packed | kDrawValid * 0x01010101u
           : left > 0 ? packed | (kDrawValid * 0x01010101u >> (8 * (4 - left)))
                      : packed;
}

// Phase 1 for neurons 4q .. 4q+3, from their draws.  The ring row is read through L2 (other
// SMs add into it between steps).
__device__ __forceinline__ void update_quad(const StepArgs &a, int64_t t, int64_t q, uint32_t draws, int32_t spk[4])
{
    const int64_t i0 = q * 4;
    const int64_t slot = t & kDMask;
    float4 u4 = *reinterpret_cast<const float4 *>(a.U + i0);
    float4 c4 = *reinterpret_cast<const float4 *>(a.I + i0);
    const uint32_t r4 = *reinterpret_cast<const uint32_t *>(a.R + i0);
    int32_t *wrow = a.ring + slot * a.npad + i0;
    const int4 w4 = __ldcg(reinterpret_cast<const int4 *>(wrow));
    *reinterpret_cast<int4 *>(wrow) = make_int4(0, 0, 0, 0);
    float uu[4] = {u4.x, u4.y, u4.z, u4.w};
    float cc[4] = {c4.x, c4.y, c4.z, c4.w};
    const int32_t ww[4] = {w4.x, w4.y, w4.z, w4.w};
    uint32_t rr[4] = {r4 & 0xFFu, (r4 >> 8) & 0xFFu, (r4 >> 16) & 0xFFu, r4 >> 24};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const uint32_t draw = (draws >> (8 * j)) & 0xFFu;
        if (!(draw & kDrawValid)) continue;
        const int32_t in =
            static_cast<int32_t>(static_cast<uint32_t>(ww[j]) + (draw & 0x7Fu) * static_cast<uint32_t>(a.w_ext_fx));
        spk[j] = neuron_step(a, uu[j], cc[j], rr[j], in);
    }
    *reinterpret_cast<float4 *>(a.U + i0) = make_float4(uu[0], uu[1], uu[2], uu[3]);
    *reinterpret_cast<float4 *>(a.I + i0) = make_float4(cc[0], cc[1], cc[2], cc[3]);
    *reinterpret_cast<uint32_t *>(a.R + i0) = rr[0] | (rr[1] << 8) | (rr[2] << 16) | (rr[3] << 24);
}

// Warp-collective (every lane must call): append the warp's spikers to the raster, whose
// entries of this step start at `begin`, and to the step's list of rows (StepArgs::queue, by
// the step's parity), and fetch those rows into L2 for phase 2.
__device__ __forceinline__ void append_spikes(const StepArgs &a, int64_t t, int64_t i0, uint32_t begin,
                                              const int32_t spk[4])
{
    const int lane = threadIdx.x & 31;
    const int cnt = spk[0] + spk[1] + spk[2] + spk[3];
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += v;
    }
    const int total = __shfl_sync(0xFFFFFFFFu, incl, 31);
    if (total == 0) return;
    int64_t rp[5] = {0, 0, 0, 0, 0};
    if (cnt != 0) {
        const longlong2 rpa = __ldg(reinterpret_cast<const longlong2 *>(a.row_ptr + i0));
        const longlong2 rpb = __ldg(reinterpret_cast<const longlong2 *>(a.row_ptr + i0 + 2));
        rp[0] = rpa.x; rp[1] = rpa.y; rp[2] = rpb.x; rp[3] = rpb.y;
        rp[4] = __ldg(a.row_ptr + i0 + 4);
    }
    uint32_t base = 0;
    if (lane == 31) base = atomicAdd(&a.ctl->cursor, static_cast<uint32_t>(total));
    base = __shfl_sync(0xFFFFFFFFu, base, 31);
    uint32_t pos = base + static_cast<uint32_t>(incl - cnt);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if (spk[j]) {
            if (pos < a.rast_cap) {
                a.rast_nrn[pos] = static_cast<int32_t>(i0 + j);
                a.rast_t[pos] = static_cast<int32_t>(t);
            } else {
                atomicOr(&a.ctl->err, kErrRaster);
            }
            if (pos - begin < static_cast<uint32_t>(a.queue_cap)) {
                const QueueEntry e = queue_entry(rp[j], rp[j + 1], static_cast<int32_t>(i0 + j), t);
                *reinterpret_cast<int4 *>(a.queue + (t & 1) * a.npad + (pos - begin)) = *reinterpret_cast<const int4 *>(&e);
            }
            ++pos;
            prefetch_row(a, rp[j], rp[j + 1]);
        }
    }
}

// One 256-synapse chunk [off, min(off + 256, re)) of a row whose sender belongs to
// population src_pop: each lane takes two quads, loads them with 16-byte streaming
// loads and adds every weight into W[(slot + d) mod 64][target].  FMT selects the
// record format; the padding entries of a row deliver nothing.
template <int FMT>
__device__ __forceinline__ void deliver_chunk(const StepArgs &a, int64_t slot, int64_t off, int64_t re, int src_pop)
{
    const int lane = threadIdx.x & 31;
    int32_t *const ring = a.ring;
    const int64_t npad = a.npad;
    int4 tg[2];
    int4 wv[2];
    uint32_t dv[2];
    uint2 hv[2];
    bool ok[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int64_t o = off + u * 128 + lane * 4;
        ok[u] = o < re;
        if (ok[u]) {
            tg[u] = ld_stream4(a.syn_tgt + o);
            if (FMT == SNN_RECORD_PLAIN9) {
                wv[u] = ld_stream4(a.syn_w + o);
                dv[u] = ld_stream_u32(a.syn_d + o);
            } else if (FMT == SNN_RECORD_PACKED_I8) {
                dv[u] = ld_stream_u32(reinterpret_cast<const uint8_t *>(a.syn_w) + o);
            } else {
                hv[u] = __ldcs(reinterpret_cast<const uint2 *>(reinterpret_cast<const uint16_t *>(a.syn_w) + o));
            }
        }
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        if (!ok[u]) continue;
        const int32_t tt[4] = {tg[u].x, tg[u].y, tg[u].z, tg[u].w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            int32_t w, target;
            int64_t d;
            if (FMT == SNN_RECORD_PLAIN9) {
                const int32_t wq[4] = {wv[u].x, wv[u].y, wv[u].z, wv[u].w};
                w = wq[e];
                target = tt[e];
                d = (dv[u] >> (8 * e)) & 0xFFu;
            } else {
                const uint32_t word = static_cast<uint32_t>(tt[e]);
                if (word & kWordPad) continue;
                target = static_cast<int32_t>(word & kWordTargetMask);
                d = (word >> kWordDelayShift) & 63u;
                const int b = static_cast<int>((word >> kWordPopShift) & 7u);
                if (FMT == SNN_RECORD_PACKED_I8) {
                    const int2 pq = __ldg(reinterpret_cast<const int2 *>(&a.tables->i8_pair[src_pop][b]));
                    const int32_t code = static_cast<int8_t>((dv[u] >> (8 * e)) & 0xFFu);
                    w = pq.x + code * pq.y;
                } else {
                    const uint32_t h = e < 2 ? (hv[u].x >> (16 * e)) : (hv[u].y >> (16 * (e - 2)));
                    w = __float2int_rn(__fmul_rn(__uint_as_float((h & 0xFFFFu) << 16), 4096.0f));
                }
            }
            if (w != 0) red_add_s32(ring + ((slot + d) & kDMask) * npad + target, w);
        }
    }
}

// Phase 2 for the spikers list[0 .. nspk), work items grid-strided over warps:
// item = (spiker, 256-synapse chunk of its row).
// Items per spike when nspk spikes share nwarps warps: enough to keep every warp busy
// while there are few spikes (one 256-synapse chunk per item), fewer and longer items
// (consecutive chunks of one row) when spikes outnumber warps.
__device__ __forceinline__ int64_t items_per_spike(int64_t cpr, int64_t nspk, int64_t nwarps)
{
    const int64_t ipj = nspk > 0 ? nwarps / nspk : cpr;
    return ipj < 1 ? 1 : (ipj > cpr ? cpr : ipj);
}

template <int FMT>
__device__ __forceinline__ void deliver_list_fmt(const StepArgs &a, int64_t t, const int32_t *list, int64_t nspk,
                                                 int64_t warp, int64_t nwarps)
{
    const int64_t cpr = a.chunks_per_row;
    const int64_t ipj = items_per_spike(cpr, nspk, nwarps);
    const int64_t per = (cpr + ipj - 1) / ipj;  // chunks per item
    const int64_t items = nspk * ipj;
    for (int64_t it = warp; it < items; it += nwarps) {
        const int64_t j = it / ipj;
        const int64_t part = it - j * ipj;
        const int32_t s = __ldcg(list + j);
        const int64_t rs = a.row_ptr[s];
        const int64_t re = a.row_ptr[s + 1];
        const int src = FMT == SNN_RECORD_PACKED_I8 ? __ldg(a.pop_id + s) : 0;
        for (int64_t c = part * per, off = rs + c * kChunk; c < (part + 1) * per && off < re; ++c, off += kChunk)
            deliver_chunk<FMT>(a, t, off, re, src);
    }
}

__device__ __forceinline__ void deliver_list(const StepArgs &a, int64_t t, const int32_t *list, int64_t nspk,
                                             int64_t warp, int64_t nwarps)
{
    if (a.format == SNN_RECORD_PACKED_I8) deliver_list_fmt<SNN_RECORD_PACKED_I8>(a, t, list, nspk, warp, nwarps);
    else if (a.format == SNN_RECORD_PACKED_BF16) deliver_list_fmt<SNN_RECORD_PACKED_BF16>(a, t, list, nspk, warp, nwarps);
    else deliver_list_fmt<SNN_RECORD_PLAIN9>(a, t, list, nspk, warp, nwarps);
}

// Graph engine.  Both kernels start while the kernel before them drains (programmatic
// launches; t_base as in k_step) and wait for it after the part that does not depend on it.
// A step is a chain of round trips of about 0.7 us: state -> append -> count and row entry ->
// records -> ring.  A step of the half-scale circuit with BLOCKED8 records took 9.8 us in a
// graph (14.2 launched one by one); overlapping launches, rows fetched into L2 by the append
// and all warps sharing few events 7.7; the step's own list of rows, read with the count, 5.8.
__global__ void __launch_bounds__(kUpdateThreads) k_update(const StepArgs a, const int k)
{
    allow_next_grid();
    const int64_t t = a.ctl->t_base + k;
    const int64_t q = a.quad_base + static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    const uint32_t draws = pipe_draws(a, t, q >> 5, true);
    wait_previous_grid();
    const uint32_t begin = __ldcg(&a.ctl->step_begin[t & 1]);
    int32_t spk[4] = {0, 0, 0, 0};
    if (q * 4 < a.n) update_quad(a, t, q, draws, spk);
    append_spikes(a, t, q * 4, begin, spk);
}

// Delivery of the step's rows: items as in deliver_list, with the entry of a warp's first item
// read in the count's round trip.
template <int FMT>
__device__ __forceinline__ void deliver_rows_fmt(const StepArgs &a, int64_t t, int64_t nspk, int64_t warp,
                                                 int64_t nwarps, int4 first)
{
    const QueueEntry *rows = a.queue + (t & 1) * a.npad;
    const int64_t cpr = a.chunks_per_row;
    const int64_t ipj = items_per_spike(cpr, nspk, nwarps);
    const int64_t per = (cpr + ipj - 1) / ipj;
    for (int64_t it = warp; it < nspk * ipj; it += nwarps) {
        const int64_t j = it / ipj, part = it - j * ipj;
        const int4 raw = it == warp && ipj == cpr ? first : __ldcg(reinterpret_cast<const int4 *>(rows + j));
        const int64_t rs = entry_first_quad(raw.x, raw.y) * 4;
        const int64_t re = rs + static_cast<int64_t>(entry_quads(raw.y)) * 4;
        const int src = FMT == SNN_RECORD_PACKED_I8 ? __ldg(a.pop_id + raw.z) : 0;
        for (int64_t c = part * per, off = rs + c * kChunk; c < (part + 1) * per && off < re; ++c, off += kChunk)
            deliver_chunk<FMT>(a, t, off, re, src);
    }
}

__global__ void __launch_bounds__(kDeliverThreads) k_deliver(const StepArgs a, const int k)
{
    allow_next_grid();
    const int64_t t = a.ctl->t_base + k;
    const int64_t nwarps = (static_cast<int64_t>(gridDim.x) * blockDim.x) >> 5;
    const int64_t warp = spread_warp();
    const int64_t j0 = warp / a.chunks_per_row;
    wait_previous_grid();
    const uint32_t cur = __ldcg(&a.ctl->cursor);
    const uint32_t begin = __ldcg(&a.ctl->step_begin[t & 1]);
    const int4 first = j0 < a.queue_cap ? __ldcg(reinterpret_cast<const int4 *>(a.queue + (t & 1) * a.npad + j0))
                                        : make_int4(0, 0, 0, 0);
    if (blockIdx.x == 0 && threadIdx.x == 0) a.ctl->step_begin[(t + 1) & 1] = cur;
    const uint32_t end = cur < a.rast_cap ? cur : a.rast_cap;
    const int64_t nspk = end > begin ? static_cast<int64_t>(end - begin) : 0;
    if (a.format == SNN_RECORD_PACKED_I8) deliver_rows_fmt<SNN_RECORD_PACKED_I8>(a, t, nspk, warp, nwarps, first);
    else if (a.format == SNN_RECORD_PACKED_BF16) deliver_rows_fmt<SNN_RECORD_PACKED_BF16>(a, t, nspk, warp, nwarps, first);
    else deliver_rows_fmt<SNN_RECORD_PLAIN9>(a, t, nspk, warp, nwarps, first);
}

// Phase 2 alone for a caller-given list of senders (measurement and tests).
__global__ void __launch_bounds__(kDeliverThreads) k_deliver_list(const StepArgs a, const int32_t *list,
                                                                  const int64_t n, const int64_t t)
{
    const int64_t nwarps = (static_cast<int64_t>(gridDim.x) * blockDim.x) >> 5;
    deliver_list(a, t, list, n, spread_warp(), nwarps);
}

__global__ void k_advance(Ctl *ctl, int64_t m)
{
    wait_previous_grid();
    ctl->t_base += m;
}

// Circuit groups run the same steps one group after another: the next group's first
// step appends its spikes from where the raster ends now.
__global__ void k_resync(Ctl *ctl) { ctl->step_begin[ctl->t_base & 1] = ctl->cursor; }

// Grid-wide barrier of a cooperative launch: the `index`-th barrier of the launch
// waits until all gridDim.x blocks have arrived index times.  The wait is bounded by
// a.barrier_timeout_ns; on timeout the error bit is set (which releases every other
// waiting block too) and false returned.
__device__ __forceinline__ bool grid_barrier(const StepArgs &a, Ctl *ctl, uint32_t index)
{
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = 1;
        // the CTA barrier above orders the block's writes before this release
        red_release_add_u32(&ctl->bar, 1u);
        const uint32_t target = index * gridDim.x + a.barrier_extra;
        if (ld_acquire_u32(&ctl->bar) < target) {
            const uint64_t t0 = global_ns();
            uint32_t spins = 0;
            while (ld_acquire_u32(&ctl->bar) < target) {
                if ((++spins & 255u) == 0 && global_ns() - t0 > a.barrier_timeout_ns) {
                    atomicOr(&ctl->err, kErrTimeout);
                    ok = 0;
                    break;
                }
                if ((spins & 63u) == 0 && (ld_acquire_u32(&ctl->err) & kErrTimeout)) {
                    ok = 0;
                    break;
                }
            }
        }
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

// ---------------------------------------------------------------------------
// Pipelined engine: one kernel per step.
//
// In the recurrence a spike decided at step s uses I after step s-1, which already
// holds W[s-1]; W[s-1] only receives spikes of steps <= s-2.  So the spike decision
// of step t+1 (A(t+1)) needs the current update of step t (B(t): I <- p11 I + W[t] +
// T w_ext) but not the delivery of step t's spikes (D(t), which writes slots t+1 ..
// t+63 and is read from step t+1 on).  Kernel K_t therefore runs, concurrently:
//   neuron warps:   B(t) then A(t+1) for their neurons (same thread, program order);
//   delivery warps: D(t) for the spikes of step t decided by K_{t-1}.
// Each neuron still sees A(0), B(0), A(1), B(1), ... in order, so the arithmetic is
// the same as the two-phase engines.  U and R after A(s) live in buffer s mod 2 (the
// state after s steps is in buffer (s-1) mod 2).
//
// Spike queue of step s (buffer s mod 4, count qcount[s mod 4]): a warp with
// spikers reserves room with one atomic and writes their entries (row bounds were
// loaded with the neuron state).  A batch in circuit groups runs one launch per group
// and step; the group's launch covers only its own groups of 128 neurons, and its
// queues and counts are its own (queue region from the group's first neuron, counts
// in the group's slot of the count array), so the groups' kernels are independent.  The rows are prefetched into L2 for the next
// kernel.  A delivery warp loads the step's spike count and the entry of its first
// item in the same round trip, then the synapses; the warp delivering chunk 0 of spike
// j records it at raster position base + j, the raster base advancing once per step
// (Ctl::step_begin[t mod 2]).  Every buffer choice depends on t mod 64 only.
// ---------------------------------------------------------------------------

// A launch of one circuit group (kGroup) takes its queue counts, queue size and first
// group of 128 neurons from the arguments; a launch over the whole index space uses the
// control block's counts, npad entries per queue and group 0.  The two are separate
// instantiations, so that the whole-network kernel carries none of the group indirection.
template <bool kGroup>
__device__ __forceinline__ uint32_t *queue_counts(const StepArgs &a)
{
    return kGroup ? a.qcount : a.ctl->qcnt;
}
template <bool kGroup>
__device__ __forceinline__ int64_t queue_entries(const StepArgs &a)
{
    return kGroup ? a.queue_cap : a.npad;
}
template <bool kGroup>
__device__ __forceinline__ int64_t first_quad_warp(const StepArgs &a)
{
    return kGroup ? (a.quad_base >> 5) : 0;
}

// The dynamic state of a quad, loaded in one round trip.
struct QuadState {
    float4 u, c;
    uint32_t r;
    int4 w;
};

template <bool kB>
__device__ __forceinline__ void pipe_load(const StepArgs &a, int ph, int64_t g, bool valid, QuadState &s)
{
    const int64_t i0 = (g * 32 + (threadIdx.x & 31)) * 4;
    s.u = make_float4(0.f, 0.f, 0.f, 0.f);
    s.c = s.u;
    s.r = 0;
    s.w = make_int4(0, 0, 0, 0);
    if (!valid) return;
    s.u = *reinterpret_cast<const float4 *>(((ph & 1) ? a.U2 : a.U) + i0);
    s.c = *reinterpret_cast<const float4 *>(a.I + i0);
    s.r = *reinterpret_cast<const uint32_t *>(((ph & 1) ? a.R2 : a.R) + i0);
    if (kB) s.w = __ldcg(reinterpret_cast<const int4 *>(a.ring + (ph & kDMask) * a.npad + i0));
}

// Neuron part for quad q = 32 g + lane: B(t) (without kB, the first kernel: t = -1, not) then
// A(t+1), from the quad's draws and state.  Warp-collective: every lane of group g must call
// it (lanes without a quad pass valid = false).
template <bool kGroup, bool kB>
__device__ __forceinline__ void pipe_quad(const StepArgs &a, const int64_t &t, int ph, int64_t g, bool valid,
                                          uint32_t draws, const QuadState &s)
{
    const int lane = threadIdx.x & 31;
    const int64_t i0 = (g * 32 + lane) * 4;
    const int phn = ph + 1;  // phase of the step whose spikes are decided here
    int32_t spk[4] = {0, 0, 0, 0};
    if (valid) {
        float *Uout = (phn & 1) ? a.U2 : a.U;
        uint8_t *Rout = (phn & 1) ? a.R2 : a.R;
        float uu[4] = {s.u.x, s.u.y, s.u.z, s.u.w};
        float cc[4] = {s.c.x, s.c.y, s.c.z, s.c.w};
        const int32_t ww[4] = {s.w.x, s.w.y, s.w.z, s.w.w};
        uint32_t rr[4] = {s.r & 0xFFu, (s.r >> 8) & 0xFFu, (s.r >> 16) & 0xFFu, s.r >> 24};
        if (kB) *reinterpret_cast<int4 *>(a.ring + (ph & kDMask) * a.npad + i0) = make_int4(0, 0, 0, 0);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t draw = (draws >> (8 * j)) & 0xFFu;
            if (!(draw & kDrawValid)) continue;
            if (kB) {
                const int32_t in = static_cast<int32_t>(static_cast<uint32_t>(ww[j]) +
                                                        (draw & 0x7Fu) * static_cast<uint32_t>(a.w_ext_fx));
                cc[j] = __fadd_rn(__fmul_rn(a.p11, cc[j]), __fmul_rn(__int2float_rn(in), 0x1p-12f));
            }
            if (rr[j] == 0u) {
                float x = __fadd_rn(__fmul_rn(a.p22, uu[j]), __fmul_rn(a.p21, cc[j]));
                if (x >= a.theta) {
                    spk[j] = 1;
                    x = a.u_reset;
                    rr[j] = static_cast<uint32_t>(a.t_ref);
                }
                uu[j] = x;
            } else {
                uu[j] = a.u_reset;
                rr[j] -= 1u;
            }
        }
        if (kB) *reinterpret_cast<float4 *>(a.I + i0) = make_float4(cc[0], cc[1], cc[2], cc[3]);
        *reinterpret_cast<float4 *>(Uout + i0) = make_float4(uu[0], uu[1], uu[2], uu[3]);
        *reinterpret_cast<uint32_t *>(Rout + i0) = rr[0] | (rr[1] << 8) | (rr[2] << 16) | (rr[3] << 24);
    }
    // the group's spikes of step t+1 into the queue: room from one atomic per warp, the
    // spikers' row bounds in the same round trip
    const int cnt = spk[0] + spk[1] + spk[2] + spk[3];
    if (!__any_sync(0xFFFFFFFFu, cnt != 0)) return;
    int64_t rp[5] = {0, 0, 0, 0, 0};
    if (cnt != 0) {
        const longlong2 rpa = __ldg(reinterpret_cast<const longlong2 *>(a.row_ptr + i0));
        const longlong2 rpb = __ldg(reinterpret_cast<const longlong2 *>(a.row_ptr + i0 + 2));
        rp[0] = rpa.x; rp[1] = rpa.y; rp[2] = rpb.x; rp[3] = rpb.y;
        rp[4] = __ldg(a.row_ptr + i0 + 4);
    }
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += v;
    }
    uint32_t base = 0;
    if (lane == 31) base = atomicAdd(&queue_counts<kGroup>(a)[phn & 3], static_cast<uint32_t>(incl));
    base = __shfl_sync(0xFFFFFFFFu, base, 31);
    if (cnt == 0) return;
    QueueEntry *region = a.queue + (phn & 3) * a.npad + base;
    int k = incl - cnt;
    const int64_t sn = t + 1;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if (!spk[j]) continue;
        const int64_t rs = rp[j];
        const int64_t re = rp[j + 1];
        const QueueEntry e = queue_entry(rs, re, static_cast<int32_t>(i0 + j), sn);
        *reinterpret_cast<int4 *>(region + k) = *reinterpret_cast<const int4 *>(&e);
        ++k;
        prefetch_row(a, rs, re);
    }
}

// A neuron warp's groups g, g + stride, ... below a.quad_warps: the draws of its first two
// groups before `wait` (a step kernel's wait for the one before), then group by group with the
// next group's state in flight.  What bounds a step is the chain wait -> state -> spikes ->
// queue, about a microsecond per round trip; counting the Poisson thresholds and loading row
// bounds for all 128 neurons sat on it.  us per step in a graph before and after: tiny circuit
// 3.17 -> 2.50, full 3.46 -> 2.90, 4x circuit (two groups per warp) 7.91 -> 5.72, 16 circuits
// in two groups 9.82 -> 8.48.
template <bool kGroup, bool kB, bool kWait>
__device__ __forceinline__ void pipe_groups(const StepArgs &a, const int64_t &t, int ph, int64_t g, int64_t stride)
{
    const int64_t nquads = (a.n + 3) / 4;
    const int lane = threadIdx.x & 31;
    uint32_t d0 = pipe_draws(a, t, g, kB), d1 = pipe_draws(a, t, g + stride, kB);
    if (kWait) wait_previous_grid();
    if (g >= a.quad_warps) return;
    QuadState s;
    pipe_load<kB>(a, ph, g, g * 32 + lane < nquads, s);
#pragma unroll 1
    for (;;) {
        const int64_t gn = g + stride;
        const bool more = gn < a.quad_warps;
        QuadState next = s;
        if (more) pipe_load<kB>(a, ph, gn, gn * 32 + lane < nquads, next);
        pipe_quad<kGroup, kB>(a, t, ph, g, g * 32 + lane < nquads, d0, s);
        if (!more) return;
        s = next;
        g = gn;
        d0 = d1;
        d1 = pipe_draws(a, t, g + stride, kB);
    }
}

// A sender's population: outside batches from the launch's own population offsets, since a
// load of pop_id would be one more round trip between a queue entry and its weights (int8
// records of the 0.44x circuit: 3.23 -> 3.13 us per step).
__device__ __forceinline__ int sender_pop(const StepArgs &a, int32_t neuron)
{
    if (!a.pop_ranges) return __ldg(a.pop_id + neuron);
    int pop = 0;
#pragma unroll
    for (int b = 1; b < SNN_MAX_POPS; ++b) pop += neuron >= a.pop_off[b] ? 1 : 0;
    return pop;
}

// D(t), run by the delivery warps: grid-stride over (spike, 256-synapse chunk) items
// of queue t mod 4.  The count, the raster base and the first item's entry are loaded
// in one round trip.  The warp taking chunk 0 of spike j records it in the raster.
template <int FMT, bool kGroup>
__device__ __forceinline__ void pipe_deliver_fmt(const StepArgs &a, const int64_t &t, int ph, int64_t dw, int64_t ndw,
                                                 uint32_t n, uint32_t rbase, int4 first)
{
    const int lane = threadIdx.x & 31;
    const QueueEntry *qbuf = a.queue + (ph & 3) * a.npad;
    const int64_t cpr = a.chunks_per_row;
    const int64_t cap = queue_entries<kGroup>(a);
    // items are (spike, run of `per` chunks); when every item is one chunk (few spikes) the
    // entry `first` loaded before n arrived belongs to this warp's first item
    const int64_t ipj = items_per_spike(cpr, n, ndw);
    const int64_t per = (cpr + ipj - 1) / ipj;
    for (int64_t it = dw;; it += ndw) {
        const int64_t j = it / ipj;
        if (j >= cap || j >= n) break;
        const int4 raw = (it == dw && ipj == cpr) ? first : __ldcg(reinterpret_cast<const int4 *>(qbuf + j));
        const int64_t part = it - j * ipj;
        if (part == 0 && lane == 0) {
            const uint64_t pos = static_cast<uint64_t>(rbase) + static_cast<uint64_t>(j);
            if (pos < a.rast_cap) {
                a.rast_nrn[pos] = raw.z;
                a.rast_t[pos] = static_cast<int32_t>(t);
            }
        }
        const int64_t rs = entry_first_quad(raw.x, raw.y) * 4;
        const int64_t re = rs + static_cast<int64_t>(entry_quads(raw.y)) * 4;
        const int src = FMT == SNN_RECORD_PACKED_I8 ? sender_pop(a, raw.z) : 0;
        for (int64_t c = part * per, off = rs + c * kChunk; c < (part + 1) * per && off < re; ++c, off += kChunk)
            deliver_chunk<FMT>(a, ph, off, re, src);
    }
}

template <bool kGroup>
__device__ __forceinline__ void pipe_deliver(const StepArgs &a, const int64_t &t, int ph, bool leader, int64_t dw,
                                             int64_t ndw, bool wait_first)
{
    if (wait_first) wait_previous_grid();
    const uint32_t n = __ldcg(&queue_counts<kGroup>(a)[ph & 3]);
    const uint32_t rbase = __ldcg(&a.ctl->step_begin[t & 1]);
    // speculative: the entry of this warp's first item under one chunk per item, issued
    // alongside the count so both arrive in one round trip
    const int64_t j0 = dw / a.chunks_per_row;
    const int4 first = j0 < queue_entries<kGroup>(a) ? __ldcg(reinterpret_cast<const int4 *>(a.queue + (ph & 3) * a.npad + j0))
                                   : make_int4(0, 0, 0, 0);
    if (leader) {
        a.ctl->step_begin[(t + 1) & 1] = rbase + n;
        a.ctl->cursor = rbase + n;
        queue_counts<kGroup>(a)[(ph + 2) & 3] = 0;  // the queue the next kernel fills after this one
        if (static_cast<uint64_t>(rbase) + n > a.rast_cap) atomicOr(&a.ctl->err, kErrRaster);
    }
    if (a.format == SNN_RECORD_PACKED_I8)
        pipe_deliver_fmt<SNN_RECORD_PACKED_I8, kGroup>(a, t, ph, dw, ndw, n, rbase, first);
    else if (a.format == SNN_RECORD_PACKED_BF16)
        pipe_deliver_fmt<SNN_RECORD_PACKED_BF16, kGroup>(a, t, ph, dw, ndw, n, rbase, first);
    else
        pipe_deliver_fmt<SNN_RECORD_PLAIN9, kGroup>(a, t, ph, dw, ndw, n, rbase, first);
}

// t_base is read before waiting on the previous kernel: it only changes in the k_advance
// that ends a run of steps, and a run's first kernel is not a programmatic launch.
template <bool kGroup>
__global__ void __launch_bounds__(kStepMaxThreads, 2) k_step(const StepArgs a, const int k)
{
    allow_next_grid();
    const int64_t t = a.ctl->t_base + k;
    const int ph = static_cast<int>(t & (kPhasePeriod - 1));  // every buffer choice depends on this only
    const int wib = threadIdx.x >> 5;
    if (wib < a.neuron_warps) {
        pipe_groups<kGroup, true, true>(a, t, ph, first_quad_warp<kGroup>(a) + static_cast<int64_t>(wib) * gridDim.x + blockIdx.x,
                                        static_cast<int64_t>(a.neuron_warps) * gridDim.x);
    } else {
        const int dwarps = static_cast<int>(blockDim.x >> 5) - a.neuron_warps;
        const bool leader = blockIdx.x == 0 && threadIdx.x == 32 * a.neuron_warps;
        const int64_t dw = static_cast<int64_t>(wib - a.neuron_warps) * gridDim.x + blockIdx.x;
        pipe_deliver<kGroup>(a, t, ph, leader, dw, static_cast<int64_t>(dwarps) * gridDim.x, true);
    }
}

__global__ void __launch_bounds__(kStepMaxThreads, 2) k_prime(const StepArgs a)
{
    const int wib = threadIdx.x >> 5;
    if (wib >= a.neuron_warps) return;
    const int64_t t = -1;
    pipe_groups<true, false, false>(a, t, -1, (a.quad_base >> 5) + static_cast<int64_t>(wib) * gridDim.x + blockIdx.x,
                                    static_cast<int64_t>(a.neuron_warps) * gridDim.x);
}

// Persistent engine: the pipelined schedule in one cooperative launch for a run of
// steps.  Iteration t does what the step kernel K_t does (neuron warps: B(t) then
// A(t+1); delivery warps: D(t)); one bounded grid barrier between iterations stands in
// for the kernel boundary, which orders D(t)'s ring sums and A(t+1)'s queue before
// iteration t+1 reads them.  Every warp keeps its neuron groups for the whole launch.
__global__ void __launch_bounds__(kStepMaxThreads, 1) k_persistent(const StepArgs a, const int64_t n_steps)
{
    Ctl *ctl = a.ctl;
    const int64_t t0 = ctl->t_base;
    const int wib = threadIdx.x >> 5;
    const int64_t nw = static_cast<int64_t>(a.neuron_warps) * gridDim.x;
    const int dwarps = static_cast<int>(blockDim.x >> 5) - a.neuron_warps;
    const bool leader = blockIdx.x == 0 && threadIdx.x == 32 * a.neuron_warps;
    const int64_t dw = static_cast<int64_t>(wib - a.neuron_warps) * gridDim.x + blockIdx.x;
    uint32_t nbar = 0;
    for (int64_t st = 0; st < n_steps; ++st) {
        const int64_t t = t0 + st;
        const int ph = static_cast<int>(t & (kPhasePeriod - 1));
        if (wib < a.neuron_warps) {
            pipe_groups<false, true, false>(a, t, ph, static_cast<int64_t>(wib) * gridDim.x + blockIdx.x, nw);
        } else {
            pipe_deliver<false>(a, t, ph, leader, dw, static_cast<int64_t>(dwarps) * gridDim.x, false);
        }
        if (!grid_barrier(a, ctl, ++nbar)) return;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) ctl->t_base = t0 + n_steps;
}


}  // namespace

// One CTA per SM while its kStepMaxNeuronWarps neuron warps cover the network's groups of
// 128 neurons in one pass; larger networks get up to three CTAs per SM, so that a neuron
// warp walks fewer groups one after another (each group is a chain of dependent loads).
int step_grid(int num_sms, int64_t quad_warps)
{
    const int64_t per_pass = static_cast<int64_t>(kStepMaxNeuronWarps) * num_sms;
    const int64_t mult = std::min<int64_t>(3, std::max<int64_t>(1, (quad_warps + per_pass - 1) / per_pass));
    return static_cast<int>(mult * num_sms);
}

int step_threads(const StepArgs &a) { return 32 * (a.neuron_warps + a.delivery_warps); }

int prepare_step_kernel(const StepArgs &) { return 0; }

int launch_step(const StepArgs &a, int k, int grid, void *stream, bool programmatic)
{
    return a.group_launch ? launch_after(k_step<true>, grid, step_threads(a), 0, stream, programmatic, a, k)
                          : launch_after(k_step<false>, grid, step_threads(a), 0, stream, programmatic, a, k);
}

void launch_prime(const StepArgs &a, int grid, void *stream)
{
    k_prime<<<grid, step_threads(a), 0, static_cast<cudaStream_t>(stream)>>>(a);
}

int update_grid(int64_t n)
{
    const int64_t quads = (n + 3) / 4;
    return static_cast<int>((quads + kUpdateThreads - 1) / kUpdateThreads);
}

void launch_update(const StepArgs &a, int k, int grid, void *stream, bool programmatic)
{
    launch_after(k_update, grid, kUpdateThreads, 0, stream, programmatic, a, k);
}

void launch_deliver(const StepArgs &a, int k, int grid, void *stream, bool programmatic)
{
    launch_after(k_deliver, grid, kDeliverThreads, 0, stream, programmatic, a, k);
}

void launch_deliver_list(const StepArgs &a, const int32_t *list, int64_t n, int64_t t, int grid, void *stream)
{
    k_deliver_list<<<grid, kDeliverThreads, 0, static_cast<cudaStream_t>(stream)>>>(a, list, n, t);
}

int deliver_list_blocks_per_sm()
{
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_deliver_list, kDeliverThreads, 0) != cudaSuccess) return 1;
    return nb > 0 ? nb : 1;
}

void launch_advance(Ctl *ctl, int64_t m, void *stream) { launch_after(k_advance, 1, 1, 0, stream, true, ctl, m); }

void launch_resync(Ctl *ctl, void *stream) { k_resync<<<1, 1, 0, static_cast<cudaStream_t>(stream)>>>(ctl); }

int persistent_blocks_per_sm(const StepArgs &a)
{
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_persistent, step_threads(a), 0) != cudaSuccess) return 0;
    return nb;
}

int launch_persistent(const StepArgs &a, int64_t n_steps, int grid, void *stream)
{
    StepArgs args = a;
    int64_t n = n_steps;
    void *params[] = {&args, &n};
    const cudaError_t e = cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(k_persistent), dim3(grid),
                                                      dim3(step_threads(a)), params, 0,
                                                      static_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? 0 : static_cast<int>(e);
}

}  // namespace snn
