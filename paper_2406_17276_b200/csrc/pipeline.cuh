// The persistent, warp-specialised row pipeline of one CTA.
//
//   fetcher warp    asks a Source for row descriptors, several at a time and ahead of the
//                   consumers, so that the latency of obtaining work (a mailbox entry, an index load)
//                   is hidden, and hands them on in the order in which they become known;
//   issuer warp     streams each described row's chunks into the ring (bulk async copies) as
//                   stages are handed back;
//   consumer warps  make the fused pass over each row (row_topk.cuh), then hand the row's
//                   per-thread maxima and partial sums to a finisher through a slot and go
//                   straight on to the next row;
//   finisher warps  row r goes to finisher r mod kFinishers: it computes the row's winners and
//                   gives them to a Sink (for the tree build: candidates' path values and the
//                   layer's row counter);
//   layer warp      runs Sink::layer_loop (for the tree build: watches the row counters of its
//                   sequences, selects each next layer and publishes its rows); its assistants
//                   run Sink::layer_assist and share the selection's work.
//
// The chunks of consecutive rows form one stream: chunk g lives in stage g % kStages and is the
// (g / kStages)-th use of that stage, which fixes every mbarrier parity; likewise row r uses
// descriptor r % kDesc and slot r % kSlots.  Every row has the same number of chunks (V is fixed).
// All waits are bounded (common.cuh); a role that times out leaves its loop, and the others then
// time out on it in turn, so the CTA always ends.  The one wait without a clock is the layer team's
// barrier: the assistants sit there between jobs, and the layer warp, whose own waits are all
// bounded, reaches it however it leaves its loop (it then posts a last job that sends them home).
#pragma once

#include "row_topk.cuh"

namespace ot {

template <class LS>
__device__ __forceinline__ void pipeline_init(CtaCore& s, LS& layer) {
    if (threadIdx.x == 0) {
        for (int i = 0; i < kStages; ++i) { mbar_init(&s.full_bar[i], 1); mbar_init(&s.empty_bar[i], kConsumerWarps); }
        for (int i = 0; i < kSlots; ++i) { mbar_init(&s.ready_bar[i], kConsumerWarps); mbar_init(&s.free_bar[i], 1); }
        for (int i = 0; i < kDesc; ++i) { mbar_init(&s.desc_full[i], 1); mbar_init(&s.desc_empty[i], kConsumerWarps); }
        s.stop_row = 0x7FFFFFFF;
        mbar_fence_init();
    }
    for (int i = threadIdx.x; i < 4 * 256; i += kThreads) (&layer.thist[0][0])[i] = 0;
    if (threadIdx.x == 0) { layer.cache_b = -1; layer.cache_d = -1; layer.todo = 0; layer.rows_done = 0; }
    __syncthreads();
}

// ---- fetcher warp ------------------------------------------------------------------------------
// Obtaining a row costs global-memory round trips (a mailbox entry, an index load) that
// take about as long as streaming the row, so kFetchLanes lanes hold one ticket each and poll
// concurrently; the warp stays converged in one polling loop so that the lanes' round trips
// overlap.  Rows are handed on in the order in which they become known (the a-th known row goes to
// descriptor a % kDesc), never in ticket order: a ticket whose item is published late must not hold
// up a row that is ready.  Tickets are only taken while fewer than kDesc rows are between "ticket
// taken" and "descriptor read by the consumers", which bounds what a CTA keeps from the others.
//   Source::claim(i)          ticket for this CTA's i-th claim, or a negative value: no more work
//   Source::poll(ticket, dsc) 1: descriptor filled, 0: not yet, 2: the ticket turned out empty, -1: no more work
// Once a Source has said "no more work" no ticket of this CTA can still turn into a row.
constexpr int kFetchLanes = 4;
template <class Source>
__device__ void fetcher_role(CtaCore& s, Source& src, int* status, long long limit = kWaitCycles) {
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    bool holding = false;                 // this lane has a ticket
    long long ticket = 0;
    int claimed = 0, known = 0, consumed = 0;      // warp-uniform counts of this CTA's rows
    int consumed_empty = 0;                        // tickets that turned out empty
    long long t0 = clock64();
    for (int turn = 0;; ++turn) {
        // rows whose descriptors the consumers have let go of
        while (consumed < known && mbar_test_wait(&s.desc_empty[consumed % kDesc], (uint32_t)(consumed / kDesc) & 1u)) ++consumed;
        // new tickets, as far as the bound allows
        const bool want = lane < kFetchLanes && !holding;
        const unsigned wm = __ballot_sync(0xFFFFFFFFu, want);
        const int my_claim = claimed + __popc(wm & below);
        const bool take = want && my_claim - consumed_empty - consumed < kDesc;
        if (take) { ticket = src.claim(my_claim); holding = true; }
        claimed += __popc(__ballot_sync(0xFFFFFFFFu, take));
        // one poll per held ticket
        RowDesc dsc;
        dsc.row = nullptr; dsc.pphat = 0.0; dsc.b = dsc.d = dsc.slot = dsc.fsize = 0; dsc.stop = 0;
        int got = 0;
        if (holding) got = ticket < 0 ? -1 : src.poll(ticket, dsc, (turn & 15) == 15);
        if (Source::kHasEmpty) {   // an entry that was handed out but not needed: the ticket is gone, and does not count as a row in hand
            const bool empty = got == 2;
            if (empty) { holding = false; got = 0; }
            consumed_empty += __popc(__ballot_sync(0xFFFFFFFFu, empty));
        }
        const unsigned rm = __ballot_sync(0xFFFFFFFFu, got > 0), em = __ballot_sync(0xFFFFFFFFu, got < 0);
        if (got > 0) {
            const int a = known + __popc(rm & below);
            s.desc[a % kDescRing] = dsc;
            mbar_arrive(&s.desc_full[a % kDesc]);              // release: publishes the descriptor
            holding = false;
        }
        known += __popc(rm);
        if (em) {                                              // no more work: one stop marker after the last row
            if (lane == __ffs(em) - 1) {
                dsc.stop = 1;
                s.desc[known % kDescRing] = dsc;
                mbar_arrive(&s.desc_full[known % kDesc]);
            }
            return;
        }
        if (rm) t0 = clock64();
        else {
            if ((turn & 63) == 63 && clock64() - t0 > limit) { set_status(status, kErrTimeout); return; }
            __nanosleep(kPollPauseNs);
        }
    }
}

// ---- issuer warp -------------------------------------------------------------------------------
// A chunk of a row that does not start on a 16-byte boundary: the 16-byte granules that cover it are copied
// whole (they may hold the end or the start of a neighbouring row), except for those that reach beyond the
// table's logits [lo, hi): what is left of the chunk there, at most seven halves at either end of the table, the warp
// copies with ordinary loads.  The chunk starts at half vec_offset(row) of the stage.
// Measured (1999 rows of 50257 logits, B200): 2591 us with two-byte loads by the issuer warp, whose round trips
// were the bound; 71.5 us with granule copies, bound by the consumers' instructions, 61.9 (3.2 TB/s) since these were cut.
__device__ __noinline__ void copy_chunk_unaligned(uint16_t* stage, const uint16_t* src, int ne, const uint16_t* lo, const uint16_t* hi,
                                                  unsigned long long* bar) {
    const int lane = threadIdx.x & 31;
    const uintptr_t lo16 = (reinterpret_cast<uintptr_t>(lo) + 15u) & ~(uintptr_t)15u, hi16 = reinterpret_cast<uintptr_t>(hi) & ~(uintptr_t)15u;
    const uintptr_t first = reinterpret_cast<uintptr_t>(src), last = reinterpret_cast<uintptr_t>(src + ne);
    const uintptr_t base = first & ~(uintptr_t)15u;                        // address of the stage's first half
    const uintptr_t b0 = base < lo16 ? lo16 : base;
    const uintptr_t up = (last + 15u) & ~(uintptr_t)15u, b1 = up > hi16 ? hi16 : up;
    const bool bulk = b0 < b1;
    const uintptr_t head_end = bulk ? (b0 > first ? b0 : first) : last;    // [first, head_end) and [tail, last) by ordinary loads
    const uintptr_t tail = bulk ? b1 : last;
    if (head_end > first || last > tail) {
        for (uintptr_t a = first + 2u * lane; a < head_end; a += 64u) stage[(a - base) >> 1] = __ldg(reinterpret_cast<const uint16_t*>(a));
        for (uintptr_t a = tail + 2u * lane; a < last; a += 64u) stage[(a - base) >> 1] = __ldg(reinterpret_cast<const uint16_t*>(a));
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");       // before a later bulk copy overwrites these bytes
        __syncwarp();
    }
    if (lane == 0) {
        if (bulk) {
            mbar_expect_tx(bar, (uint32_t)(b1 - b0));
            bulk_load(stage + ((b0 - base) >> 1), reinterpret_cast<const void*>(b0), (uint32_t)(b1 - b0), bar);
        } else {
            mbar_arrive(bar);
        }
    }
    __syncwarp();
}

// lo / hi: the first logit of the table and the one past its last (looked at when rows are not aligned).
template <bool kAligned>
__device__ void issuer_role(CtaCore& s, int V, const uint16_t* lo, const uint16_t* hi, int* status) {
    const int lane = threadIdx.x & 31;
    const int nchunks = (V + kChunkElems - 1) / kChunkElems;
    long long g = 0;
    for (int r = 0;; ++r) {
        const int e = r % kDesc;
        if (!mbar_wait_warp(&s.desc_full[e], (uint32_t)(r / kDesc) & 1u, status)) return;
        const uint16_t* row = s.desc[r % kDescRing].row;
        const int go = s.desc[r % kDescRing].stop ? 0 : 1;
        const int nc = go ? nchunks : 1;                       // the stop marker takes one (empty) chunk slot
        for (int c = 0; c < nc; ++c, ++g) {
            const int st = (int)(g % kStages);
            if (g >= kStages && !mbar_wait_warp(&s.empty_bar[st], (uint32_t)((g / kStages) - 1) & 1u, status)) return;
            if (!go) {
                if (lane == 0) mbar_arrive(&s.full_bar[st]);
                return;
            }
            const int ne = chunk_elems(V, c);
            if (kAligned) {
                if (lane == 0) {
                    mbar_expect_tx(&s.full_bar[st], (uint32_t)ne * 2u);
                    bulk_load(&s.stage[st][0], row + (size_t)c * kChunkElems, (uint32_t)ne * 2u, &s.full_bar[st]);
                }
            } else {
                copy_chunk_unaligned(&s.stage[st][0], row + (size_t)c * kChunkElems, ne, lo, hi, &s.full_bar[st]);
            }
        }
    }
}

// ---- consumer warps ----------------------------------------------------------------------------
// A warp takes its share of a chunk out of the ring into registers and hands the stage back at once
// (so the issuer can refill it while the exponentials run); a row's descriptor is only looked at for
// its stop flag.
template <int kForm>
__device__ void consumer_role(CtaCore& s, int cwarp, int V, int* status) {
    constexpr bool kAligned = form_aligned(kForm), kLong = form_long(kForm), kTracked = form_tracked(kForm);
    const int lane = threadIdx.x & 31, tid = cwarp * 32 + lane;     // index among the consumer threads
    const int nchunks = (V + kChunkElems - 1) / kChunkElems;
    ThreadAcc acc;
    acc.reset();
    ChunkRegs ch;
    uint32_t cm = 0;                                           // tracked rows: lane c keeps the warp's maximum of chunk c
    int off = 0;                                               // half of the stage at which the row in hand starts
    long long g = 0;
    for (int r = 0;; ++r) {
        for (int c = 0; c < nchunks; ++c, ++g) {
            const int st = (int)(g % kStages);
            if (!mbar_wait_warp(&s.full_bar[st], (uint32_t)(g / kStages) & 1u, status)) return;
            if (c == 0) {
                if (s.desc[r % kDescRing].stop) {
                    if (tid == 0) s.stop_row = r;                  // the finishers poll this
                    return;
                }
                if (!kAligned) off = vec_offset(s.desc[r % kDescRing].row);
                __syncwarp();
                if (lane == 0) mbar_arrive(&s.desc_empty[r % kDesc]);      // this warp has looked at the descriptor
            }
            const int ne = chunk_elems(V, c);
            if (kAligned) chunk_take(ch, reinterpret_cast<const uint4*>(&s.stage[st][0]), ne >> 3, tid);
            else chunk_take_shifted(ch, reinterpret_cast<const uint4*>(&s.stage[st][0]), ne, off, tid);
            __syncwarp();
            if (lane == 0) mbar_arrive(&s.empty_bar[st]);          // the data is in registers: the stage is free
            chunk_chain(ch);
            if (kTracked) { const uint32_t key = chunk_key(ch); if (lane == c) cm = key; }
            const unsigned long long C2 = chunk_apply(acc, ch);
            chunk_exps<kLong>(acc, ch, C2, (ne + 7) >> 3);
        }
        // hand the row to its finisher
        const int sl = r % kSlots;
        if (r >= kSlots && !mbar_wait_warp(&s.free_bar[sl], (uint32_t)((r / kSlots) - 1) & 1u, status)) return;
        store_thread_result(s.slot[sl], acc, tid);
        if (kTracked) {
            uint32_t gm = cm;
            if (nchunks > kChunkGroups) {                          // (lanes beyond the row's chunks hold 0)
#pragma unroll
                for (int o = kChunkGroups; o < kMaxTracked; o += kChunkGroups) {
                    const uint32_t u = __shfl_down_sync(0xFFFFFFFFu, cm, o);
                    if (lane + o < kMaxTracked) gm = max(gm, u);
                }
            }
            if (lane < kChunkGroups) s.slot[sl].cmax[lane][cwarp] = (uint16_t)gm;
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&s.ready_bar[sl]);
        acc.reset();
    }
}

// ---- finisher warps ----------------------------------------------------------------------------
// Sink::row_done(const RowDesc&, const RowOut&, FinScratch&) is called by the whole warp.
template <int kForm, class Sink>
__device__ void finisher_role(CtaCore& s, Sink& sink, int fidx, int V, int k, int* status) {
    const int lane = threadIdx.x & 31;
    FinScratch& f = s.fin[fidx];
    for (int r = fidx;; r += kFinishers) {
        const int sl = r % kSlots;
        const uint32_t parity = (uint32_t)(r / kSlots) & 1u;
        // wait for the row, or learn that the stream ended before it (every lane polls)
        if (!mbar_try_wait(&s.ready_bar[sl], parity)) {
            long long t0 = 0;
            int turns = 0, ok = 1;
            while (!mbar_try_wait(&s.ready_bar[sl], parity)) {
                if (s.stop_row <= r) { ok = 0; break; }
                if ((++turns & 255) == 0) {
                    const long long now = clock64();
                    if (t0 == 0) t0 = now;
                    else if (now - t0 > kWaitCycles) { set_status(status, kErrTimeout); ok = 0; break; }
                }
            }
            if (!__all_sync(0xFFFFFFFFu, ok)) return;
        }
        const RowSlot& slot = s.slot[sl];
        const RowDesc dsc = s.desc[r % kDescRing];
        RowOut out;
        finish_row_warp<kForm>(f, slot, dsc.row, V, k, out);
        __syncwarp();
        if (lane == 0) mbar_arrive(&s.free_bar[sl]);                              // the slot can be refilled
        sink.row_done(dsc, out, f);
    }
}

// kForm: see RowForm.  lo / hi bound the table.
template <int kForm, class Smem, class Source, class Sink>
__device__ __forceinline__ void run_pipeline(Smem& sm, Source& src, Sink& sink, int V, int k, const uint16_t* lo, const uint16_t* hi, int* status) {
    CtaCore& s = sm.core;
    pipeline_init(s, sm.layer);
    grid_dependency_wait();                                // shared memory is set up; global memory from here on
    const int warp = threadIdx.x >> 5;
    if (warp < kConsumerWarps) { consumer_role<kForm>(s, warp, V, status); return; }
    const int helper = warp - kConsumerWarps;
    if (helper == kHelperIssuer) issuer_role<form_aligned(kForm)>(s, V, lo, hi, status);
    else if (helper == kHelperFetcher) fetcher_role(s, src, status);
    else if (helper == kHelperLayer) sink.layer_loop(sm.layer);
    else if (helper < kHelperFirstFinisher) sink.layer_assist(sm.layer, helper - kHelperLayer);
    else finisher_role<kForm>(s, sink, helper - kHelperFirstFinisher, V, k, status);
}

}  // namespace ot
