// K2 / K3: layer selection (the n candidates of largest path value), running E_sub(T, n) and the
// tree packer by the layer team.
//
// Selection never sorts: one count into coarse bins (or, as the fallback, a radix select on the 64-bit keys) finds the
// threshold of the "need" largest, then an ordered compaction (ballot scans) emits the kept elements in index
// order, which is exactly the storage order the method wants (candidate-index order for a layer;
// (depth, slot) order for the running top-n, which is also the packed order of the final tree).
#pragma once

#include "row_topk.cuh"

namespace ot {

constexpr int kRowMul = 31;                 // row of (token t, depth d) = (t*31 + d) mod H
__device__ __forceinline__ int row_of(int token, int depth, int H) {
    return (int)(((unsigned)token * (unsigned)kRowMul + (unsigned)depth) % (unsigned)H);     // below 2^31 (supported_cfg); in 64 bits this is 1 % of a build
}

// Mailbox item: bit 63 valid | b (15 bits) | layer d (9) | void flag (1) | frontier slot (10, from bit 22) | table row of the node to
// expand (22).  A second word at the same mailbox position carries the node's path value (bit 63
// valid; a path value is never negative).  Both words validate themselves, so a row can be expanded
// from them alone and the publisher needs no fence before writing them.
constexpr int kMaxTableRows = 1 << 22;
constexpr int kMaxLayers = 510;             // layers a build may draft: layer d+1 must fit the item's 9-bit field
__device__ __forceinline__ unsigned long long item_encode(int b, int d, int slot, int row) {
    return (1ull << 63) | ((unsigned long long)b << 48) | ((unsigned long long)d << 39) |
           ((unsigned long long)slot << 22) | (unsigned long long)row;
}

// An entry that was handed out but is not needed after all (the pruned draft reserves a layer's entries
// before it knows how many rows the layer will have): fetchers drop such a ticket.
constexpr unsigned long long kItemVoid = 1ull << 38;

__device__ __forceinline__ unsigned long long phat_word(double p) {
    return (1ull << 63) | (unsigned long long)__double_as_longlong(p);
}

// Positive doubles order like their bit patterns; +1 keeps every valid key above the "invalid" key 0.
__device__ __forceinline__ unsigned long long phat_key(double p) { return (unsigned long long)__double_as_longlong(p) + 1ull; }

__device__ __forceinline__ unsigned long long warp_or_u64(unsigned long long v) {
    const uint32_t lo = __reduce_or_sync(0xFFFFFFFFu, (uint32_t)v), hi = __reduce_or_sync(0xFFFFFFFFu, (uint32_t)(v >> 32));
    return ((unsigned long long)hi << 32) | lo;
}
__device__ __forceinline__ unsigned long long warp_and_u64(unsigned long long v) {
    const uint32_t lo = __reduce_and_sync(0xFFFFFFFFu, (uint32_t)v), hi = __reduce_and_sync(0xFFFFFFFFu, (uint32_t)(v >> 32));
    return ((unsigned long long)hi << 32) | lo;
}

// Per-sequence state and arrays in the workspace (device pointers already offset to the sequence).
struct SeqWork {
    double* cand_phat;     // [n*k, padded to a multiple of 4, 16-byte aligned]  path values of one layer's candidates (Eq. 2), slot-major
    int32_t* cand_tok;     // [n*k]
    int32_t* T_tok;        // [D*n]    drafted nodes, gid = (depth-1)*n + slot
    int32_t* T_par;        // [D*n]    slot of the parent in the previous layer
    double* T_phat;        // [D*n]
    int32_t* R;            // [2][n]   running top-n as gids in ascending order, double-buffered by layer parity
    double* E_prev;        // [1]      E of Algorithm 1
    int32_t* st;           // [8], 16-byte aligned   1: rows finished since the build began, 2: |R|
    int32_t* fmap;         // [n]      pruned draft: layer slot of the node behind each frontier row
};
enum { kStL1 = 0, kStDone = 1, kStNR = 2, kStQueue = 3, kStFront = 4 };
// 0: how the root's row was handled (top bit: decided; the rest: rows of layer 2 if its finisher grew layer 1 itself, else 0)
// 3: layer-by-layer build: entry of the queue of sequences whose rows are all in (sequence + 1)
// 4 ... 7: layer-by-layer build: where the tree stands, two 64-bit words (see Front)

struct TreeOut {           // mirrors opt_tree_out, pointers offset to the sequence
    int32_t *token, *parent, *depth;
    double* phat;
    int32_t *n_sel, *depth_reached;
    double* expected_len;
    double* esub_trace;    // may be null
};

// A candidate word that was not there yet when it was looked at is read again until it is (bounded).
// Rare, so out of line.
__device__ __noinline__ unsigned long long poll_phat_word(const unsigned long long* p, int* status, int polls = kWaitPolls) {
    unsigned long long x = ld_relaxed_u64(p);
    for (int t = 0; !(x >> 63) && t < polls; ++t) x = ld_relaxed_u64(p);
    if (!(x >> 63)) { set_status(status, kErrTimeout); x = ~0ull; }
    return x;
}
__device__ __noinline__ unsigned int poll_tok_word(const unsigned int* p, int* status, int polls = kWaitPolls) {
    unsigned int x = ld_relaxed_u32(p);
    for (int t = 0; !(x >> 31) && t < polls; ++t) x = ld_relaxed_u32(p);
    if (!(x >> 31)) { set_status(status, kErrTimeout); x = ~0u; }
    return x;
}

// ------------------------------------------------------------------------------------------------
// What the layer team's selections are made of (kTeam threads: the layer warp and its assistants;
// thread tt of the team).  Every step that loops over the candidates is split over the team;
// the decisions in between are computed by each warp for itself from the same shared-memory
// counts, so all warps take the same path and meet at the same barriers.
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ int team_excl_scan(int v, int* wtot, int tw, int& total) {
    int wt;
    const int base = warp_excl_scan(v, wt);
    if ((threadIdx.x & 31) == 0) wtot[tw] = wt;
    team_sync();
    int before = 0;
    total = 0;
#pragma unroll
    for (int q = 0; q < kTeamWarps; ++q) { const int x = wtot[q]; total += x; before += q < tw ? x : 0; }
    return base + before;
}

// Key of a candidate's path-value word (0: no such child).
__device__ __forceinline__ unsigned long long key_of_word(unsigned long long x) {
    return x == ~0ull ? 0ull : (x & 0x7FFFFFFFFFFFFFFFull) + 1ull;
}

// Threshold of the `need` largest keys among keyf(0..N); key 0 means "not an element".  key_or / key_and
// are the bitwise OR / AND over all non-zero keys (the caller folds them into the sweep that stages the keys): the
// bits on which all keys agree need no pass, and a pass whose threshold bin holds exactly the elements still needed
// ends the search.  On return the selection is {key > thr} plus the first need_eq elements (lowest indices) with
// key == thr.  Requires 1 <= need <= number of non-zero keys.  The digit counts rotate through three
// arrays that are all zero on entry: pass p counts into array p % 3 and clears the one pass p-1
// read, so one barrier per pass is enough.  Returns the array that is left non-zero (the caller
// clears it after its next barrier), or -1.
template <class LS, class KeyFn>
__device__ int team_radix_select(LS& s, KeyFn keyf, int N, int need, int tt, unsigned long long key_or, unsigned long long key_and,
                                 unsigned long long& thr, int& need_eq) {
    const int lane = threadIdx.x & 31;
    const unsigned long long diff = key_or ^ key_and;
    if (diff == 0ull) { thr = key_or; need_eq = need; return -1; }       // all elements equal
    int top = 64 - __clzll((long long)diff);                             // the low `top` bits vary
    unsigned long long prefix = top == 64 ? 0ull : ((key_or >> top) << top);
    int pass = 0;
    while (top > 0) {
        const int wbits = top < 8 ? top : 8, shift = top - wbits;
        const unsigned int dmask = (1u << wbits) - 1u;
        int* hist = s.thist[pass % 3];
        #pragma unroll 2                                   // (1: 0.3 to 1.1 % of a step more; 4: 1 to 2 % more for small layers)
        for (int i = tt; i < N; i += kTeam) {
            const unsigned long long key = keyf(i);
            const bool match = key != 0ull && (top == 64 || (key >> top) == (prefix >> top));
            if (match) atomicAdd(&hist[(int)((unsigned int)(key >> shift) & dmask)], 1);
        }
        team_sync();
        int c[8], mine = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) { c[j] = hist[lane * 8 + j]; mine += c[j]; }
        {   // the array read one pass ago is free again
            int* z = s.thist[(pass + 2) % 3];
            z[tt] = 0; z[tt + kTeam] = 0;
        }
        int incl = mine;                                   // suffix sums over lanes from the top
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int u = __shfl_down_sync(0xFFFFFFFFu, incl, o);
            if (lane + o < 32) incl += u;
        }
        const int above = incl - mine;
        const bool here = above < need && need <= incl;
        int bin = 0, nd = 0, cb = 0;
        if (here) {
            int a = above;
            bin = lane * 8;
#pragma unroll
            for (int b = 7; b >= 0; --b) {                 // highest bin whose suffix count reaches need
                if (nd == 0) {
                    if (a + c[b] >= need) { bin = lane * 8 + b; nd = need - a; cb = c[b]; }
                    else a += c[b];
                }
            }
        }
        const int src = __ffs(__ballot_sync(0xFFFFFFFFu, here)) - 1;
        bin = __shfl_sync(0xFFFFFFFFu, bin, src);
        need = __shfl_sync(0xFFFFFFFFu, nd, src);
        cb = __shfl_sync(0xFFFFFFFFu, cb, src);
        prefix |= (unsigned long long)bin << shift;
        top = shift;
        ++pass;
        if (cb == need && prefix != 0ull) { thr = prefix - 1ull; need_eq = 0; return (pass - 1) % 3; }   // the whole bin belongs
    }
    thr = prefix;
    need_eq = need;
    return (pass - 1) % 3;
}

// The words of a candidate that never came (see sweep_candidates): token 0, path value 0.
constexpr unsigned long long kLostPhat = 1ull << 63;
constexpr unsigned kLostTok = 1u << 31;
// Once a wait of a team has run out the team waits no more: the build comes to its end, with the status set.  (Inlined, n = 1024 takes 3 % more.)
__device__ __noinline__ void wait_ran_out(int job_at, int* status) {
    set_status(status, kErrTimeout);
    atomicExch(&smem_at<LayerJob>(job_at).polls, 0);
}

// Candidate words i = u * kTeam + tt (u < kW) of [first, end), into registers (all ones elsewhere); gph and gtk are the words' arrays
// shifted by `first`.  Words that are not there yet are read again, all at once, until they are (at most job.polls times), with a short
// pause so that the polling does not hold up the words themselves.  A word that never came reads as token 0 of path value 0: the layer
// has as many nodes as it was to get, and all that follows works on nodes that exist, with the status set.
template <int kW>
__device__ __forceinline__ void sweep_candidates(const unsigned long long* gph, const unsigned int* gtk, int first, int end, int tt, unsigned long long (&x)[kW],
                                                 unsigned int (&t32)[kW], LayerJob& job, int* status) {
#pragma unroll
    for (int u = 0; u < kW; ++u) {
        const int i = u * kTeam + tt;
        const bool word = i >= first && i < end;
        x[u] = word ? ld_relaxed_u64(&gph[i]) : ~0ull;
        t32[u] = word ? ld_relaxed_u32(&gtk[i]) : ~0u;
    }
    #pragma unroll 1
    for (int t = 0;; ++t) {
        bool missing = false;
#pragma unroll
        for (int u = 0; u < kW; ++u) {
            const int i = u * kTeam + tt;
            if (!(x[u] >> 63)) { x[u] = ld_relaxed_u64(&gph[i]); missing = missing || !(x[u] >> 63); }
            if (!(t32[u] >> 31)) { t32[u] = ld_relaxed_u32(&gtk[i]); missing = missing || !(t32[u] >> 31); }
        }
        if (!__any_sync(0xFFFFFFFFu, missing)) break;
        __nanosleep(20);
        if (t >= job.polls) {
            wait_ran_out(smem_offset(&job), status);
#pragma unroll
            for (int u = 0; u < kW; ++u) { if (!(x[u] >> 63)) x[u] = kLostPhat; if (!(t32[u] >> 31)) t32[u] = kLostTok; }
            break;
        }
    }
}

// A layer's candidate words, all of them read, are made zero for the rows of the next layer but one: a sequence's even and odd layers
// have arrays of their own, so the clearing need not come before the next layer is sent out, and the fence of every thread of the team
// that puts it before the rows of the layer after that (at the end of the job, after its last barrier) costs nothing: a finisher on another SM cannot
// store a word before its row has been sent out, so no clear can take a word away.  With one array the fence lay
// between selection and publication, 3.7 % of a build of 32 sequences.  (A fence on the reading side as well, in the fetcher, costs a
// step of one sequence 3 %; the finisher's store there depends on the mailbox word.)
// By `stride` threads, this one the tt-th.
__device__ __forceinline__ void clear_candidates(double* cand_phat, int32_t* cand_tok, int N, int tt, int stride) {
    #pragma unroll 1
    for (int i = tt * 2; i < N; i += 2 * stride) *reinterpret_cast<uint4*>(cand_phat + i) = make_uint4(0, 0, 0, 0);
    #pragma unroll 1
    for (int i = tt * 4; i < N; i += 4 * stride) *reinterpret_cast<uint4*>(cand_tok + i) = make_uint4(0, 0, 0, 0);
}

// The largest bin of the 1024 counts in s.thist at which at least `need` elements lie at or above; `at_or_above` is their
// number (the elements must be that many).  Every warp for itself.
template <class LS>
__device__ __forceinline__ int warp_coarse_bin(const LS& s, int need, int& at_or_above) {
    const int lane = threadIdx.x & 31;
    const int* h = &s.thist[0][0];
    int mine = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {                                               // (rotated: no bank conflicts)
        const int4 v = reinterpret_cast<const int4*>(h)[lane * 8 + ((q + lane) & 7)];
        mine += (v.x + v.y) + (v.z + v.w);
    }
    auto find = [&](int v, int want, int& above) -> int {                       // the lane in which the want-th from the top lies
        int incl = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_down_sync(0xFFFFFFFFu, incl, o);
            if (lane + o < 32) incl += u;
        }
        const unsigned hm = __ballot_sync(0xFFFFFFFFu, incl - v < want && want <= incl);
        const int src = hm ? __ffs(hm) - 1 : 0;
        above = __shfl_sync(0xFFFFFFFFu, incl - v, src);
        return src;
    };
    int a0, a1;
    const int l0 = find(mine, need, a0);
    const int c = h[l0 * 32 + lane];
    const int l1 = find(c, need - a0, a1);
    at_or_above = a0 + a1 + __shfl_sync(0xFFFFFFFFu, c, l1);
    return l0 * 32 + l1;
}
// Coarse bin of a path-value key: sixteen bins per factor of two, 1 at the top, everything below 1.125 * 2^-64 at the bottom.
constexpr int kCoarseShift = 48, kCoarseBase = 16 * 0x3FF - 1023, kFineShift = kCoarseShift - 10;
__device__ __forceinline__ int coarse_bin(unsigned long long key) {
    const int e = (int)(key >> kCoarseShift) - kCoarseBase;
    return e < 0 ? 0 : (e > 1023 ? 1023 : e);
}

// The fallback of team_pick: a radix select over the keys the team holds, key i of thread i % kTeam in s.keys[i] (N of them).
// Returns this thread's taken keys as a mask (bit u: key u * kTeam + tt).
template <class LS>
__device__ __noinline__ unsigned pick_by_radix(int at, int N, int need, int tt) {
    LS& s = smem_at<LS>(at);
    const int lane = tt & 31, tw = tt >> 5;
    team_sync();                                           // (keys written, the counts cleared)
    unsigned long long thr;
    int need_eq;
    const int dirty = team_radix_select(s, [&](int i) { return s.keys[i]; }, N, need, tt, ~0ull, 0ull, thr, need_eq);
    // ties at the threshold: lowest indices first
    unsigned take = 0, tied = 0;
    for (int u = 0; u * kTeam < N; ++u) {
        const int i = u * kTeam + tt;
        const unsigned long long key = i < N ? s.keys[i] : 0ull;
        const unsigned m = __ballot_sync(0xFFFFFFFFu, key == thr && key != 0ull);
        if (lane == 0) s.pick[u * kTeamWarps + tw] = m;
        take |= (key > thr ? 1u : 0u) << u;
        tied |= ((m >> lane) & 1u) << u;
    }
    team_sync();
    if (dirty >= 0) { s.thist[dirty][tt] = 0; s.thist[dirty][tt + kTeam] = 0; }
    const int nm = (N + kTeam - 1) / kTeam * kTeamWarps;
    int total;
    const int base = warp_excl_scan(lane < nm ? __popc(s.pick[lane]) : 0, total);
    for (int u = 0; u * kTeam < N; ++u) {
        const int before = __shfl_sync(0xFFFFFFFFu, base, u * kTeamWarps + tw) + __popc(s.pick[u * kTeamWarps + tw] & ((1u << lane) - 1u));
        if (((tied >> u) & 1u) && before < need_eq) take |= 1u << u;
    }
    team_sync();                                           // (s.pick may be written again)
    return take;
}

// Selection among keys held in registers: thread tt of the team has key[u] of element i = u * kTeam + tt (0: not an element;
// N <= kW * kTeam elements).  The `need` largest are taken, ties by lowest index (all of them when `all`).  Returns the mask of this
// thread's taken keys; the elements taken before key[u] are picked_before(s, base, u, tt), all together `total`.
// Bound by the latency of a chain of barriers, shared-memory accesses and shuffles, so there is one pass: the keys are counted into
// coarse bins of their path values, the bin in which the threshold lies is listed (a
// handful of keys) and the list is ranked.  A bin of more than kList keys (many equal path values, or values below 2^-64)
// goes to a radix select over all.  A layer of 500 candidates takes 2.3 us from its last word to its last row sent out; with a radix
// select over keys in shared memory and a compaction by contiguous stretches it took 3.9 to 9 (equal path values at the threshold).
// Steps (B200, us, before / now): n = 50, V = 32000 132.9 / 118.0; n = 64, V = 128256 274.8 / 253.3; 32 sequences pruned 208.4 / 186.6.
template <int kW, class LS>
__device__ __forceinline__ unsigned team_pick(LS& s, const unsigned long long (&key)[kW], int N, int need, bool all, int tt, int& total, int& base) {
    static_assert(kW * kTeamWarps <= 32, "one lane scans one ballot");
    const int lane = tt & 31, tw = tt >> 5;
    unsigned take = 0;
    if (all) {
#pragma unroll
        for (int u = 0; u < kW; ++u) take |= (key[u] != 0ull ? 1u : 0u) << u;
    } else {
        int* coarse = &s.thist[0][0];
        if (tt == 0) s.listn = 0;
#pragma unroll
        for (int u = 0; u < kW; ++u) if (key[u]) atomicAdd(&coarse[coarse_bin(key[u])], 1);
        team_sync();
        int S;
        const int bin = warp_coarse_bin(s, need, S);
        const int left = need - (S - coarse[bin]);         // of the bin's keys
        const unsigned long long low = bin > 0 ? (unsigned long long)(bin + kCoarseBase) << kCoarseShift : 1ull;
        const unsigned long long high = bin < 1023 ? (unsigned long long)(bin + 1 + kCoarseBase) << kCoarseShift : ~0ull;
        unsigned mid = 0;
        unsigned long long where = 0ull;                   // a byte per key: its place in the list
#pragma unroll
        for (int u = 0; u < kW; ++u) {
            if (key[u] >= high) take |= 1u << u;
            else if (key[u] >= low) {
                const int q = atomicAdd(&s.listn, 1);
                if (q < LS::kList) { s.list[q] = key[u]; s.listi[q] = u * kTeam + tt; where |= (unsigned long long)q << (8 * u); }
                mid |= 1u << u;
            }
        }
        team_sync();
#pragma unroll
        for (int q = 0; q < 1024 / (4 * kTeam); ++q) reinterpret_cast<int4*>(coarse)[q * kTeam + tt] = make_int4(0, 0, 0, 0);   // (every warp has its bin)
        const int L = s.listn;
        if (L <= left) {
            take |= mid;
        } else if (L <= LS::kList) {
            const unsigned long long a = lane < L ? s.list[lane] : 0ull, b = lane + 32 < L ? s.list[lane + 32] : 0ull;
            const int ia = lane < L ? s.listi[lane] : 0, ib = lane + 32 < L ? s.listi[lane + 32] : 0;
            int ra = 0, rb = 0;                            // listed elements that come before this lane's two
            #pragma unroll 2
            for (int e = 0; e < L; ++e) {
                const unsigned long long x = s.list[e];
                const int xi = s.listi[e];
                ra += x > a || (x == a && xi < ia) ? 1 : 0;
                rb += x > b || (x == b && xi < ib) ? 1 : 0;
            }
            const unsigned ma = __ballot_sync(0xFFFFFFFFu, lane < L && ra < left), mb = __ballot_sync(0xFFFFFFFFu, lane + 32 < L && rb < left);
#pragma unroll
            for (int u = 0; u < kW; ++u) {
                const int q = (int)(where >> (8 * u)) & 255;
                if (((mid >> u) & 1u) && (((q < 32 ? ma : mb) >> (q & 31)) & 1u)) take |= 1u << u;
            }
        } else {
#pragma unroll
            for (int u = 0; u < kW; ++u) { const int i = u * kTeam + tt; if (i < N) s.keys[i] = key[u]; }
            take = pick_by_radix<LS>(smem_offset(&s), N, need, tt);
        }
    }
#pragma unroll
    for (int u = 0; u < kW; ++u) {
        const unsigned m = __ballot_sync(0xFFFFFFFFu, (take >> u) & 1u);
        if (lane == 0) s.pick[u * kTeamWarps + tw] = m;
    }
    team_sync();
    base = warp_excl_scan(lane < kW * kTeamWarps ? __popc(s.pick[lane]) : 0, total);
    return take;
}
template <class LS>
__device__ __forceinline__ int picked_before(const LS& s, int base, int u, int tt) {       // (whole warp)
    const int m = u * kTeamWarps + (tt >> 5);
    return __shfl_sync(0xFFFFFFFFu, base, m) + __popc(s.pick[m] & ((1u << (tt & 31)) - 1u));
}

// Sends out a node of layer d of sequence b as frontier row `row` of layer d + 1 (row g0 + row of the build's running count).
__device__ __forceinline__ void publish_node(const RowQueue& q, int b, int d, unsigned g0, int row, int token, unsigned long long key, int* status) {
    if (token < 0 || token >= q.V) { set_status(status, kErrInternal); token = 0; }
    const unsigned g = g0 + (unsigned)row, e = q.by_grid.div(g), c = g - e * q.by_grid.d;
    if (e < (unsigned)q.mcap) {
        const unsigned pos = c * (unsigned)q.mcap + e;     // (below 2^31: opt_tree_create)
        st_relaxed_u64(&q.phat[pos], (1ull << 63) | (key - 1ull));
        st_relaxed_u64(&q.items[pos], item_encode(b, d + 1, row, (int)q.by_H.mod((unsigned)token * (unsigned)kRowMul + (unsigned)d)));
    } else {
        set_status(status, kErrInternal);
    }
}

// An entry of a reservation that is not needed.
__device__ __forceinline__ void void_entry(const RowQueue& q, unsigned g, int* status) {
    const unsigned e = q.by_grid.div(g), c = g - e * q.by_grid.d;
    if (e < (unsigned)q.mcap) {
        const unsigned pos = c * (unsigned)q.mcap + e;
        st_relaxed_u64(&q.phat[pos], 1ull << 63);
        st_relaxed_u64(&q.items[pos], (1ull << 63) | kItemVoid);
    } else {
        set_status(status, kErrInternal);
    }
}

// The team's part of a layer selection (N = fsize * k <= kW * kTeam): the new layer's nodes go to T, their tokens and keys to
// s.ltok / s.lkeys, and, when the job says so, their rows out (g0, the layer warp's, numbers them).  Returns nl after a last barrier.
// It starts while the layer's rows are still being finished and waits for the candidate words themselves.
template <int kW, class LS>
__device__ __noinline__ int select_layer_team(int at, int tt, unsigned g0, int* status) {
    LS& s = smem_at<LS>(at);
    const LayerJob& j = s.job;
    const int N = j.fsize * j.k, nvalid = j.fsize * j.kk, nl = nvalid < j.n ? nvalid : j.n, gid0 = (j.d - 1) * j.n;
    unsigned long long x[kW];
    unsigned int t32[kW];
    sweep_candidates<kW>(reinterpret_cast<const unsigned long long*>(j.cand_phat), reinterpret_cast<const unsigned int*>(j.cand_tok), 0, N, tt, x, t32, s.job, status);
#pragma unroll
    for (int u = 0; u < kW; ++u) x[u] = key_of_word(x[u]);
    if (tt == 0) s.job.g0 = g0;
    int total, base;
    const unsigned take = team_pick<kW>(s, x, N, nl, nl >= nvalid, tt, total, base);
#pragma unroll
    for (int u = 0; u < kW; ++u) {
        if (u * kTeam >= N) break;
        const int pos = picked_before(s, base, u, tt);
        if ((take >> u) & 1u) {
            s.ltok[pos] = t32[u] == ~0u ? -1 : (int)(t32[u] & 0x7FFFFFFFu);
            s.lkeys[pos] = x[u];
            s.gids[pos] = u * kTeam + tt;
        }
    }
    if (tt == 0 && total != nl) set_status(status, kErrInternal);
    team_sync();
    // (a node per thread from here on: with each taken candidate handled where it was found, up to kW of them one after the other
    // in a warp, this took 2.1 us for 500 candidates and 4 for 1024)
    g0 = s.job.g0;
    #pragma unroll 1
    for (int i = tt; i < nl; i += kTeam) {
        const int tok = s.ltok[i], gid = gid0 + i;
        const unsigned long long key = s.lkeys[i];
        if (j.publish) publish_node(j.queue, j.b, j.d, g0, i, tok, key, status);
        const int frow = (int)j.by_k.div((unsigned)s.gids[i]);
        j.T_tok[gid] = tok;
        j.T_par[gid] = j.fmap ? __ldcg(&j.fmap[frow]) : frow;
        j.T_phat[gid] = __longlong_as_double((long long)(key - 1ull));
    }
    team_sync();
    return nl;
}

// Key of member i of the running top-n, and its gid.
template <class LS>
__device__ __forceinline__ unsigned long long running_key(const LS& s, const LayerJob& j, int i, int& gid) {
    if (j.cached) { gid = s.rsel[i]; return phat_key(s.vals[i]); }
    gid = __ldcg(&j.Rold[i]);
    return phat_key(__ldcg(&j.T_phat[gid]));
}

// Pruned draft, and the layer at the depth limit: both halves of a layer job in one selection: the new running top-n is the n largest
// of the old one and the layer's candidates together (what a candidate outside them could add to T
// can never matter, see opt_tree_build_pruned).  Elements 0 .. nR_old are the old top-n (gids ascending), off .. off+N the
// candidate words.  Their order is tie order (shallower first, then candidate index).  On return s.rsel / s.vals hold
// the new top-n (gids ascending; also written to j.Rnew), its new members are T's nodes
// gid0 .. gid0+cnt in candidate order, and s.kept_old is the number of old members kept.  When the job says so the new members' rows
// are sent out (as frontier rows 0 .. cnt, left in fmap) and the rest of the reservation voided.  Returns |new top-n|.
template <int kW, class LS>
__device__ __noinline__ int select_running_team(int at, int tt, unsigned g0, int* status) {
    LS& s = smem_at<LS>(at);
    const LayerJob& j = s.job;
    const int N = j.fsize * j.k, nRo = j.nR_old, off = j.off, M = off + N;
    const int nvalid = j.fsize * j.kk, need = nRo + nvalid < j.n ? nRo + nvalid : j.n, gid0 = (j.d - 1) * j.n;
    const unsigned long long* gph = reinterpret_cast<const unsigned long long*>(j.cand_phat) - off;
    const unsigned int* gtk = reinterpret_cast<const unsigned int*>(j.cand_tok) - off;
    unsigned long long x[kW];
    unsigned int t32[kW];                                  // candidates: token word; old members: gid
    sweep_candidates<kW>(gph, gtk, off, M, tt, x, t32, s.job, status);
#pragma unroll
    for (int u = 0; u < kW; ++u) {
        const int i = u * kTeam + tt;
        x[u] = key_of_word(x[u]);
        if (i < nRo) { int gid; x[u] = running_key(s, j, i, gid); t32[u] = (unsigned)gid; }
    }
    if (tt == 0) s.job.g0 = g0;
    int total, base;
    const unsigned take = team_pick<kW>(s, x, M, need, nRo + nvalid <= j.n, tt, total, base);
    const int kept_old = __shfl_sync(0xFFFFFFFFu, base, off / 32);         // taken before element `off`
    if (tt == 0) s.kept_old = kept_old;
#pragma unroll
    for (int u = 0; u < kW; ++u) {
        const int i = u * kTeam + tt;
        if (u * kTeam >= M) break;
        const int pos = picked_before(s, base, u, tt);
        if ((take >> u) & 1u) {
            if (i >= off) {
                const int slot = pos - kept_old;
                s.ltok[slot] = t32[u] == ~0u ? -1 : (int)(t32[u] & 0x7FFFFFFFu);
                s.lkeys[slot] = x[u];
                s.gids[slot] = i - off;
            }
            s.rsel[pos] = i < off ? (int)t32[u] : gid0 + pos - kept_old;
            s.vals[pos] = __longlong_as_double((long long)(x[u] - 1ull));
        }
    }
    if (tt == 0 && total != need) set_status(status, kErrInternal);
    team_sync();
    const int cnt = total - kept_old, reserve = j.publish ? (nvalid < j.n ? nvalid : j.n) : cnt;
    g0 = s.job.g0;
    #pragma unroll 1
    for (int i = tt; i < reserve; i += kTeam) {
        if (i >= cnt) { void_entry(j.queue, g0 + (unsigned)i, status); continue; }
        const int tok = s.ltok[i], gid = gid0 + i;
        const unsigned long long key = s.lkeys[i];
        if (j.publish) publish_node(j.queue, j.b, j.d, g0, i, tok, key, status);
        j.T_tok[gid] = tok;
        j.T_par[gid] = __ldcg(&j.fmap[j.by_k.div((unsigned)s.gids[i])]);       // layer slot of the node behind the candidate's frontier row
        j.T_phat[gid] = __longlong_as_double((long long)(key - 1ull));
    }
    #pragma unroll 1
    for (int i = tt; i < need; i += kTeam) j.Rnew[i] = s.rsel[i];
    clear_candidates(j.cand_phat, j.cand_tok, N, tt, kTeam);
    const bool renumber = j.publish != 0;                  // (the layer warp may set up its next job once the last barrier is past)
    int32_t* const fmap = j.fmap;
    team_sync();
    if (renumber) for (int i = tt; i < cnt; i += kTeam) fmap[i] = i;       // (read above; the next job's first barrier puts it before its reads)
    return need;
}

// The same selection with every sweep over the candidate words in global memory (rare, see select_layer_team_big).
template <class LS>
__device__ __noinline__ int team_select_global(int at, const unsigned long long* gph, int N, int need, int tt) {
    LS& s = smem_at<LS>(at);
    const int tw = tt >> 5;
    unsigned long long prefix = 0ull;
    int left = need;
    team_sync();                                           // (the counts have been cleared)
    for (int shift = 56; shift >= 0; shift -= 8) {         // one digit per sweep; the counts go to s.thist[0]
        #pragma unroll 4
        for (int i = tt; i < N; i += kTeam) {
            const unsigned long long key = key_of_word(ld_relaxed_u64(&gph[i]));
            if (key != 0ull && (shift == 56 || (key >> (shift + 8)) == (prefix >> (shift + 8))))
                atomicAdd(&s.thist[0][(int)((key >> shift) & 255ull)], 1);
        }
        team_sync();
        int a = 0, b = 255;
        while (b > 0 && a + s.thist[0][b] < left) { a += s.thist[0][b]; --b; }
        left -= a;
        prefix |= (unsigned long long)b << shift;
        team_sync();
        s.thist[0][tt] = 0; s.thist[0][tt + kTeam] = 0;
        team_sync();
    }
    const unsigned long long thr = prefix;                 // the need-th largest key; `left` of its copies belong
    const int per = (N + kTeam - 1) / kTeam, lo = min(tt * per, N), hi = min(lo + per, N);
    int gt = 0, eq = 0;
    #pragma unroll 4
    for (int i = lo; i < hi; ++i) {
        const unsigned long long key = key_of_word(ld_relaxed_u64(&gph[i]));
        gt += key > thr ? 1 : 0;
        eq += key == thr && key != 0ull ? 1 : 0;
    }
    int total_eq, total;
    const int eq_before = team_excl_scan(eq, s.scan_a, tw, total_eq);
    int eq_take = left - eq_before;
    eq_take = eq_take < 0 ? 0 : (eq_take > eq ? eq : eq_take);
    int pos = team_excl_scan(gt + eq_take, s.scan_b, tw, total);
    #pragma unroll 1
    for (int i = lo; total == need && i < hi; ++i) {
        const unsigned long long key = key_of_word(ld_relaxed_u64(&gph[i]));
        bool take = key > thr;
        if (key == thr && key != 0ull && eq_take > 0) { take = true; --eq_take; }
        if (take) { s.lkeys[pos] = key; s.ltok[pos] = i; ++pos; }
    }
    return total;
}

// The team's selection for layers with more candidates than it holds in registers
// (kStageCap < N <= n*k).  Bound by the round trips of 128 threads to the candidate words in L2 (8192 of them take 3 us,
// 6 with their counting), so there are two sweeps and no more: the first counts the candidates into coarse bins of their path
// values, the second brings those at or above the bin in which the threshold lies, usually few more than n, into shared
// memory, each warp into a segment of its own; the keys of that bin are listed and the threshold is found by ranking
// them.  (If the bin is too full one more sweep splits it in 1024; if over a thousand ties or a threshold below
// 2^-64 make that useless too, or a warp's segment overflows, further sweeps read global memory once per digit.)
// Measured (two sequences, n = 512, k = 16, B200): 1059 us per step with a sweep per digit and tokens fetched one by one, 452
// with bit marks, a gather and a radix select after the second sweep, 431 with the segments; 401 then with the running top-n of
// team_pick, 378 with the rows sent out by the team as their tokens come in instead of by one warp afterwards.
template <class LS>
__device__ __noinline__ int select_layer_team_big(int at, int tt, unsigned g0, int* status) {
    LS& s = smem_at<LS>(at);
    const LayerJob& j = s.job;
    const int k = j.k;
    int32_t *const T_tok = j.T_tok, *const T_par = j.T_par;
    double* const T_phat = j.T_phat;
    const int32_t* const fmap = j.fmap;
    const int lane = threadIdx.x & 31, tw = tt >> 5;
    const int N = j.fsize * k;
    const int nvalid = j.fsize * j.kk;
    const int nl = nvalid < j.n ? nvalid : j.n;
    const int gid0 = (j.d - 1) * j.n;
    double* const cand_phat = j.cand_phat;
    int32_t* const cand_tok = j.cand_tok;
    const unsigned long long* gph = reinterpret_cast<const unsigned long long*>(cand_phat);
    const unsigned int* gtk = reinterpret_cast<const unsigned int*>(cand_tok);
    int* coarse = &s.thist[0][0];
    if (tt == 0) { s.listn = 0; s.job.g0 = g0; }
    #pragma unroll 1
    for (int i0 = tt; i0 - tt < N; i0 += 8 * kTeam) {
        unsigned long long x[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) x[u] = i0 + u * kTeam < N ? ld_relaxed_u64(&gph[i0 + u * kTeam]) : ~0ull;
        // what is not written yet is read again, all of it at once (bounded)
        #pragma unroll 1
        for (int t = 0;; ++t) {
            bool missing = false;
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (!(x[u] >> 63)) { x[u] = ld_relaxed_u64(&gph[i0 + u * kTeam]); missing = missing || !(x[u] >> 63); }
            if (!__any_sync(0xFFFFFFFFu, missing)) break;
            if (t >= j.polls) {
                wait_ran_out(smem_offset(&s.job), status);
#pragma unroll
                for (int u = 0; u < 8; ++u) if (!(x[u] >> 63)) x[u] = kLostPhat;
                break;
            }
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const unsigned long long key = key_of_word(x[u]);
            if (key) atomicAdd(&coarse[coarse_bin(key)], 1);
        }
    }
    team_sync();
    int S;
    const int bin = warp_coarse_bin(s, nl, S);
    unsigned long long low = bin > 0 ? (unsigned long long)(bin + kCoarseBase) << kCoarseShift : 1ull;      // what counts is at or above this key
    unsigned long long high = bin < 1023 ? (unsigned long long)(bin + 1 + kCoarseBase) << kCoarseShift : ~0ull;
    int over = S - coarse[bin];                            // candidates at or above `high`
    if (S > LS::kSurvivors && bin > 0) {
        team_sync();
        #pragma unroll
        for (int q = 0; q < 1024 / kTeam; ++q) coarse[q * kTeam + tt] = 0;
        team_sync();
        #pragma unroll 1
        for (int i0 = tt; i0 < N; i0 += 8 * kTeam) {
            unsigned long long x[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) x[u] = i0 + u * kTeam < N ? ld_relaxed_u64(&gph[i0 + u * kTeam]) : ~0ull;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const unsigned long long key = key_of_word(x[u]);
                if (key && coarse_bin(key) == bin) atomicAdd(&coarse[(int)((key >> kFineShift) & 1023ull)], 1);
            }
        }
        team_sync();
        const int sub = warp_coarse_bin(s, nl - over, S);
        S += over;
        over = S - coarse[sub];
        low |= (unsigned long long)sub << kFineShift;
        high = low + (1ull << kFineShift);
    }
    // second sweep
    constexpr int kSeg = LS::kSurvivors / kTeamWarps;
    auto put_index = [&](int at_v, int i) { if (LS::kWideGids) s.gids[at_v] = i; else s.index16[at_v] = (uint16_t)i; };
    auto index_at = [&](int at_v) -> int { return LS::kWideGids ? s.gids[at_v] : (int)s.index16[at_v]; };
    const unsigned below = (1u << lane) - 1u;
    const int per = (((N + kTeamWarps - 1) / kTeamWarps) + 255) & ~255;        // candidates per warp
    const int lo = min(tw * per, N), hi = min(lo + per, N);
    int mine = 0;
    #pragma unroll 1
    for (int i0 = lo; i0 < hi; i0 += 256) {
        unsigned long long x[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) x[u] = i0 + u * 32 + lane < hi ? ld_relaxed_u64(&gph[i0 + u * 32 + lane]) : ~0ull;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const unsigned long long key = key_of_word(x[u]);
            const unsigned m = __ballot_sync(0xFFFFFFFFu, key >= low);
            const int pos = mine + __popc(m & below);
            if (key >= low && pos < kSeg) {
                s.keys[tw * kSeg + pos] = key;
                put_index(tw * kSeg + pos, i0 + u * 32 + lane);
            }
            mine += __popc(m);
        }
    }
    if (lane == 0) s.scan_c[tw] = mine;
    team_sync();
    #pragma unroll
    for (int q = 0; q < 1024 / kTeam; ++q) coarse[q * kTeam + tt] = 0;         // (every warp has its bin)
    int start[kTeamWarps];                                 // survivors before each warp's segment
    bool fits = true;
    S = 0;
#pragma unroll
    for (int q = 0; q < kTeamWarps; ++q) { start[q] = S; const int c = s.scan_c[q]; fits = fits && c <= kSeg; S += c; }
    int total = 0;
    if (fits) {
        auto at_of = [&](int v) -> int {                   // survivor v, in index order: its place
            int q = 0;
#pragma unroll
            for (int e = 1; e < kTeamWarps; ++e) q = v >= start[e] ? e : q;
            int st = start[0];
#pragma unroll
            for (int e = 1; e < kTeamWarps; ++e) st = q == e ? start[e] : st;
            return q * kSeg + v - st;
        };
        const int mper = (S + kTeam - 1) / kTeam, v0 = min(tt * mper, S), v1 = min(v0 + mper, S);
        unsigned long long thr = low - 1ull;               // all of them
        int need_eq = 0, dirty = -1, L = 0;
        if (nl < S) {
            #pragma unroll 1
            for (int v = v0; v < v1; ++v) {
                const unsigned long long key = s.keys[at_of(v)];
                if (key < high) { const int q = atomicAdd(&s.listn, 1); if (q < LS::kList) s.list[q] = key; }
            }
            team_sync();
            L = s.listn;
        }
        if (nl < S && L <= LS::kList) {
            const int need = nl - over;
            const unsigned long long a = lane < L ? s.list[lane] : 0ull, b = lane + 32 < L ? s.list[lane + 32] : 0ull;
            int ga = 0, gb = 0, ea = 0, eb = 0;            // keys above / equal to this lane's two
            #pragma unroll 2
            for (int e = 0; e < L; ++e) {
                const unsigned long long x = s.list[e];
                ga += x > a ? 1 : 0; ea += x == a ? 1 : 0;
                gb += x > b ? 1 : 0; eb += x == b ? 1 : 0;
            }
            const bool ha = a != 0ull && ga < need && need <= ga + ea, hb = b != 0ull && gb < need && need <= gb + eb;
            const unsigned hm = __ballot_sync(0xFFFFFFFFu, ha || hb);
            const int src = hm ? __ffs(hm) - 1 : 0;
            thr = __shfl_sync(0xFFFFFFFFu, ha ? a : b, src);
            need_eq = __shfl_sync(0xFFFFFFFFu, need - (ha ? ga : gb), src);
        } else if (nl < S) {
            dirty = team_radix_select(s, [&](int v) { return s.keys[at_of(v)]; }, S, nl, tt, ~0ull, 0ull, thr, need_eq);
        }
        int gt = 0, eq = 0;
        #pragma unroll 1
        for (int v = v0; v < v1; ++v) { const unsigned long long key = s.keys[at_of(v)]; gt += key > thr ? 1 : 0; eq += key == thr ? 1 : 0; }
        int total_eq, eq_take = 0;
        if (need_eq > 0) {
            const int eq_before = team_excl_scan(eq, s.scan_a, tw, total_eq);
            eq_take = need_eq - eq_before;
            eq_take = eq_take < 0 ? 0 : (eq_take > eq ? eq : eq_take);
        }
        int pos = team_excl_scan(gt + eq_take, s.scan_b, tw, total);
        if (dirty >= 0) { s.thist[dirty][tt] = 0; s.thist[dirty][tt + kTeam] = 0; }
        #pragma unroll 1
        for (int v = v0; total == nl && v < v1; ++v) {
            const int at_v = at_of(v);
            const unsigned long long key = s.keys[at_v];
            bool take = key > thr;
            if (key == thr && eq_take > 0) { take = true; --eq_take; }
            if (take) { s.lkeys[pos] = key; s.ltok[pos] = index_at(at_v); ++pos; }
        }
    } else {
        total = team_select_global<LS>(at, gph, N, nl, tt);
    }
    // s.ltok[i] is the candidate index of the new layer's node i, s.lkeys[i] its key
    if (total != nl) {                                     // (words that came between the sweeps, after a wait that ran out: nothing was taken)
        for (int i = tt; i < nl; i += kTeam) { s.ltok[i] = 0; s.lkeys[i] = phat_key(0.0); }
        if (tt == 0) set_status(status, kErrInternal);
    }
    team_sync();
    g0 = s.job.g0;
    #pragma unroll 1
    for (int i0 = tt; i0 < nl; i0 += 4 * kTeam) {
        int c[4];
        unsigned int t32[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            c[u] = i0 + u * kTeam < nl ? s.ltok[i0 + u * kTeam] : 0;
            t32[u] = ld_relaxed_u32(&gtk[c[u]]);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = i0 + u * kTeam;
            if (i >= nl) break;
            if (!(t32[u] >> 31)) t32[u] = poll_tok_word(&gtk[c[u]], status, j.polls);
            const int tok = t32[u] == ~0u ? 0 : (int)(t32[u] & 0x7FFFFFFFu);        // (all ones: it never came)
            if (j.publish) publish_node(j.queue, j.b, j.d, g0, i, tok, s.lkeys[i], status);
            const int frow = (int)j.by_k.div((unsigned)c[u]);
            T_tok[gid0 + i] = tok;
            T_par[gid0 + i] = fmap ? __ldcg(&fmap[frow]) : frow;
            T_phat[gid0 + i] = __longlong_as_double((long long)(s.lkeys[i] - 1ull));
            s.ltok[i] = tok;
        }
    }
    team_sync();
    return nl;
}

// A layer job's selection (kind 1) and the one over the running top-n and the candidates together (kind 2), by size.
template <class LS>
__device__ __forceinline__ void select_job(int at, int tt, unsigned g0, int* status) {
    const LayerJob& j = smem_at<LS>(at).job;
    const int N = j.fsize * j.k;
    if (N <= 4 * kTeam) select_layer_team<4, LS>(at, tt, g0, status);
    else if (N <= kStageCap) select_layer_team<8, LS>(at, tt, g0, status);
    else select_layer_team_big<LS>(at, tt, g0, status);
}
template <class LS>
__device__ __forceinline__ int running_job(int at, int tt, unsigned g0, int* status) {
    const LayerJob& j = smem_at<LS>(at).job;
    return j.off + j.fsize * j.k <= 4 * kTeam ? select_running_team<4, LS>(at, tt, g0, status) : select_running_team<8, LS>(at, tt, g0, status);
}

// Once per sequence, when it is finished: T_opt = the running top-n (s.rsel / s.vals, already in
// (depth, parent's index, sibling rank) order), packed with parent indices.  By `stride` threads, this
// one the tt-th: the team, or the layer warp alone for trees so small that handing them over costs more (see kPackAlone).
template <class LS>
__device__ __noinline__ void pack_tree(int at, TreeOut out, int tt, int stride, int* status) {
    LS& s = smem_at<LS>(at);
    const LayerJob& j = s.job;
    const int d = j.d, nR = j.nR_old, n = j.n, max_depth = j.max_depth;
    const int32_t *const T_tok = j.T_tok, *const T_par = j.T_par;
    if (out.esub_trace) for (int i = d + tt; i < max_depth; i += stride) out.esub_trace[i] = 0.0;
    #pragma unroll 1
    for (int i = tt; i < n; i += stride) {
        int32_t tok = -1, par = -1, dep = 0;
        double ph = 0.0;
        if (i < nR) {
            const int gid = s.rsel[i];
            dep = gid / n + 1;
            tok = __ldcg(&T_tok[gid]);
            ph = s.vals[i];
            if (dep > 1) {
                const int pg = (dep - 2) * n + __ldcg(&T_par[gid]);
                int lo = 0, hi = i;                        // the parent is packed before its child
                while (lo < hi) {
                    const int mid = (lo + hi) >> 1;
                    if (s.rsel[mid] < pg) lo = mid + 1; else hi = mid;
                }
                if (lo >= i || s.rsel[lo] != pg) set_status(status, kErrInternal);   // closure violated
                par = lo;
            }
        }
        out.token[i] = tok; out.parent[i] = par; out.depth[i] = dep; out.phat[i] = ph;
    }
    if (tt == 0) { *out.n_sel = nR; *out.depth_reached = d; *out.expected_len = s.last_esub; }
}

// E_sub(T, n) from the running top-n in the scratch, in one fixed order (lanes stride the packed order); whole warp.
template <class LS>
__device__ __forceinline__ double running_esub(const LS& s, int nR) {
    double part = 0.0;
    #pragma unroll 1
    for (int i = threadIdx.x & 31; i < nR; i += 32) part += s.vals[i];
    return warp_sum(part);
}

// Layer job, second half: the running top-n with the new layer (j.fsize nodes, left in s by the selection): the n largest of the
// old one and the layer.  j.cached: s.rsel / s.vals still hold the old one (else it is read from j.Rold).  On return s.rsel / s.vals
// hold the new one (ascending gids; also written to j.Rnew); returns |R|.  Clears the layer's candidate words on the way.
template <int kW, class LS>
__device__ __forceinline__ int update_running(LS& s, int tt, int* status) {
    const LayerJob& j = s.job;
    clear_candidates(j.cand_phat, j.cand_tok, j.ncand, tt, kTeam);
    const int nRo = j.nR_old, NR = nRo + j.fsize, need = NR < j.n ? NR : j.n, gid0 = (j.d - 1) * j.n;
    unsigned long long key[kW];
    int gid[kW];
#pragma unroll
    for (int u = 0; u < kW; ++u) {
        const int i = u * kTeam + tt;
        key[u] = 0ull; gid[u] = 0;
        if (i >= NR) continue;
        if (i < nRo) key[u] = running_key(s, j, i, gid[u]);
        else { gid[u] = gid0 + (i - nRo); key[u] = s.lkeys[i - nRo]; }
    }
    int total, base;
    const unsigned take = team_pick<kW>(s, key, NR, need, NR <= j.n, tt, total, base);
#pragma unroll
    for (int u = 0; u < kW; ++u) {
        if (u * kTeam >= NR) break;
        const int pos = picked_before(s, base, u, tt);
        if ((take >> u) & 1u) {
            j.Rnew[pos] = gid[u];
            s.rsel[pos] = gid[u];
            s.vals[pos] = __longlong_as_double((long long)(key[u] - 1ull));
        }
    }
    if (tt == 0 && total != need) set_status(status, kErrInternal);
    team_sync();
    return need;
}

// The same with the keys in shared memory, for more of them than the team holds in registers (node budgets beyond 512).
template <class LS>
__device__ __noinline__ int update_running_staged(int at, int tt, int* status) {
    LS& s = smem_at<LS>(at);
    const LayerJob& j = s.job;
    clear_candidates(j.cand_phat, j.cand_tok, j.ncand, tt, kTeam);
    int32_t* const Rnew = j.Rnew;
    const int lane = tt & 31, tw = tt >> 5;
    const int nRo = j.nR_old, NR = nRo + j.fsize, need = NR < j.n ? NR : j.n, gid0 = (j.d - 1) * j.n;
    unsigned long long ko = 0ull, ka = ~0ull;
    #pragma unroll 1
    for (int i = tt; i < NR; i += kTeam) {
        int gid;
        unsigned long long key;
        if (i >= nRo) { gid = gid0 + (i - nRo); key = s.lkeys[i - nRo]; }
        else key = running_key(s, j, i, gid);
        s.gids[i] = gid;
        s.keys[i] = key;
        ko |= key; ka &= key;
    }
    ko = warp_or_u64(ko); ka = warp_and_u64(ka);
    if (lane == 0) { s.red_or[tw] = ko; s.red_and[tw] = ka; }
    team_sync();
    ko = 0ull; ka = ~0ull;
#pragma unroll
    for (int q = 0; q < kTeamWarps; ++q) { ko |= s.red_or[q]; ka &= s.red_and[q]; }
    unsigned long long thr = 0ull;                         // (keys are never 0: all are taken when nothing has to be left out)
    int need_eq = 0, dirty = -1;
    auto staged = [&](int i) { return s.keys[i]; };
    if (need < NR) dirty = team_radix_select(s, staged, NR, need, tt, ko, ka, thr, need_eq);
    const int per = (NR + kTeam - 1) / kTeam, lo = min(tt * per, NR), hi = min(lo + per, NR);
    int gt = 0, eq = 0;
    #pragma unroll 1
    for (int i = lo; i < hi; ++i) { const unsigned long long key = s.keys[i]; gt += key > thr ? 1 : 0; eq += key == thr ? 1 : 0; }
    int total_eq, total, eq_take = 0;
    if (need_eq > 0) {
        const int eq_before = team_excl_scan(eq, s.scan_a, tw, total_eq);
        eq_take = need_eq - eq_before;
        eq_take = eq_take < 0 ? 0 : (eq_take > eq ? eq : eq_take);
    }
    int pos = team_excl_scan(gt + eq_take, s.scan_b, tw, total);
    if (dirty >= 0) { s.thist[dirty][tt] = 0; s.thist[dirty][tt + kTeam] = 0; }
    #pragma unroll 1
    for (int i = lo; i < hi; ++i) {
        const unsigned long long key = s.keys[i];
        bool take = key > thr;
        if (key == thr && eq_take > 0) { take = true; --eq_take; }
        if (!take) continue;
        Rnew[pos] = s.gids[i];
        s.rsel[pos] = s.gids[i];
        s.vals[pos] = __longlong_as_double((long long)(key - 1ull));
        ++pos;
    }
    if (total != need) set_status(status, kErrInternal);
    team_sync();
    return need;
}

template <class LS>
__device__ __noinline__ int update_running_team(int at, int tt, int* status) {
    LS& s = smem_at<LS>(at);
    const int NR = s.job.nR_old + s.job.fsize;
    if (NR <= 4 * kTeam) return update_running<4>(s, tt, status);
    if (LS::kBudget > 2 * kTeam && NR <= 8 * kTeam) return update_running<8>(s, tt, status);
    return update_running_staged<LS>(at, tt, status);
}

}  // namespace ot
