// OPT-Tree draft-tree construction, tree mask and greedy verification for B200 (sm_100a):
// kernels and the C ABI declared in include/opt_tree.h.
#include "../../include/opt_tree.h"

#include <cuda_runtime.h>
#include <math.h>
#include <new>
#include <stdio.h>
#include <string.h>

#include "pipeline.cuh"
#include "select.cuh"

namespace ot {

constexpr int kSmallThreads = 256;          // block size of the mask / init kernels
// Verify: one CTA per target row, a thread keeps eight 16-byte loads in flight.  With 128 threads sixteen CTAs fit an
// SM, so the n + 1 rows of 32 sequences (c4: 2080 CTAs) are all resident at once instead of in two uneven waves.  Fewer
// rows are bound by the round trips of a CTA's loop (32000 logits: four of them with 128 threads, one with 512) and take
// wider CTAs as long as all are resident: 512 threads up to three rows per SM, 256 up to eight (sampled: six).
// Measured (B200, us with 128 / 256 / 512 threads): 65 rows of 128256 logits greedy 24.9 / 15.5 / 12.5; 244 rows of 32000
// greedy - / 9.4 / 8.6, sampled - / 13.4 / 12.3; 488 rows 12.2 / 10.5 / 13.1 and 20.2 / 17.0 / 18.7; 784 rows 14.0 / 12.1 / - and
// 22.4 / 20.8 / -; 1026 rows 15.9 / 14.6 / - and 26.2 / 27.9 / -.
constexpr int kVerifyMany = 128, kVerifySome = 256, kVerifyFew = 512;

// ------------------------------------------------------------------------------------------------
// Workspace
// ------------------------------------------------------------------------------------------------
struct Workspace {
    // build
    double* cand_phat;     // [B][2][cand_stride]   even and odd layers
    int32_t* cand_tok;     // [B][2][cand_stride]
    int32_t* T_tok;        // [B][D*n]
    int32_t* T_par;        // [B][D*n]
    double* T_phat;        // [B][D*n]
    int32_t* R;            // [B][2][n]
    double* E_prev;        // [B]
    int32_t* st;           // [B][8]
    int32_t* fmap;         // [B][n]   pruned draft: layer slot behind each frontier row
    // layer-by-layer build (logits handed in per layer)
    double* front_phat;    // [B][2][n]   path values of the nodes whose logits come next (even and odd layers)
    // row mailboxes of the build: one per CTA, filled by the layer warps, never wrapped within a build.
    // The rows of a build are numbered by one running count (q_ctl[kQCursor]): row g goes to CTA
    // g % grid, entry g / grid of its mailbox.
    unsigned long long* mb_items;  // [grid][mcap]  one item per (sequence, layer, frontier slot)
    unsigned long long* mb_phat;   // [grid][mcap]  bit 63 valid | bits of the node's path value (a double >= 0)
    int32_t* q_ctl;        // [8]  2: sequences finished, 3: all done, 4: rows numbered so far
    // verify
    int32_t* g;            // [B][n+1]  target argmax after the root (0) and after node i (i+1)
    int32_t* vdone;        // [B]
    int32_t* status;       // [1]
    // device copies of inputs / outputs for the host-buffer step
    int32_t *h_root, *h_base;                          // [B]
    int32_t *o_token, *o_parent, *o_depth; double* o_phat;
    int32_t *o_nsel, *o_dreach; double* o_elen;
    uint64_t* o_mask; int32_t* o_pos;
    int32_t *o_alen, *o_atok, *o_anode, *o_next;
};
enum { kQFinished = 2, kQDone = 3, kQCursor = 4, kQCall = 5, kQLeft = 6,    // 5, 6: layer-by-layer build: steps since the beginning, CTAs that have left this one
       kQTail = 0, kQHead = 1 };    // and sequences put into / taken from the queue of those whose rows are all in

constexpr int kMaxGrid = 4096;              // CTAs of the persistent kernels (SMs x occupancy) this layout supports

// Consecutive rows go to consecutive CTAs, so a CTA receives its even share of all rows of a build
// (one root and at most Dcap layers of n rows per sequence); its mailbox holds them all.
static size_t mailbox_capacity(const opt_tree_config& c, int grid) {
    const size_t Dcap = c.max_depth < c.n ? c.max_depth : c.n;
    const size_t rows = (size_t)c.max_batch * (1 + Dcap * (size_t)c.n);
    // + 8: a fetcher takes a few tickets beyond the last row it will ever get; those must stay inside
    return (rows + grid - 1) / grid + 8;
}

// Entries per sequence in the candidate arrays: n*k rounded up to a multiple of four (16-byte vectors).
static size_t cand_stride(int n, int k) { return ((size_t)n * k + 3) & ~(size_t)3; }

struct Layout {
    size_t total = 0;
    template <class T> size_t take(size_t count) {
        size_t off = (total + 255) & ~(size_t)255;
        total = off + count * sizeof(T);
        return off;
    }
};

static size_t carve(const opt_tree_config& c, int grid, char* base, Workspace* w) {
    const size_t B = c.max_batch, n = c.n, D = c.max_depth, W = (c.n + 63) / 64;
    const size_t cs = cand_stride(c.n, c.k);
    Layout L;
    size_t o;
#define OT_TAKE(field, T, count) o = L.take<T>(count); if (w) w->field = reinterpret_cast<T*>(base + o);
    OT_TAKE(cand_phat, double, 2 * B * cs)
    OT_TAKE(cand_tok, int32_t, 2 * B * cs)
    OT_TAKE(T_tok, int32_t, B * D * n)
    OT_TAKE(T_par, int32_t, B * D * n)
    OT_TAKE(T_phat, double, B * D * n)
    OT_TAKE(R, int32_t, B * 2 * n)
    OT_TAKE(E_prev, double, B)
    OT_TAKE(st, int32_t, B * 8)
    OT_TAKE(fmap, int32_t, B * n)
    OT_TAKE(front_phat, double, 2 * B * n)
    OT_TAKE(mb_items, unsigned long long, mailbox_capacity(c, grid) * grid)
    OT_TAKE(mb_phat, unsigned long long, mailbox_capacity(c, grid) * grid)
    OT_TAKE(q_ctl, int32_t, 8)
    OT_TAKE(g, int32_t, B * (n + 1))
    OT_TAKE(vdone, int32_t, B)
    OT_TAKE(status, int32_t, 1)
    OT_TAKE(h_root, int32_t, B)
    OT_TAKE(h_base, int32_t, B)
    OT_TAKE(o_token, int32_t, B * n)
    OT_TAKE(o_parent, int32_t, B * n)
    OT_TAKE(o_depth, int32_t, B * n)
    OT_TAKE(o_phat, double, B * n)
    OT_TAKE(o_nsel, int32_t, B)
    OT_TAKE(o_dreach, int32_t, B)
    OT_TAKE(o_elen, double, B)
    OT_TAKE(o_mask, uint64_t, B * n * W)
    OT_TAKE(o_pos, int32_t, B * n)
    OT_TAKE(o_alen, int32_t, B)
    OT_TAKE(o_atok, int32_t, B * (D + 1))
    OT_TAKE(o_anode, int32_t, B * D)
    OT_TAKE(o_next, int32_t, B)
#undef OT_TAKE
    return (L.total + 255) & ~(size_t)255;
}

struct Params {            // by-value kernel parameters
    int V, H, n, k, kk, Dcap, max_depth, B;
    float delta;
    int aligned;
    int mcap, grid, cstride;
    FixedDiv by_grid, by_H, by_k;
    int prune;             // draft only from layer nodes that are still among the n largest
};

__device__ __forceinline__ RowQueue row_queue(const Workspace& w, const Params& p) {
    return RowQueue{w.mb_items, w.mb_phat, p.by_grid, p.by_H, p.mcap, p.V};
}

// What is the same for all jobs of a launch.
__device__ __forceinline__ void set_job_constants(LayerJob& j, const Workspace& w, const Params& p) {
    j.n = p.n; j.k = p.k; j.kk = p.kk; j.max_depth = p.max_depth; j.polls = kWaitPolls;
    j.queue = row_queue(w, p);
    j.by_k = p.by_k;
}

// d: the layer whose candidates are meant.
__device__ __forceinline__ SeqWork seq_work(const Workspace& w, const Params& p, int b, int d) {
    SeqWork s;
    s.cand_phat = w.cand_phat + ((size_t)b * 2 + (d & 1)) * p.cstride;
    s.cand_tok = w.cand_tok + ((size_t)b * 2 + (d & 1)) * p.cstride;
    s.T_tok = w.T_tok + (size_t)b * p.max_depth * p.n;
    s.T_par = w.T_par + (size_t)b * p.max_depth * p.n;
    s.T_phat = w.T_phat + (size_t)b * p.max_depth * p.n;
    s.R = w.R + (size_t)b * 2 * p.n;
    s.E_prev = w.E_prev + b;
    s.st = w.st + (size_t)b * 8;
    s.fmap = w.fmap + (size_t)b * p.n;
    return s;
}
__device__ __forceinline__ TreeOut tree_out(const opt_tree_out& o, const Params& p, int b) {
    TreeOut t;
    t.token = o.token + (size_t)b * p.n;
    t.parent = o.parent + (size_t)b * p.n;
    t.depth = o.depth + (size_t)b * p.n;
    t.phat = o.phat + (size_t)b * p.n;
    t.n_sel = o.n_sel + b;
    t.depth_reached = o.depth_reached + b;
    t.expected_len = o.expected_len + b;
    t.esub_trace = o.esub_trace ? o.esub_trace + (size_t)b * p.max_depth : nullptr;
    return t;
}

// ------------------------------------------------------------------------------------------------
// Kernels
// ------------------------------------------------------------------------------------------------
// Clears the mailboxes, sends the root row of sequence b to CTA b % grid and resets the per-sequence state.
// The build kernel that follows may come up meanwhile: it sets up its shared memory and waits (see grid_dependency_wait).
// 32 sequences 250.5 -> 248.3 us per step, pruned 214.0 -> 210.5.  The same in the mask and verification kernels gains nothing.
__global__ void init_build_kernel(Workspace w, Params p, const int32_t* __restrict__ root_token) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    grid_dependency_wait();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < p.grid * p.mcap) {
        const int c = i / p.mcap, j = i - c * p.mcap;
        const long long b = (long long)c + (long long)j * p.grid;         // the j-th root sent to CTA c
        unsigned long long item = 0ull, ph = 0ull;
        if (b < p.B) {
            int token = root_token[b];
            if (token < 0 || token >= p.V) { set_status(w.status, kErrInternal); token = 0; }
            item = item_encode((int)b, 1, 0, row_of(token, 0, p.H));
            ph = phat_word(1.0);                                          // the root counts as factor 1
        }
        w.mb_items[i] = item;
        w.mb_phat[i] = ph;
    }
    for (long long j = i; j < 2ll * p.B * p.cstride; j += (long long)gridDim.x * blockDim.x) {
        reinterpret_cast<unsigned long long*>(w.cand_phat)[j] = 0ull;
        w.cand_tok[j] = 0;
    }
    // frontier row f stands for layer slot f unless a pruned layer says otherwise
    for (long long j = i; j < (long long)p.B * p.n; j += (long long)gridDim.x * blockDim.x) w.fmap[j] = (int32_t)(j % p.n);
    if (i < p.B) {
        int32_t* st = w.st + (size_t)i * 8;
        st[kStDone] = 0; st[kStNR] = 0; st[kStL1] = 0;
        w.E_prev[i] = 0.0;
    }
    if (i == 0) { w.q_ctl[kQFinished] = 0; w.q_ctl[kQDone] = 0; w.q_ctl[kQCursor] = p.B; }   // the roots are rows 0 .. B-1
}

// Source of the tree build: the rows other CTAs' layer warps have put into this CTA's mailbox.
template <bool kPrune>
struct BuildSource {
    static constexpr bool kHasEmpty = kPrune;              // only the pruned draft voids entries
    Workspace w; Params p;
    const uint16_t* draft;
    __device__ long long claim(int i) { return i < p.mcap ? (long long)blockIdx.x * p.mcap + i : -1; }
    // Both words of an entry validate themselves; the "all done" flag is looked at only when
    // check_done is set.
    __device__ int poll(long long idx, RowDesc& d, bool check_done) {
        const unsigned long long item = ld_relaxed_u64(&w.mb_items[idx]), ph = ld_relaxed_u64(&w.mb_phat[idx]);
        if (!((item & ph) >> 63)) return check_done && ld_acquire_s32(&w.q_ctl[kQDone]) ? -1 : 0;
        if (kPrune && (item & kItemVoid)) return 2;
        d.b = (int)((item >> 48) & 0x7FFFu); d.d = (int)((item >> 39) & 0x1FFu);
        d.slot = (int)((item >> 22) & 0x3FFu); d.fsize = 0;
        d.pphat = __longlong_as_double((long long)(ph & 0x7FFFFFFFFFFFFFFFull));
        int row = (int)(item & 0x3FFFFFu);
        if (row >= p.H) { set_status(w.status, kErrInternal); row = 0; }
        d.row = draft + (size_t)row * p.V;
        return 1;
    }
};

// Sink of the tree build.  Finisher warps: candidates' path values (Eq. 2) and the layer's row
// counter.  Layer warp: the layer warp of CTA c owns sequences c, c + gridDim.x, ...; it watches
// their row counters, and when a layer is complete does the layer selection, publishes the next
// layer's rows, brings the running top-n up to date and applies the loop test of Algorithm 1.
// kPrune: the pruned draft (opt_tree_build_pruned); a compile-time choice so that the ordinary build
// carries none of its code.
template <bool kPrune>
struct BuildSink {
    Workspace w; Params p; opt_tree_out out;
    int32_t* rows_read;                                    // pruned draft: rows of each sequence sent out so far (may be null)
    // Layer 1 by the finisher of the root's row.  The root's children are the only candidates of layer 1; when
    // they all fit the node budget nothing has to be selected: the finisher stores them as layer 1, as the
    // running top-n with its E_sub, applies the loop test and, if the tree grows on, sends out the rows of
    // layer 2 itself, which takes the layer team's round trip out of the first layer.  Returns false (nothing
    // done) when layer 1 needs a selection or the tree ends with it; the layer team then does it the ordinary way.
    __device__ bool first_layer_direct(const RowDesc& d, const RowOut& r, const SeqWork& sw) {
        const int lane = threadIdx.x & 31;
        const double ph = lane < r.kk ? d.pphat * r.p : 0.0;              // Eq. 2
        const double esub = warp_sum(ph);                                  // (the order update_running_team sums in)
        const bool more = 1 < p.Dcap && (esub > (double)p.delta);          // loop test of Algorithm 1 with E = 0
        if (r.kk > p.n || !more) return false;
        const TreeOut to = tree_out(out, p, d.b);
        unsigned g0 = 0;
        if (lane == 0) g0 = atomicAdd(reinterpret_cast<unsigned int*>(&w.q_ctl[kQCursor]), (unsigned)r.kk);
        g0 = __shfl_sync(0xFFFFFFFFu, g0, 0);
        if (lane < r.kk) {
            int token = r.tok;
            publish_node(row_queue(w, p), d.b, 1, g0, lane, token, phat_key(ph), w.status);
            if (token < 0 || token >= p.V) token = 0;
            sw.T_tok[lane] = token; sw.T_par[lane] = 0; sw.T_phat[lane] = ph;
            sw.R[p.n + lane] = lane;                                       // the running top-n after layer 1 (buffer of odd layers)
            if (kPrune) sw.fmap[lane] = lane;
        }
        if (lane == 0) {
            if (to.esub_trace) to.esub_trace[0] = esub;
            sw.st[kStNR] = r.kk;
            *sw.E_prev = esub;
        }
        return true;
    }
    __device__ void row_done(const RowDesc& d, const RowOut& r, FinScratch&) {
        const int lane = threadIdx.x & 31;
        const SeqWork sw = seq_work(w, p, d.b, d.d);
        if (d.d == 1) {                                                    // the root's row
            const bool direct = first_layer_direct(d, r, sw);
            __syncwarp();
            // Layer 1, the running top-n and E do not validate themselves: this word says, with release, that they are there.
            // (Layer 2's rows are on their way already, so this is off the chain.)
            if (lane == 0) {
                if (direct) {
                    st_release_s32(&sw.st[kStL1], (int)(0x80000000u | (unsigned)r.kk));
                    atom_add_relaxed_s32(&sw.st[kStDone], 1);
                } else {
                    *reinterpret_cast<volatile unsigned int*>(&sw.st[kStL1]) = 0x80000000u;
                }
            }
            if (direct) return;
        }
        // Candidate words validate themselves (top bit; an absent child is all ones), so neither they nor
        // the row count need a fence: the layer warp re-reads whatever it finds not yet written.  Except where layers can be
        // large: their selection looks only at the tokens of the nodes it takes, so the count is what says that a row's words
        // are all there and can be cleared (await_rows).
        if (lane < p.k) {
            unsigned long long* ph = reinterpret_cast<unsigned long long*>(sw.cand_phat) + d.slot * p.k + lane;
            unsigned int* tk = reinterpret_cast<unsigned int*>(sw.cand_tok) + d.slot * p.k + lane;
            *ph = lane < r.kk ? phat_word(d.pphat * r.p) : ~0ull;
            *tk = lane < r.kk ? (0x80000000u | (unsigned int)r.tok) : ~0u;
        }
        __syncwarp();
        if (lane == 0) {                                             // the count runs on over the layers of a build
            if (p.n * p.k > kStageCap) atom_add_release_s32(&sw.st[kStDone], 1);
            else atom_add_relaxed_s32(&sw.st[kStDone], 1);
        }
    }
    // The rows of a new layer take the next numbers of the build's running row count and with them
    // their CTAs (row g: CTA g % grid, mailbox entry g / grid).  Whatever the order in which the
    // sequences publish, every CTA is sent the same number of rows to within one, and a layer spreads
    // over as many SMs as it has rows.  reserve_layer only starts the atomic: lane 0 keeps the result
    // in a register, and nothing waits for it until the team has its candidates (threshold off: it goes to the job) or publish_layer
    // writes the entries.
    __device__ unsigned reserve_layer(int nl) {
        unsigned g0 = 0;
        if ((threadIdx.x & 31) == 0) g0 = atomicAdd(reinterpret_cast<unsigned int*>(&w.q_ctl[kQCursor]), (unsigned)nl);
        return g0;
    }
    // pick != null (pruned draft): only the layer slots pick[0..nl) are sent out, as frontier rows 0..nl;
    // the map from frontier row to layer slot is left in fmap for the next selection.
    template <class LS>
    __device__ void publish_layer(LS& ls, int nl, unsigned g0, int32_t* fmap = nullptr, const int* pick = nullptr) {
        g0 = __shfl_sync(0xFFFFFFFFu, g0, 0);
        for (int i = threadIdx.x & 31; i < nl; i += 32) {
            const int slot = pick ? pick[i] : i;
            if (fmap) fmap[i] = slot;
            publish_node(ls.job.queue, ls.job.b, ls.job.d, g0, i, ls.ltok[slot], ls.lkeys[slot], w.status);
        }
        __syncwarp();
    }
    // Entries g0+from .. g0+to of a reservation are not needed.
    template <class LS>
    __device__ void void_entries(LS& ls, unsigned g0, int from, int to) {
        g0 = __shfl_sync(0xFFFFFFFFu, g0, 0);
        for (int i = from + (int)(threadIdx.x & 31); i < to; i += 32) void_entry(ls.job.queue, g0 + (unsigned)i, w.status);
        __syncwarp();
    }
    // What every selection job has in common (lane 0).
    __device__ void set_job(LayerJob& j, int kind, const SeqWork& sw, int b, int d, int fsize) {
        j.kind = kind; j.b = b; j.d = d; j.fsize = fsize;
        j.cand_phat = sw.cand_phat; j.cand_tok = sw.cand_tok;
        j.T_tok = sw.T_tok; j.T_par = sw.T_par; j.T_phat = sw.T_phat;
        j.Rold = sw.R + ((d - 1) & 1) * p.n; j.Rnew = sw.R + (d & 1) * p.n;
    }
    // Pruned draft, a whole layer job with one selection (see select_running_team).  Returns the number
    // of rows of the next layer, or -1 if the sequence is finished.
    template <class LS>
    __device__ int merged_layer_job(LS& ls, const SeqWork& sw, int b, int d, int fsize, int nR_old, int off) {
        const int lane = threadIdx.x & 31;
        const int nvalid = fsize * p.kk, reserve = nvalid < p.n ? nvalid : p.n;
        const unsigned g0 = d < p.Dcap ? reserve_layer(reserve) : 0u;      // entries for the next layer, before its size is known
        const bool early = d < p.Dcap && p.delta == -INFINITY;             // (the loop test only looks at the depth)
        if (lane == 0) {
            LayerJob& j = ls.job;
            set_job(j, 2, sw, b, d, fsize);
            j.fmap = sw.fmap; j.nR_old = nR_old; j.off = off;
            j.cached = ls.cache_b == b && ls.cache_d == d - 1;             // this warp's last job was this sequence's previous layer
            j.publish = early;
        }
        __syncwarp();
        team_sync();
        const int nR = running_job<LS>(smem_offset(&ls), lane, g0, w.status);
        const int cnt = nR - ls.kept_old;                   // new members = the rows of the next layer
        const double esub = running_esub(ls, nR);
        const double eprev = d == 1 ? 0.0 : __ldcg(sw.E_prev);
        bool more = d < p.Dcap && (esub - eprev > (double)p.delta);
        const TreeOut to = tree_out(out, p, b);
        if (lane == 0) {
            if (to.esub_trace) to.esub_trace[d - 1] = esub;
            sw.st[kStNR] = nR;
            *sw.E_prev = esub;
            ls.cache_b = b; ls.cache_d = d;
        }
        __syncwarp();
        if (more && cnt > 0) {
            if (!early) {
                publish_layer(ls, cnt, g0, sw.fmap);        // members are sent out in slot order
                void_entries(ls, g0, cnt, reserve);
            }
            fence_gpu();                                    // the cleared candidate words before the rows of layer d + 2
            return cnt;
        }
        if (d < p.Dcap && !early) void_entries(ls, g0, 0, reserve);
        int d_end = d;
        if (more) {                                         // nothing left to draft from: the loop would go on testing a gain of zero
            d_end = p.delta < 0.0f ? p.Dcap : d + 1;
            if (to.esub_trace) for (int i = d + lane; i < d_end; i += 32) to.esub_trace[i] = esub;
            __syncwarp();
        }
        pack(ls, sw, to, b, d_end, nR, esub);
        return -1;
    }
    // The tree of sequence b from the running top-n in the scratch.  A tree of up to two nodes per lane of the layer warp is
    // packed by that warp: with the team's barriers one sequence of n = 10 takes 83.2 us a step, without 81.9; at n = 512 the
    // team's four warps save about 10 us.
    static constexpr int kPackAlone = 64;
    template <class LS>
    __device__ void pack(LS& ls, const SeqWork& sw, const TreeOut& to, int b, int d, int nR, double esub) {
        if ((threadIdx.x & 31) == 0) {
            LayerJob& j = ls.job;
            j.kind = 4; j.d = d; j.nR_old = nR; j.b = b;
            j.T_tok = sw.T_tok; j.T_par = sw.T_par;
            ls.last_esub = esub;
        }
        __syncwarp();
        const bool alone = p.n <= kPackAlone;
        if (!alone) team_sync();
        pack_tree<LS>(smem_offset(&ls), to, (int)(threadIdx.x & 31), alone ? 32 : kTeam, w.status);
        if (!alone) team_sync();                            // the scratch may be written again
        __syncwarp();
    }
    // A large layer's words may be cleared once all its rows have been counted: a token that came in later would pass for one of a
    // later layer.  (Bounded.)  The path values have all been seen by then, so this hardly ever waits, and the next
    // layer is on its way: two sequences of n = 512 431.8 us before, 432.0 with it.  (Waiting for the 8192 tokens: 443.)
    __device__ void await_rows(const int32_t* done, int rows) {
        if ((threadIdx.x & 31) == 0) {
            int t = 0;
            while (ld_acquire_s32(done) < rows && t < kWaitPolls) ++t;
            if (t == kWaitPolls) set_status(w.status, kErrTimeout);
        }
        __syncwarp();
    }
    // The layer warp follows its sequences (layer_follow); whenever a layer is complete it hands the
    // selection to the whole team: the job goes into shared memory, the team barrier starts it.  The
    // assistants wait at that barrier in between and leave when they find a job of kind 0.
    template <class LS>
    __device__ void layer_loop(LS& ls) {
        if ((threadIdx.x & 31) == 0) set_job_constants(ls.job, w, p);
        __syncwarp();
        layer_follow(ls);
        if ((threadIdx.x & 31) == 0) ls.job.kind = 0;
        __syncwarp();
        team_sync();
    }
    template <class LS>
    __device__ void layer_assist(LS& ls, int tw) {
        const int tt = tw * 32 + (int)(threadIdx.x & 31);
        for (;;) {
            team_sync();
            const int kind = ls.job.kind, at = smem_offset(&ls);
            if (kind == 0) return;
            // (kinds 2 and 3 clear candidate words; the fence puts the clears before what this thread sends out in later jobs)
            if (kind == 2) { running_job<LS>(at, tt, 0u, w.status); fence_gpu(); }
            else if (kind == 3) { update_running_team<LS>(at, tt, w.status); fence_gpu(); }
            else if (kind == 4) { pack_tree<LS>(at, tree_out(out, p, ls.job.b), tt, kTeam, w.status); team_sync(); }
            else select_job<LS>(at, tt, 0u, w.status);
        }
    }
    // Rows of a layer of f rows that may still be missing when the team starts on it.  Candidate words validate themselves, so the
    // team can start at once and wait for the words.  It does as long as a layer's rows of all sequences take the SMs at most four
    // times round; beyond that the polling would slow the rows down (a team reads every missing word again and again), and it
    // starts when at most sixteen rows or a quarter of a large layer are missing.  Steps (B200, us) with none ahead / always sixteen or a
    // quarter / always all / this rule: one sequence, n = 50 123.1 / 120.5 / 115.4 / 115.5; 2 of n = 512 399 / 385 / 373 / 380; 32 of n = 64
    // 250.3 / 246.6 / 261.2 / 245.1; 64 of n = 256, V = 152064 16190 / 16190 / 16830 / 16230; 32 pruned 200.6 / 190.1 / 192.9 / 188.6.
    // A warp that follows several sequences must not wait for one of them.
    __device__ int rows_ahead(int f) const {
        if (p.B > (int)gridDim.x) return 0;
        return p.B * f <= 4 * (int)gridDim.x ? f : min(max(16, f >> 2), f - 1);
    }
    template <class LS>
    __device__ void layer_follow(LS& ls) {
        const int lane = threadIdx.x & 31;
        constexpr int kOwn = 4;                            // sequences one layer warp follows at a time
        for (int b0 = blockIdx.x; b0 < p.B; b0 += kOwn * gridDim.x) {
            // layer in flight (0 = finished / none), its row count, rows expected in all layers so far
            int cur_d[kOwn], cur_f[kOwn], cur_tot[kOwn];
            int live = 0;
#pragma unroll
            for (int q = 0; q < kOwn; ++q) {
                const bool has = b0 + q * (int)gridDim.x < p.B;
                cur_d[q] = has ? 1 : 0; cur_f[q] = 1; cur_tot[q] = 1; live += has ? 1 : 0;
            }
            long long t0 = clock64();
            while (live > 0) {
                bool progressed = false;
#pragma unroll 1                                          // one copy of the body: it is long, and instruction fetch is what the helper warps wait for
                for (int q = 0; q < kOwn; ++q) {
                    if (cur_d[q] == 0) continue;
                    const int b = b0 + q * (int)gridDim.x;
                    const SeqWork sw = seq_work(w, p, b, cur_d[q]);
                    const int ahead = cur_d[q] > 1 ? rows_ahead(cur_f[q]) : 0;
                    if (ahead < cur_f[q]) {
                        int done = 0;
                        if (lane == 0) done = ld_acquire_s32(&sw.st[kStDone]);
                        done = __shfl_sync(0xFFFFFFFFu, done, 0);
                        if (done < cur_tot[q] - ahead) continue;
                    }
                    progressed = true;
                    if (cur_d[q] == 1) {
                        // the finisher of the root's row says whether it grew layer 1 itself (then layer 2 is on its way)
                        unsigned int how = 0;
                        if (lane == 0) {
                            how = poll_tok_word(reinterpret_cast<const unsigned int*>(&sw.st[kStL1]), w.status);
                            fence_gpu();                      // what the finisher wrote before that word
                        }
                        __syncwarp();
                        how = __shfl_sync(0xFFFFFFFFu, how, 0) & 0x7FFFFFFFu;
                        if (how != 0x7FFFFFFFu && how > 0) {
                            cur_d[q] = 2; cur_f[q] = (int)how; cur_tot[q] += (int)how;
                            if (kPrune && lane == 0 && rows_read) rows_read[b] = cur_tot[q];
                            continue;
                        }
                    }
                    const int d = cur_d[q], fsize = cur_f[q];
                    const int nvalid = fsize * p.kk, nl = nvalid < p.n ? nvalid : p.n;
                    // Without a threshold the loop test only looks at the depth: the next layer's rows
                    // can go out before the running top-n is brought up to date.
                    // The pruned draft always takes the one-selection layer job; the ordinary build takes it for
                    // the layer at the depth limit, after which nothing is drafted: the nodes of that layer that
                    // do not reach the running top-n need not be stored, and one selection does instead of two.
                    if (kPrune || d == p.Dcap) {
                        const int nR_old = d == 1 ? 0 : __ldcg(&sw.st[kStNR]);
                        const int off = (nR_old + 31) & ~31;
                        if (off + fsize * p.k <= kStageCap) {
                            const int sent = merged_layer_job(ls, sw, b, d, fsize, nR_old, off);
                            if (sent > 0) { cur_d[q] = d + 1; cur_f[q] = sent; cur_tot[q] += sent; }
                            if (kPrune && lane == 0 && rows_read) rows_read[b] = cur_tot[q];
                            if (sent <= 0) {
                                cur_d[q] = 0; --live;
                                __threadfence();
                                if (lane == 0 && atomicAdd(&w.q_ctl[kQFinished], 1) == p.B - 1) st_release_s32(&w.q_ctl[kQDone], 1);
                            }
                            __syncwarp();
                            continue;
                        }
                    }
                    const bool early = !kPrune && d < p.Dcap && p.delta == -INFINITY;
                    unsigned g0 = 0;
                    if (early) g0 = reserve_layer(nl);        // the rows' numbers, while the candidates load
                    if (lane == 0) {
                        LayerJob& j = ls.job;
                        set_job(j, 1, sw, b, d, fsize);
                        j.fmap = kPrune ? sw.fmap : nullptr;
                        j.publish = early;
                    }
                    __syncwarp();
                    team_sync();
                    select_job<LS>(smem_offset(&ls), lane, g0, w.status);
                    double esub;
                    int nR;
                    {
                        const bool cached = ls.cache_b == b && ls.cache_d == d - 1;   // rsel / vals hold the top-n before this layer
                        if (fsize * p.k > kStageCap) await_rows(&sw.st[kStDone], cur_tot[q]);
                        const int nR_old = d == 1 ? 0 : __ldcg(&sw.st[kStNR]);
                        __syncwarp();
                        if (lane == 0) {
                            LayerJob& j = ls.job;
                            j.kind = 3; j.ncand = fsize * p.k; j.fsize = nl; j.nR_old = nR_old; j.cached = cached;
                            ls.cache_b = b; ls.cache_d = d;
                        }
                        __syncwarp();
                        team_sync();
                        nR = update_running_team<LS>(smem_offset(&ls), lane, w.status);
                        esub = running_esub(ls, nR);
                    }
                    const double eprev = d == 1 ? 0.0 : __ldcg(sw.E_prev);
                    bool more = d < p.Dcap && (esub - eprev > (double)p.delta);       // loop test of Algorithm 1
                    const TreeOut to = tree_out(out, p, b);
                    if (lane == 0) {
                        if (to.esub_trace) to.esub_trace[d - 1] = esub;
                        sw.st[kStNR] = nR;
                        *sw.E_prev = esub;
                    }
                    __syncwarp();
                    if (!more) pack(ls, sw, to, b, d, nR, esub);
                    int sent = nl;                             // rows of the next layer
                    if (kPrune && more) {
                        // The new layer's nodes among the n largest are the tail of the ascending list rsel
                        // (their gids are the largest); only they are drafted from.
                        const int gid0 = (d - 1) * p.n;
                        int mine = 0;
                        for (int i = lane; i < nR; i += 32) mine += ls.rsel[i] >= gid0 ? 1 : 0;
                        sent = __reduce_add_sync(0xFFFFFFFFu, mine);
                        for (int i = lane; i < sent; i += 32) ls.gids[i] = ls.rsel[nR - sent + i] - gid0;
                        __syncwarp();
                        if (sent > 0) {
                            publish_layer(ls, sent, reserve_layer(sent), sw.fmap, ls.gids);
                        } else {
                            // Nothing left to draft from: further layers change neither T_opt nor E_sub.  The loop
                            // of Algorithm 1 would go on testing a gain of zero: to the depth limit if the
                            // threshold is negative, else for one more layer.
                            const int d_end = p.delta < 0.0f ? p.Dcap : d + 1;
                            if (to.esub_trace) for (int i = d + lane; i < d_end; i += 32) to.esub_trace[i] = esub;
                            __syncwarp();
                            pack(ls, sw, to, b, d_end, nR, esub);
                            more = false;
                        }
                    } else if (more && !early) {
                        publish_layer(ls, nl, reserve_layer(nl));
                    }
                    if (more) {
                        cur_d[q] = d + 1; cur_f[q] = sent; cur_tot[q] += sent;
                        fence_gpu();                          // the cleared candidate words before the rows of layer d + 2
                    }
                    if (kPrune && lane == 0 && rows_read) rows_read[b] = cur_tot[q];
                    if (!more) {
                        cur_d[q] = 0; --live;
                        __threadfence();
                        if (lane == 0 && atomicAdd(&w.q_ctl[kQFinished], 1) == p.B - 1) st_release_s32(&w.q_ctl[kQDone], 1);
                    }
                    __syncwarp();
                }
                if (progressed) t0 = clock64();
                else {
                    if (clock64() - t0 > kWaitCycles) { set_status(w.status, kErrTimeout); return; }
                    __nanosleep(kPollPauseNs);
                }
            }
        }
    }
};

// Algorithm 1 for a whole batch in one launch: persistent CTAs take rows from their mailboxes; layers
// of different sequences overlap freely because sequences never exchange data.
template <bool kPrune, int NCAP, int kForm>
__global__ void __launch_bounds__(kThreads)
build_kernel(Workspace w, Params p, const uint16_t* __restrict__ draft, opt_tree_out out, int32_t* rows_read) {
    CtaSmemT<NCAP>& s = *reinterpret_cast<CtaSmemT<NCAP>*>(ot_smem);
    BuildSource<kPrune> src{w, p, draft};
    BuildSink<kPrune> sink{w, p, out, rows_read};
    run_pipeline<kForm>(s, src, sink, p.V, p.k, draft, draft + (size_t)p.H * p.V, w.status);
}

// The row step alone over a list of rows (static round-robin over the CTAs).
struct ListSource {
    static constexpr bool kHasEmpty = false;
    const uint16_t* logits; const int32_t* rows; int nrows, V, H, first, stride; int* status;
    __device__ long long claim(int r) {
        const long long idx = (long long)first + (long long)r * stride;
        return idx < nrows ? idx : -1;
    }
    __device__ int poll(long long idx, RowDesc& d, bool) {
        int row = rows ? rows[idx] : (int)idx;             // no list: row idx of a dense buffer
        if (row < 0 || row >= H) { set_status(status, kErrInternal); row = 0; }
        d.row = logits + (size_t)row * V; d.slot = (int)idx; d.b = d.d = 0; d.fsize = 1;
        return 1;
    }
};
struct ListSink {
    int32_t* tok_out; double* prob_out; int k;
    template <class LS> __device__ void layer_loop(LS&) {}
    template <class LS> __device__ void layer_assist(LS&, int) {}
    __device__ void row_done(const RowDesc& d, const RowOut& r, FinScratch&) {
        const int lane = threadIdx.x & 31;
        if (lane < k) {
            tok_out[(size_t)d.slot * k + lane] = r.tok;
            prob_out[(size_t)d.slot * k + lane] = r.p;
        }
    }
};
template <int kForm>
__global__ void __launch_bounds__(kThreads)
row_topk_kernel(Params p, const uint16_t* __restrict__ logits, const int32_t* __restrict__ rows, int nrows,
                int32_t* tok_out, double* prob_out, int* status) {
    CtaSmem& s = *reinterpret_cast<CtaSmem*>(ot_smem);
    ListSource src{logits, rows, nrows, p.V, p.H, (int)blockIdx.x, (int)gridDim.x, status};
    ListSink sink{tok_out, prob_out, p.k};
    run_pipeline<kForm>(s, src, sink, p.V, p.k, logits, logits + (size_t)p.H * p.V, status);
}

// ------------------------------------------------------------------------------------------------
// Layer-by-layer build: the caller (a real draft model) hands in the logits of one layer's nodes at a time.  One launch
// per layer: the row pipeline over the dense buffer, its finishers leave the candidates (Eq. 2) as they do in the
// persistent build, and the CTA whose finisher completes a sequence's last row has its layer team select the layer, update
// the running top-n / E_sub, apply the loop test and hand back the next layer's tokens; a sequence that stops is packed on
// the spot.  A CTA whose team is at work finishes its rows later than others and so tends to complete the next sequences too:
// what it completes meanwhile goes to a queue that every idle team looks at, and that a CTA leaves only empty.  No CTA waits
// for another one's rows, so nothing is assumed about which of them run together.
// Ten layers, V = 32000 (us): two launches per layer (rows, then a CTA per sequence that formed the candidates) / the CTA that
// completes a sequence takes it / with the queue: 8 sequences of n = 50 354 / 268 / 237; 32 of n = 64 519 / 739 / 375; 64 of n = 24
// 436 / 672 / 347; 8 of n = 256, k = 16 969 / 622 / 463.
// ------------------------------------------------------------------------------------------------
// Where a sequence's tree stands: `rows` nodes of layer `layer` are to be expanded next (0: the tree is finished); `before`: how many
// were to get that layer.  A step may
// be asked of fewer sequences than the one before, so every sequence counts its own layers.  While a step runs, its CTAs
// must all see the state from before it: a sequence's even and odd layers have a word each, with the number of the
// step from which on it holds, and the newest that holds already counts.
struct Front { int layer, rows, before; };
static_assert(kMaxLayers < 512 && kMaxN < 2048, "fields of the word below");
constexpr int kNever = 0x7FFFFFFF;
__device__ __forceinline__ unsigned long long front_word(int call, int layer, int rows, int before) {
    return ((unsigned long long)(unsigned)call << 32) | ((unsigned)layer << 22) | ((unsigned)before << 11) | (unsigned)rows;
}
__device__ __forceinline__ unsigned long long* front_words(const Workspace& w, int b) {
    return reinterpret_cast<unsigned long long*>(w.st + (size_t)b * 8 + kStFront);
}
__device__ __forceinline__ Front front_at(const Workspace& w, int b, int call) {
    unsigned long long e, o;
    ld_relaxed_2u64(front_words(w, b), e, o);
    if ((int)(e >> 32) > call) e = 0ull;
    if ((int)(o >> 32) > call) o = 0ull;
    const unsigned long long v = (e >> 32) >= (o >> 32) ? e : o;
    return Front{(int)((v >> 22) & 511u), (int)(v & 2047u), (int)((v >> 11) & 2047u)};
}

__global__ void layers_begin_kernel(Workspace w, Params p) {
    grid_dependency_wait();
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    for (long long j = i; j < 2ll * p.B * p.cstride; j += (long long)gridDim.x * blockDim.x) {
        reinterpret_cast<unsigned long long*>(w.cand_phat)[j] = 0ull;
        w.cand_tok[j] = 0;
    }
    if (i == 0) { w.q_ctl[kQCall] = 0; w.q_ctl[kQLeft] = 0; w.q_ctl[kQTail] = 0; w.q_ctl[kQHead] = 0; }
    if (i >= p.B) return;
    int32_t* st = w.st + (size_t)i * 8;
    st[kStQueue] = 0;
    st[kStDone] = 0; st[kStNR] = 0;
    front_words(w, (int)i)[0] = front_word(0, 0, 1, 0);            // the root
    front_words(w, (int)i)[1] = front_word(kNever, 0, 0, 0);
    w.E_prev[i] = 0.0;
    w.front_phat[(size_t)i * 2 * p.n] = 1.0;                       // the root counts as factor 1
}

// Rows of the dense buffer [B][fstride][V]; rows at or beyond a sequence's count are not read.
struct LayersSource {
    static constexpr bool kHasEmpty = true;
    Workspace w; Params p;
    const uint16_t* logits;
    int fstride, call;                                     // steps before this one
    __device__ long long claim(int i) {
        const long long idx = (long long)blockIdx.x + (long long)i * gridDim.x;
        return idx < (long long)p.B * fstride ? idx : -1;
    }
    __device__ int poll(long long idx, RowDesc& d, bool) {
        const int b = (int)(idx / fstride), f = (int)(idx - (long long)b * fstride);
        // (the path values of even and odd layers come with the word that says which counts: one round trip instead of two; with the
        // 16-byte load in front_at 32 sequences of n = 64 381.5 -> 378.2 us, 8 of n = 50 244.6 -> 242.1, 16 of n = 50 274.9 -> 270.7)
        const double* fp = &w.front_phat[(size_t)b * 2 * p.n + f];
        const double even = __ldcg(fp), odd = __ldcg(fp + p.n);
        const Front at = front_at(w, b, call);
        if (f >= at.rows || at.rows > fstride) return 2;
        d.row = logits + (size_t)idx * p.V;
        d.b = b; d.d = at.layer + 1; d.slot = f; d.fsize = at.rows;
        d.pphat = (at.layer & 1) ? odd : even;
        return 1;
    }
};
template <class LS>
struct LayersSink {
    Workspace w; Params p; opt_tree_out out;
    int fstride, call, at;                                 // at: offset of the layer scratch in shared memory
    int32_t *next_tokens, *next_parent, *next_count;
    __device__ void row_done(const RowDesc& d, const RowOut& r, FinScratch&) {
        const int lane = threadIdx.x & 31;
        const SeqWork sw = seq_work(w, p, d.b, d.d);
        if (lane < p.k) {
            unsigned long long* ph = reinterpret_cast<unsigned long long*>(sw.cand_phat) + d.slot * p.k + lane;
            unsigned int* tk = reinterpret_cast<unsigned int*>(sw.cand_tok) + d.slot * p.k + lane;
            *ph = lane < r.kk ? phat_word(d.pphat * r.p) : ~0ull;
            *tk = lane < r.kk ? (0x80000000u | (unsigned int)r.tok) : ~0u;
        }
        __syncwarp();
        if (lane == 0) {
            LS& ls = smem_at<LS>(at);
            if (atomicAdd(&sw.st[kStDone], 1) + 1 == d.fsize) {            // (the words validate themselves: no fence)
                // this CTA's team, or, if that has a sequence already, the team that comes first
                if (atomicCAS(const_cast<int*>(&ls.todo), 0, d.b + 1) != 0) {
                    const int pos = atomicAdd(&w.q_ctl[kQTail], 1);
                    st_release_s32(&w.st[(size_t)pos * 8 + kStQueue], d.b + 1);
                }
            }
            __threadfence_block();
            atomicAdd(&ls.rows_done, 1);
        }
        __syncwarp();
    }
    static constexpr int kClaimed = 0x7FFFFFFF;
    // 1 + the sequence in place h of the queue, whose number was given out before the entry was written; the place is free again.
    __device__ __noinline__ int take_queued(int h) {
        int32_t* e = &w.st[(size_t)h * 8 + kStQueue];
        int v = ld_acquire_s32(e);
        for (int t = 0; v == 0 && t < kWaitPolls; ++t) v = ld_acquire_s32(e);
        if (v == 0) set_status(w.status, kErrTimeout);
        *e = 0;
        return v;
    }
    __device__ void layer_loop(LS& ls) {
        const int lane = threadIdx.x & 31;
        // sequences that stopped at an earlier layer, or whose layer does not fit the buffer
        for (int b = (int)blockIdx.x + lane * (int)gridDim.x; b < p.B; b += 32 * (int)gridDim.x) {
            const int fs = front_at(w, b, call).rows;
            if (fs >= 1 && fs <= fstride) continue;
            if (fs > fstride) set_status(w.status, kErrInternal);           // (a step with a wider buffer may follow)
            next_count[b] = 0;
        }
        // The candidate words of the step before, in the array of the other layers' parity, are cleared for the next step while this
        // one's rows stream.  (All of them were stored by the time that step's kernel ended.)
        for (int b = (int)blockIdx.x; b < p.B; b += (int)gridDim.x) {
            const Front now = front_at(w, b, call);
            if (now.rows > 0) {
                const SeqWork sw = seq_work(w, p, b, now.layer);
                clear_candidates(sw.cand_phat, sw.cand_tok, now.before * p.k, lane, 32);
            }
        }
        __syncwarp();
        if (lane == 0) set_job_constants(ls.job, w, p);
        const CtaCore& core = smem_at<CtaCore>(0);
        int seen = 0;
        long long t0 = clock64();
        for (int turn = 0;; ++turn) {
            const int v = __shfl_sync(0xFFFFFFFFu, ls.todo, 0);
            if (v) {
                step(ls, v - 1);
                if (lane == 0) ls.todo = 0;
                __syncwarp();
                t0 = clock64();
                continue;
            }
            // Every row of this CTA finished: it leaves when it finds the queue empty (what its own finishers put there came before
            // they counted the row).
            const int done = __shfl_sync(0xFFFFFFFFu, *reinterpret_cast<volatile int*>(&ls.rows_done), 0);
            const bool last = __any_sync(0xFFFFFFFFu, lane == 0 && done >= core.stop_row);
            if (last || (turn & 7) == 7) {
                int got = 0;                               // lane 0: 1 + the sequence taken, -1: the queue is empty
                if (lane == 0) {
                    __threadfence_block();
                    // (the team is claimed first, so that the finishers send what they complete to the queue)
                    if (atomicCAS(const_cast<int*>(&ls.todo), 0, kClaimed) == 0) {
                        const unsigned int* q = reinterpret_cast<const unsigned int*>(w.q_ctl);
                        const int h = (int)ld_relaxed_u32(&q[kQHead]), t = (int)ld_relaxed_u32(&q[kQTail]);
                        if (h >= t) got = -1;
                        else if (atomicCAS(&w.q_ctl[kQHead], h, h + 1) == h) got = take_queued(h);
                        if (got <= 0) ls.todo = 0;
                    }
                }
                got = __shfl_sync(0xFFFFFFFFu, got, 0);
                if (got > 0) {
                    step(ls, got - 1);
                    if (lane == 0) ls.todo = 0;
                    __syncwarp();
                    t0 = clock64();
                    continue;
                }
                if (last && got < 0) break;
            }
            if (done != seen) { seen = done; t0 = clock64(); }
            else if (__any_sync(0xFFFFFFFFu, clock64() - t0 > kWaitCycles)) { set_status(w.status, kErrTimeout); break; }
            __nanosleep(kPollPauseNs);
            __syncwarp();
        }
        if (lane == 0) {
            ls.job.kind = 0;
            __threadfence();
            if (atomicAdd(&w.q_ctl[kQLeft], 1) == (int)gridDim.x - 1) {
                w.q_ctl[kQLeft] = 0; w.q_ctl[kQTail] = 0; w.q_ctl[kQHead] = 0; w.q_ctl[kQCall] = call + 1;
            }
        }
        __syncwarp();
        team_sync();
    }
    __device__ void layer_assist(LS& ls, int tw) {
        const int tt = tw * 32 + (int)(threadIdx.x & 31);
        for (;;) {
            team_sync();
            const int kind = ls.job.kind;
            if (kind == 0) return;
            work(ls, kind, tt);
        }
    }
    // The team's part of a job; ends with a barrier.
    __device__ void work(LS& ls, int kind, int tt) {
        if (kind == 3) update_running_team<LS>(at, tt, w.status);
        else if (kind == 4) { pack_tree<LS>(at, tree_out(out, p, ls.job.b), tt, kTeam, w.status); team_sync(); }
        else if (kind == 6) { hand_back(ls, tt); team_sync(); }
        else select_job<LS>(at, tt, 0u, w.status);
    }
    __device__ void hand_back(LS& ls, int tt) {
        const int b = ls.job.b, nl = ls.job.fsize, gid0 = (ls.job.d - 1) * p.n;
        const int32_t* T_par = ls.job.T_par;
        double* front = w.front_phat + ((size_t)b * 2 + (ls.job.d & 1)) * p.n;
        for (int i = tt; i < nl; i += kTeam) {
            next_tokens[(size_t)b * p.n + i] = ls.ltok[i];
            next_parent[(size_t)b * p.n + i] = __ldcg(&T_par[gid0 + i]);
            front[i] = __longlong_as_double((long long)(ls.lkeys[i] - 1ull));
        }
    }
    __device__ void do_job(LS& ls, int kind) {               // the job's fields are set by lane 0
        const int lane = threadIdx.x & 31;
        if (lane == 0) ls.job.kind = kind;
        __syncwarp();
        team_sync();
        work(ls, kind, lane);
    }
    // One layer of one sequence.
    __device__ void step(LS& ls, int b) {
        const int nR_old = __ldcg(&w.st[(size_t)b * 8 + kStNR]);       // (0 before the first layer, like E; one round trip for all three)
        const double eprev = __ldcg(&w.E_prev[b]);
        const Front now = front_at(w, b, call);
        const int lane = threadIdx.x & 31, d = now.layer + 1, fsize = now.rows;
        const SeqWork sw = seq_work(w, p, b, d);
        const int nvalid = fsize * p.kk, nl = nvalid < p.n ? nvalid : p.n;
        if (lane == 0) {
            LayerJob& j = ls.job;
            j.b = b; j.d = d; j.fsize = fsize;
            j.cand_phat = sw.cand_phat; j.cand_tok = sw.cand_tok;
            j.T_tok = sw.T_tok; j.T_par = sw.T_par; j.T_phat = sw.T_phat; j.fmap = nullptr;
            j.nR_old = nR_old; j.cached = 0; j.publish = 0;
            j.Rold = sw.R + ((d - 1) & 1) * p.n; j.Rnew = sw.R + (d & 1) * p.n;
        }
        do_job(ls, 1);
        if (lane == 0) { ls.job.ncand = 0; ls.job.fsize = nl; }         // (the next step clears the candidates)
        do_job(ls, 3);
        const int NR = nR_old + nl, nR = NR < p.n ? NR : p.n;
        const double esub = running_esub(ls, nR);
        const bool more = d < p.Dcap && (esub - eprev > (double)p.delta);     // loop test of Algorithm 1
        const TreeOut to = tree_out(out, p, b);
        __syncwarp();
        if (lane == 0) {
            if (to.esub_trace) to.esub_trace[d - 1] = esub;
            sw.st[kStNR] = nR; *sw.E_prev = esub;
            sw.st[kStDone] = 0;
            st_relaxed_u64(front_words(w, b) + (d & 1), front_word(call + 1, d, more ? nl : 0, fsize));
            next_count[b] = more ? nl : 0;
            ls.job.nR_old = nR; ls.last_esub = esub;
        }
        do_job(ls, more ? 6 : 4);
    }
};
template <int NCAP, int kForm>
__global__ void __launch_bounds__(kThreads)
layers_kernel(Workspace w, Params p, const uint16_t* __restrict__ logits, int fstride, opt_tree_out out, int32_t* next_tokens,
              int32_t* next_parent, int32_t* next_count) {
    CtaSmemT<NCAP>& s = *reinterpret_cast<CtaSmemT<NCAP>*>(ot_smem);
    grid_dependency_wait();
    const int call = __ldcg(&w.q_ctl[kQCall]);               // (every thread has it before any CTA can leave: see run_pipeline's barrier)
    LayersSource src{w, p, logits, fstride, call};
    LayersSink<LayerScratchT<NCAP>> sink{w, p, out, fstride, call, smem_offset(&s.layer), next_tokens, next_parent, next_count};
    run_pipeline<kForm>(s, src, sink, p.V, p.k, logits, logits + (size_t)p.B * fstride * p.V, w.status);
}

// Tree attention mask + position ids: one CTA per sequence, a thread per node (in rounds of the block
// size when n is larger): the node's ancestor chain is walked, in shared memory, and its bits gathered in registers.
__global__ void __launch_bounds__(kSmallThreads)
mask_kernel(const int32_t* __restrict__ parent, const int32_t* __restrict__ depth, const int32_t* __restrict__ n_sel,
            const int32_t* __restrict__ base_pos, int n, uint64_t* mask, int32_t* position_ids, int* status) {
    grid_dependency_wait();
    const int b = blockIdx.x;
    const int W = (n + 63) >> 6;
    const int ns = n_sel[b];
    int* par = reinterpret_cast<int*>(ot_smem);
    for (int i = threadIdx.x; i < n; i += kSmallThreads) par[i] = parent[(size_t)b * n + i];
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += kSmallThreads) {
        uint64_t bits[kMaxN / 64];
#pragma unroll
        for (int wd = 0; wd < kMaxN / 64; ++wd) bits[wd] = 0ull;
        int pos = 0;
        if (i < ns) {
            int a = i, steps = 0;
            while (a >= 0 && steps <= n) {                  // an ancestor chain is at most n long
                if (a >= n) { set_status(status, kErrInternal); break; }
#pragma unroll
                for (int wd = 0; wd < kMaxN / 64; ++wd)
                    if ((a >> 6) == wd) bits[wd] |= 1ull << (a & 63);
                a = par[a];
                ++steps;
            }
            pos = (base_pos ? base_pos[b] : 0) + depth[(size_t)b * n + i];
        }
#pragma unroll
        for (int wd = 0; wd < kMaxN / 64; ++wd)
            if (wd < W) mask[((size_t)b * n + i) * W + wd] = bits[wd];
        position_ids[(size_t)b * n + i] = pos;
    }
}

// After verification: the bitmask expanded to the dense (n+1) x (n+1) form, position 0 being the
// root, and the step positions whose keys and values stay in the caches (the root and the matched
// nodes, in path order).  One CTA per sequence.
__global__ void __launch_bounds__(kSmallThreads)
post_verify_kernel(const int32_t* __restrict__ n_sel, const uint64_t* __restrict__ mask, const int32_t* __restrict__ accept_len,
                   const int32_t* __restrict__ accept_nodes, int n, int max_depth, uint8_t* dense, int32_t* kv_gather,
                   int32_t* kv_keep, int* status) {
    grid_dependency_wait();
    const int b = blockIdx.x, tid = threadIdx.x;
    const int S = n + 1, W = (n + 63) >> 6;
    const int ns = n_sel[b];
    const uint64_t* mb = mask + (size_t)b * n * W;
    uint8_t* db = dense + (size_t)b * S * S;
    for (int idx = tid; idx < S * S; idx += kSmallThreads) {
        const int r = idx / S, c = idx - r * S;
        bool on = r == c;
        if (r >= 1 && r - 1 < ns) {
            if (c == 0) on = true;
            else on = (mb[(size_t)(r - 1) * W + ((c - 1) >> 6)] >> ((c - 1) & 63)) & 1ull;
        }
        db[idx] = on ? 1 : 0;
    }
    int A = accept_len[b];
    if (A < 1 || A > max_depth + 1) { set_status(status, kErrInternal); A = 1; }
    for (int j = tid; j <= max_depth; j += kSmallThreads) {
        int g = -1;
        if (j == 0) g = 0;
        else if (j < A) {
            const int node = accept_nodes[(size_t)b * max_depth + j - 1];
            if (node < 0 || node >= ns) set_status(status, kErrInternal);
            else g = 1 + node;
        }
        kv_gather[(size_t)b * (max_depth + 1) + j] = g;
    }
    if (tid == 0) kv_keep[b] = A;
}

__device__ __forceinline__ uint4 ld_nc_v4(const uint4* p) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}

template <int T>
struct VerifySmem {
    unsigned long long red_u64[T / 32];
    int flag;
};

// The end of a verification CTA: position j's token y (thread 0's) is recorded; the CTA that records a sequence's
// last token walks the tree: accept the child that carries the recorded token, until none does.  The tree and the
// tokens go to shared memory first and one warp walks (a step is a few shared loads and a ballot per 32 nodes; with
// the arrays read from L2 at every step by the whole block it took about a microsecond: 32 sequences, 2080 rows of 32000
// logits, 26.5 us then, 20.4 now, 6.5 TB/s).
// walk: 3 n + 1 ints of dynamic shared memory.
template <int T>
__device__ void verify_tail(VerifySmem<T>& s, int* walk, const Workspace& w, const Params& p, int b, int j, int ns, int y,
                            const int32_t* tok, const int32_t* par, int32_t* accept_len, int32_t* accept_tokens,
                            int32_t* accept_nodes, int32_t* next_root) {
    const int tid = threadIdx.x, lane = tid & 31;
    int32_t* g = w.g + (size_t)b * (p.n + 1);
    if (tid == 0) {
        g[j] = y;
        __threadfence();
        s.flag = (atomicAdd(&w.vdone[b], 1) == ns);
        __threadfence();
    }
    __syncthreads();
    if (!s.flag) return;

    int *wtok = walk, *wpar = walk + p.n, *wg = walk + 2 * p.n;
    for (int i = tid; i < ns; i += T) { wtok[i] = tok[i]; wpar[i] = par[i]; }
    for (int i = tid; i <= ns; i += T) wg[i] = __ldcg(&g[i]);
    __syncthreads();
    if (tid >= 32) return;
    int32_t* at = accept_tokens + (size_t)b * (p.max_depth + 1);
    int32_t* an = accept_nodes + (size_t)b * p.max_depth;
    int cur = -1, A = 0, yy;
    for (;;) {
        yy = wg[cur + 1];
        if (lane == 0) at[A] = yy;
        if (++A > p.max_depth) break;
        int hit = -1;                                        // (a child is packed behind its parent; siblings carry distinct tokens)
        for (int i0 = (cur + 1) & ~31; i0 < ns && hit < 0; i0 += 32) {
            const int i = i0 + lane;
            const unsigned m = __ballot_sync(0xFFFFFFFFu, i < ns && wpar[i] == cur && wtok[i] == yy);
            if (m) hit = i0 + __ffs(m) - 1;
        }
        if (hit < 0) break;
        if (lane == 0) an[A - 1] = hit;
        cur = hit;
    }
    for (int i = A + lane; i <= p.max_depth; i += 32) at[i] = -1;
    for (int i = A - 1 + lane; i < p.max_depth; i += 32) an[i] = -1;
    if (lane == 0) {
        accept_len[b] = A;
        next_root[b] = yy;
        w.vdone[b] = 0;
    }
}

// Keys of the halves [0, h0) and [h1, V) of a row, at most seven at either end, that lie outside its whole 16-byte
// granules: the best of those this thread takes.  (With the whole of an unaligned row read in single logits the
// verification of 784 rows of 32003 logits took 31 us; 13.8 now.)
__device__ __noinline__ unsigned long long best_of_ends(const uint16_t* row, int V, int h0, int h1) {
    const int tid = threadIdx.x;
    unsigned long long best = 0ull;
    if (tid < h0) best = cand_key(__ldg(row + tid), (uint32_t)tid);
    if (tid < V - h1) {
        const unsigned long long key = cand_key(__ldg(row + h1 + tid), (uint32_t)(h1 + tid));
        best = key > best ? key : best;
    }
    return best;
}

// Greedy verification.  CTA (j, b): j = 0 takes the target row after the root, j >= 1 the row after
// kept node j-1; each finds the row's argmax (lowest token on ties).  The last CTA of a sequence
// then walks the tree: accept the child that carries the target's token, until none does.
// (0: no minimum of resident CTAs is asked for.  The narrow forms then take 32 registers and read 6.5 TB/s; asked for 16 or 8
// CTAs they do so with worse scheduling, 22.1 us instead of 20.4 on 2080 rows, and asked for one they take 56 registers, 24.3 us.)
template <int T>
__global__ void __launch_bounds__(T, T == kVerifyFew ? 3 : 0)
verify_kernel(Workspace w, Params p, const uint16_t* __restrict__ target, const int32_t* __restrict__ root_token,
              opt_tree_out tree, int32_t* accept_len, int32_t* accept_tokens, int32_t* accept_nodes, int32_t* next_root) {
    int* verify_walk = reinterpret_cast<int*>(ot_smem);
    __shared__ VerifySmem<T> s;
    grid_dependency_wait();
    const int b = blockIdx.y, j = blockIdx.x, tid = threadIdx.x;
    const int32_t* tok = tree.token + (size_t)b * p.n;
    const int32_t* par = tree.parent + (size_t)b * p.n;
    int ns = tree.n_sel[b];                                  // (all three loads at once: an unused slot's token is never looked at)
    int token = j == 0 ? root_token[b] : tok[j - 1];
    const int depth = j == 0 ? 0 : tree.depth[(size_t)b * p.n + j - 1];
    if (ns > p.n) { set_status(w.status, kErrInternal); ns = p.n; }        // (the walk's shared memory is sized for n nodes)
    if (j > ns) return;
    if (token < 0 || token >= p.V) { set_status(w.status, kErrInternal); token = 0; }
    const uint16_t* row = target + (size_t)row_of(token, depth, p.H) * p.V;

    // the row's whole granules, from half h0 on (a row may start anywhere: unaligned rows only differ by their ends)
    const int h0 = min((8 - vec_offset(row)) & 7, p.V);
    const uint4* vec = reinterpret_cast<const uint4*>(row + h0);
    const int nv = (p.V - h0) >> 3;
    float best = -INFINITY;
    int best_v = -1;
#pragma unroll 1
    for (int v0 = tid; v0 < nv; v0 += 8 * T) {
        uint4 q[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
            q[u] = v0 + u * T < nv ? ld_nc_v4(vec + v0 + u * T) : make_uint4(0xFF80FF80u, 0xFF80FF80u, 0xFF80FF80u, 0xFF80FF80u);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const uint32_t m2 = max_bf16x2(max_bf16x2(q[u].x, q[u].y), max_bf16x2(q[u].z, q[u].w));
            const float f = fmaxf(__uint_as_float(m2 << 16), __uint_as_float(m2 & 0xFFFF0000u));
            if (v0 + u * T < nv && (f > best || best_v < 0)) { best = f; best_v = v0 + u * T; }
        }
    }
    unsigned long long best_key = 0ull;
    if (best_v >= 0) {
        const uint4 q = vec[best_v];
        const uint32_t ww[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int e = 7; e >= 0; --e) {
            const uint32_t bits = (e & 1) ? (ww[e >> 1] >> 16) : (ww[e >> 1] & 0xFFFFu);
            if (bf16_bits_to_float(bits) == best) best_key = cand_key(bits, (uint32_t)(h0 + best_v * 8 + e));
        }
    }
    if (h0 + nv * 8 < p.V || h0 > 0) {
        const unsigned long long key = best_of_ends(row, p.V, h0, h0 + nv * 8);
        best_key = key > best_key ? key : best_key;
    }
    best_key = warp_max_u64(best_key);
    if ((tid & 31) == 0) s.red_u64[tid >> 5] = best_key;
    __syncthreads();
    if (tid == 0)
        for (int q = 1; q < T / 32; ++q) best_key = s.red_u64[q] > best_key ? s.red_u64[q] : best_key;
    verify_tail<T>(s, verify_walk, w, p, b, j, ns, (int32_t)cand_token(best_key), tok, par, accept_len, accept_tokens, accept_nodes, next_root);
}

// ------------------------------------------------------------------------------------------------
// Verification with sampling (temperature tau > 0): at every position the next token is drawn from
// softmax(x / tau) of the target row by inverse CDF in token order, with one uniform per (sequence,
// position) from the counter-based generator Philox4x32-10 (Salmon et al. 2011; key = seed, counter =
// (position, sequence, step low, step high)); the walk is the greedy one on the drawn tokens.
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ void philox4x32_10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, uint32_t k0, uint32_t k1,
                                              uint32_t& o0, uint32_t& o1) {
#pragma unroll 1
    for (int round = 0; round < 10; ++round) {
        const uint32_t h0 = __umulhi(0xD2511F53u, c0), l0 = 0xD2511F53u * c0;
        const uint32_t h1 = __umulhi(0xCD9E8D57u, c2), l1 = 0xCD9E8D57u * c2;
        const uint32_t n0 = h1 ^ c1 ^ k0, n2 = h0 ^ c3 ^ k1;
        c0 = n0; c1 = l1; c2 = n2; c3 = l0;
        k0 += 0x9E3779B9u; k1 += 0xBB67AE85u;
    }
    o0 = c0; o1 = c1;
}
__device__ __forceinline__ double uniform53(unsigned long long seed, unsigned long long step, int sequence, int position) {
    uint32_t o0, o1;
    philox4x32_10((uint32_t)position, (uint32_t)sequence, (uint32_t)step, (uint32_t)(step >> 32), (uint32_t)seed,
                  (uint32_t)(seed >> 32), o0, o1);
    const unsigned long long bits = (((unsigned long long)o1 << 32) | o0) >> 11;
    return (double)bits * (1.0 / 9007199254740992.0);
}

// Sampling works on segments of 64 vectors (512 logits): one warp, two coalesced 16-byte loads per lane.
constexpr int kSegVecs = 64;
constexpr int kSegTokens = kSegVecs * 8;
constexpr int kMaxSeg = 640;                 // rows of up to 327 680 logits take the one-pass path
constexpr int kSampleExpLimit = 1 << 22;     // |exponent| beyond which the single-precision pass cannot scale
struct alignas(8) SegPart { float sum; int E; };       // a segment's sum of 2^(x*c - E), E an integer
template <int T, bool kAligned>
struct SampleSmem {
    union { SegPart part[kMaxSeg]; double cum[kMaxSeg]; };   // per segment: its partial sum, then the running sum up to and including it
    int top[kAligned ? 1 : kMaxSeg];                         // unaligned rows: key of each segment's largest logit
    double wsum[T / 32];
    double S;
    float wmax[T / 32];
    int wE[T / 32];
    int chosen, last_live, seg, live_seg;
};

// The plain way, for rows the one-pass path does not take (very long rows, extreme magnitudes): thread t owns the tokens
// [t*L, (t+1)*L); the row's maximum, then every thread's sum of double-precision exponentials in token order, a scan over
// the threads, and the thread in whose stretch u*S falls walks it once more.  Returns the drawn token to every thread.
template <int T, bool kAligned>
__device__ __noinline__ int sample_row_plain(SampleSmem<T, kAligned>& q, const uint16_t* row, int V, bool vec, double tau, double u) {
    const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
    const int L = (((V + T - 1) / T) + 7) & ~7;       // tokens per thread, a multiple of 8
    const int lo = min(tid * L, V), hi = min(lo + L, V);
    auto logit = [&](int v) -> float { return bf16_bits_to_float(__ldg(row + v)); };
    const uint4* rv = reinterpret_cast<const uint4*>(row);
    float mx = -INFINITY;
    if (vec) {
        for (int v8 = lo >> 3; v8 < hi >> 3; ++v8) {
            const uint4 x = ld_nc_v4(rv + v8);
            const uint32_t m2 = max_bf16x2(max_bf16x2(x.x, x.y), max_bf16x2(x.z, x.w));
            mx = fmaxf(mx, fmaxf(__uint_as_float(m2 << 16), __uint_as_float(m2 & 0xFFFF0000u)));
        }
    } else {
        for (int v = lo; v < hi; ++v) mx = fmaxf(mx, logit(v));
    }
    mx = warp_max_f32(mx);
    __syncthreads();                                         // (the scratch may still be in use by the one-pass path)
    if (lane == 0) q.wmax[wp] = mx;
    if (tid == 0) { q.chosen = -1; q.last_live = -1; }
    __syncthreads();
    mx = q.wmax[0];
#pragma unroll
    for (int i = 1; i < T / 32; ++i) mx = fmaxf(mx, q.wmax[i]);
    const double m = (double)mx;
    double mine = 0.0;
    int live = -1;                                           // last token of the stretch with a positive term
    for (int v = lo; v < hi; ++v) {
        const double e = exp(((double)logit(v) - m) / tau);
        mine += e;
        if (e > 0.0) live = v;
    }
    double incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double up = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += up;
    }
    if (lane == 31) q.wsum[wp] = incl;
    __syncthreads();
    double base = 0.0, S = 0.0;                              // running sums before this warp / of the row, added up in one fixed order
#pragma unroll
    for (int i = 0; i < T / 32; ++i) { if (i == wp) base = S; S += q.wsum[i]; }
    // a thread's stretch begins exactly where the previous thread's ends: the same expression on both sides
    double prev = __shfl_up_sync(0xFFFFFFFFu, incl, 1);
    if (lane == 0) prev = 0.0;
    const double excl_t = base + prev, incl_t = base + incl;
    const double t = u * S;
    atomicMax(&q.last_live, live);
    if (incl_t > t && !(excl_t > t) && hi > lo) {            // the stretch in which the running sum passes t: one thread
        double run = excl_t;
        int y = live;
        for (int v = lo; v < hi; ++v) {
            run += exp(((double)logit(v) - m) / tau);
            if (run > t) { y = v; break; }
        }
        atomicMax(&q.chosen, y);
    }
    __syncthreads();
    int y = q.chosen;
    if (y < 0) y = q.last_live < 0 ? 0 : q.last_live;        // rounding left no stretch: the last token with a positive term
    return y;
}

// A segment of a row that does not lie on 16-byte boundaries, by one warp: the sum of e^((x - M) / tau), M its largest logit
// (`key`: in ordered form), in double precision throughout.
__device__ __forceinline__ double segment_f64(const uint16_t* row, int sg, int nv, int V, double c64, uint32_t& key) {
    const int lane = threadIdx.x & 31, o = vec_offset(row);
    auto vec_at = [&](int vi) -> uint4 {
        if (vi >= 1 && vi * 8 + 16 <= V) {                   // the two granules that hold the vector lie within the row
            const uint4* g = reinterpret_cast<const uint4*>(row + (size_t)vi * 8 - o);
            return shift_halves(ld_nc_v4(g), ld_nc_v4(g + 1), o);
        }
        return vi < nv ? load_row_vec_unaligned(row, vi, V) : make_uint4(0xFF80FF80u, 0xFF80FF80u, 0xFF80FF80u, 0xFF80FF80u);
    };
    const uint4 a = vec_at(sg * kSegVecs + lane), b = vec_at(sg * kSegVecs + 32 + lane);
    const uint32_t ww[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    uint32_t m2 = ww[0];
#pragma unroll
    for (int i = 1; i < 8; ++i) m2 = max_bf16x2(m2, ww[i]);
    key = __reduce_max_sync(0xFFFFFFFFu, max(ord16(m2 & 0xFFFFu), ord16(m2 >> 16)));
    if (key <= kOrdNegInf) return 0.0;                       // (warp-uniform) no finite logit
    const double M = (double)bf16_bits_to_float(ord16_inv(key));
    double sum = 0.0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const float lo = __uint_as_float(ww[i] << 16), hi = __uint_as_float(ww[i] & 0xFFFF0000u);
        sum += lo == -INFINITY ? 0.0 : exp2(((double)lo - M) * c64);
        sum += hi == -INFINITY ? 0.0 : exp2(((double)hi - M) * c64);
    }
    return warp_sum(sum);
}

// CTA (j, b) as in verify_kernel.  One pass over the row: warp w takes the segments w, w + T/32, ...; a
// segment's terms 2^(x*c - E) (c = log2(e) / tau, E an integer just above the segment's largest exponent)
// are summed in single precision with ex2.approx and kept per segment, so the running sum is known in
// token order at segment granularity.  The exponent x*c is formed with c split into a 16-bit head and a
// tail: x is bf16, so x * head is exact, and the rounding of c does not grow with |x*c| (low temperatures).
// Then: a double-precision scan over the segments, the segment in which u*S falls, and inside that segment
// (512 logits, 512 / T per thread) double-precision exponentials and an exact scan.  What can differ from a
// double-precision inverse CDF over the whole row is the placement of u*S relative to a segment's start, by
// the rounding of the single-precision sums (a few 1e-7 of S).
// Unaligned rows (kAligned false) take the same pass with segments counted from the row's first logit, whatever its address,
// and double-precision terms and sums: their draws are those of a double-precision inverse CDF throughout.  The exponentials are
// what bounds them: 784 rows of 32003 logits 80 us (284 by the plain way, 27 with single-precision sums, which moved draws),
// 51 rows 27 us (129, 16), 130 rows of 128257 70 us (446, 27).  Eight, four and two CTAs per SM, for the registers these take.
template <int T, bool kAligned>
__global__ void __launch_bounds__(T, kAligned ? (T == kVerifyMany ? 16 : (T == kVerifySome ? 6 : 3)) : (T == kVerifyMany ? 8 : (T == kVerifySome ? 4 : 2)))
verify_sampled_kernel(Workspace w, Params p, const uint16_t* __restrict__ target, const int32_t* __restrict__ root_token,
                      opt_tree_out tree, double tau, unsigned long long seed, unsigned long long step, int32_t* accept_len,
                      int32_t* accept_tokens, int32_t* accept_nodes, int32_t* next_root) {
    int* verify_walk = reinterpret_cast<int*>(ot_smem);
    __shared__ VerifySmem<T> s;
    __shared__ SampleSmem<T, kAligned> q;
    grid_dependency_wait();
    const int b = blockIdx.y, j = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
    const int32_t* tok = tree.token + (size_t)b * p.n;
    const int32_t* par = tree.parent + (size_t)b * p.n;
    int ns = tree.n_sel[b];                                  // (all three loads at once: an unused slot's token is never looked at)
    int token = j == 0 ? root_token[b] : tok[j - 1];
    const int depth = j == 0 ? 0 : tree.depth[(size_t)b * p.n + j - 1];
    if (ns > p.n) { set_status(w.status, kErrInternal); ns = p.n; }        // (the walk's shared memory is sized for n nodes)
    if (j > ns) return;
    if (token < 0 || token >= p.V) { set_status(w.status, kErrInternal); token = 0; }
    const uint16_t* row = target + (size_t)row_of(token, depth, p.H) * p.V;
    const double u = uniform53(seed, step, b, j);
    const int nv = (p.V + 7) >> 3, nseg = (nv + kSegVecs - 1) / kSegVecs;
    const double c64 = kLog2eD / tau;
    bool fast = nseg <= kMaxSeg && c64 < 1e30;
    int y = 0;
    if (fast) {
        if (tid == 0) { q.chosen = -1; q.last_live = -1; q.seg = 0x7FFFFFFF; q.live_seg = -1; }
        constexpr int kStep = T / 32;
        if (!kAligned) {
#pragma unroll 1
            for (int sg = wp; sg < nseg; sg += kStep) {
                uint32_t key;
                const double sum = segment_f64(row, sg, nv, p.V, c64, key);
                if (lane == 0) { q.cum[sg] = sum; q.top[sg] = (int)key; }
            }
        }
        const float c32 = (float)c64;
        const float c_hi = __uint_as_float(__float_as_uint(c32) & 0xFFFFFF00u);      // 16 significant bits
        const float c_lo = (float)(c64 - (double)c_hi);
        const uint4* rv = reinterpret_cast<const uint4*>(row);
        // two segments per turn: four 16-byte loads in flight per lane
        const unsigned long long chi2 = pack2(c_hi, c_hi), clo2 = pack2(c_lo, c_lo);
#pragma unroll 1
        for (int sg0 = wp; kAligned && sg0 < nseg; sg0 += 2 * kStep) {
            const uint4 pad = make_uint4(0xFF80FF80u, 0xFF80FF80u, 0xFF80FF80u, 0xFF80FF80u);
            uint4 qq[2][2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int v0 = (sg0 + h * kStep) * kSegVecs + lane, v1 = v0 + 32;
                qq[h][0] = v0 < nv ? ld_nc_v4(rv + v0) : pad;
                qq[h][1] = v1 < nv ? ld_nc_v4(rv + v1) : pad;
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int sg = sg0 + h * kStep;
                if (sg >= nseg) break;                            // (warp-uniform)
                const uint32_t ww[8] = {qq[h][0].x, qq[h][0].y, qq[h][0].z, qq[h][0].w, qq[h][1].x, qq[h][1].y, qq[h][1].z, qq[h][1].w};
                uint32_t m2 = ww[0];
#pragma unroll
                for (int i = 1; i < 8; ++i) m2 = max_bf16x2(m2, ww[i]);
                const uint32_t wkey = __reduce_max_sync(0xFFFFFFFFu, max(ord16(m2 & 0xFFFFu), ord16(m2 >> 16)));
                float sum = 0.0f, Ef = 0.0f;
                if (wkey > kOrdNegInf) {                          // (warp-uniform) the segment holds a finite logit
                    const float fmx = bf16_bits_to_float(ord16_inv(wkey));
                    Ef = rintf(fminf(fmaxf(fmaf(fmx, c32, 1.0f), -1e9f), 1e9f));
                    const unsigned long long nE2 = pack2(-Ef, -Ef);
                    unsigned long long acc2 = 0ull;
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const uint32_t cw = max_bf16x2(ww[i], 0xF149F149u);       // -inf -> -1e30: keeps the two-step product finite
                        const unsigned long long x2 = pack2(__uint_as_float(cw << 16), __uint_as_float(cw & 0xFFFF0000u));
                        float a0, a1;
                        unpack2(fma2(x2, clo2, fma2(x2, chi2, nE2)), a0, a1);
                        acc2 = add2(acc2, pack2(ex2_approx(a0), ex2_approx(a1)));
                    }
                    float s0, s1;
                    unpack2(acc2, s0, s1);
                    sum = s0 + s1;
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
                }
                if (lane == 0) { q.part[sg].sum = sum; q.part[sg].E = (int)Ef; }
            }
        }
        __syncthreads();
        int e = -0x7FFFFFFF;
        for (int sg = tid; sg < nseg; sg += T) {
            if (kAligned) { if (q.part[sg].sum > 0.0f) e = max(e, q.part[sg].E); }
            else if (q.cum[sg] > 0.0) e = max(e, q.top[sg]);
        }
        e = __reduce_max_sync(0xFFFFFFFFu, e);
        if (lane == 0) q.wE[wp] = e;
        __syncthreads();
        int Eg = q.wE[0];
#pragma unroll
        for (int i = 1; i < T / 32; ++i) Eg = max(Eg, q.wE[i]);
        fast = kAligned ? Eg > -kSampleExpLimit && Eg < kSampleExpLimit : Eg > 0;        // the same for every thread
        const double Mg = kAligned ? 0.0 : (double)bf16_bits_to_float(ord16_inv((uint32_t)max(Eg, 0)));     // the row's largest logit
        // term of logit x on the scale of the running sums
        auto term = [&](float x) { return kAligned ? exp2((double)x * c64 - (double)Eg) : exp2(((double)x - Mg) * c64); };
        if (fast) {
            if (wp == 0) {                                    // running sums over the segments, in token order
                double carry = 0.0;
                for (int s0 = 0; s0 < nseg; s0 += 32) {
                    const int sg = s0 + lane;
                    double v = 0.0;
                    if (sg < nseg) {
                        if (kAligned) { const SegPart pt = q.part[sg]; v = pt.sum > 0.0f ? ldexp((double)pt.sum, pt.E - Eg) : 0.0; }
                        else { v = q.cum[sg]; if (v > 0.0) v *= term(bf16_bits_to_float(ord16_inv((uint32_t)q.top[sg]))); }
                    }
                    double incl = v;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const double up = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                        if (lane >= o) incl += up;
                    }
                    incl += carry;
                    __syncwarp();
                    if (sg < nseg) q.cum[sg] = incl;
                    carry = __shfl_sync(0xFFFFFFFFu, incl, 31);
                }
                if (lane == 0) q.S = carry;
            }
            __syncthreads();
            const double t = u * q.S;
            for (int sg = tid; sg < nseg; sg += T) {
                const double c = q.cum[sg];
                if (c > t) atomicMin(&q.seg, sg);
                if (c > (sg > 0 ? q.cum[sg - 1] : 0.0)) atomicMax(&q.live_seg, sg);
            }
            __syncthreads();
            int sg = q.seg;
            if (sg == 0x7FFFFFFF) sg = q.live_seg < 0 ? 0 : q.live_seg;          // u*S rounded up to S: the last segment with a positive sum
            const double before = sg > 0 ? q.cum[sg - 1] : 0.0;
            // inside the segment: kPer logits per thread, double precision
            constexpr int kPer = kSegTokens / T;
            const int t0 = sg * kSegTokens + kPer * tid;
            double ev[kPer];
            int live = -1;
#pragma unroll
            for (int i = 0; i < kPer; ++i) {
                const int tk = t0 + i;
                const float xf = tk < p.V ? bf16_bits_to_float(__ldg(row + tk)) : -INFINITY;
                ev[i] = xf == -INFINITY ? 0.0 : term(xf);
                if (ev[i] > 0.0) live = tk;
            }
            double mine = ev[0];
#pragma unroll
            for (int i = 1; i < kPer; ++i) mine += ev[i];
            double incl = mine;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const double up = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                if (lane >= o) incl += up;
            }
            if (lane == 31) q.wsum[wp] = incl;
            __syncthreads();
            double base = before;                             // running sum where this warp's stretch begins (one fixed order)
            for (int i = 0; i < wp; ++i) base += q.wsum[i];
            double prev = __shfl_up_sync(0xFFFFFFFFu, incl, 1);
            if (lane == 0) prev = 0.0;
            const double excl_t = base + prev, incl_t = base + incl;
            atomicMax(&q.last_live, live);
            if (incl_t > t && !(excl_t > t)) {                // this thread's logits: one thread
                double run = excl_t;
                int yy = live;
#pragma unroll
                for (int i = 0; i < kPer; ++i) {
                    run += ev[i];
                    if (run > t && ev[i] > 0.0) { yy = t0 + i; break; }
                }
                atomicMax(&q.chosen, yy);
            }
            __syncthreads();
            y = q.chosen;
            if (y < 0) y = q.last_live < 0 ? min(sg * kSegTokens, p.V - 1) : q.last_live;   // the exact sums end just below u*S: the segment's last live token
        }
    }
    if (!fast) y = sample_row_plain(q, row, p.V, kAligned, tau, u);
    verify_tail<T>(s, verify_walk, w, p, b, j, ns, y, tok, par, accept_len, accept_tokens, accept_nodes, next_root);
}

// ------------------------------------------------------------------------------------------------
// Self-test of the bounded waits: one CTA whose warps each enter one kind of wait on something that
// nobody will ever complete or write (a fresh mbarrier, words that stay zero, a source that never has
// a row), with a limit of microseconds.  Every wait must give up, record kErrTimeout in its own
// status word and let the kernel end.  No bulk copy is in flight and nothing else runs in the CTA.
// ------------------------------------------------------------------------------------------------
struct NeverSource {
    static constexpr bool kHasEmpty = false;
    __device__ long long claim(int i) { return i; }
    __device__ int poll(long long, RowDesc&, bool) { return 0; }
};
__global__ void __launch_bounds__(kThreads)
wait_probe_kernel(int* result, const unsigned long long* zero_words, long long limit, int polls) {
    CtaSmem& s = *reinterpret_cast<CtaSmem*>(ot_smem);
    pipeline_init(s.core, s.layer);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp == 0) {
        mbar_wait_warp(&s.core.full_bar[0], 0u, &result[0], limit);
    } else if (warp == 1) {
        if (lane == 0) mbar_wait_thread(&s.core.full_bar[1], 0u, &result[1], limit);
    } else if (warp == 2) {
        if (lane == 0) poll_phat_word(zero_words, &result[2], polls);
    } else if (warp == 3) {
        if (lane == 0) poll_tok_word(reinterpret_cast<const unsigned int*>(zero_words + 1), &result[3], polls);
    } else if (warp == 4) {
        NeverSource src;
        fetcher_role(s.core, src, &result[4], limit);
    }
}

// Self-test of a layer selection whose candidate words never come: one CTA, of which only the layer team works.  It selects layer 2 of
// sequence 0 from `rows` frontier rows, of which only the first `written` have their words, and leaves the selection's nodes in the caller's
// arrays.  joint: the selection over the running top-n (one node of layer 1) and the candidates together.
template <int NCAP>
__global__ void __launch_bounds__(kThreads)
selection_probe_kernel(Workspace w, Params p, int rows, int written, int joint, int polls, int* status, int32_t* tok, int32_t* par, double* phat) {
    using LS = LayerScratchT<NCAP>;
    CtaSmemT<NCAP>& s = *reinterpret_cast<CtaSmemT<NCAP>*>(ot_smem);
    LS& ls = s.layer;
    pipeline_init(s.core, ls);
    const int tt = (int)threadIdx.x - (kConsumerWarps + kHelperLayer) * 32;
    if (tt < 0 || tt >= kTeam) return;
    const SeqWork sw = seq_work(w, p, 0, 2);
    for (int i = tt; i < rows * p.k; i += kTeam) {         // path values 1/2, 1/4, 1/8, 1/2 ...: ties as well
        const bool there = i < written * p.k;
        sw.cand_phat[i] = there ? __longlong_as_double((long long)phat_word(1.0 / (2 << (i % 3)))) : 0.0;
        sw.cand_tok[i] = there ? (int)(0x80000000u | (unsigned)(i % p.V)) : 0;
    }
    for (int i = tt; i < p.n; i += kTeam) sw.fmap[i] = i;
    if (tt == 0) {
        LayerJob& j = ls.job;
        set_job_constants(j, w, p);
        j.polls = polls;
        j.kind = joint ? 2 : 1; j.b = 0; j.d = 2; j.fsize = rows; j.ncand = 0;
        j.cand_phat = sw.cand_phat; j.cand_tok = sw.cand_tok;
        j.T_tok = sw.T_tok; j.T_par = sw.T_par; j.T_phat = sw.T_phat;
        j.fmap = sw.fmap; j.nR_old = 1; j.off = 32; j.cached = 0; j.publish = 1;
        j.Rold = sw.R + p.n; j.Rnew = sw.R;
        sw.R[p.n] = 0; sw.T_tok[0] = 0; sw.T_par[0] = 0; sw.T_phat[0] = 1.0;
    }
    __threadfence();
    team_sync();
    const int at = smem_offset(&ls), nvalid = rows * p.kk;
    int nl = nvalid < p.n ? nvalid : p.n;
    if (joint) nl = running_job<LS>(at, tt, 0u, status) - ls.kept_old;
    else select_job<LS>(at, tt, 0u, status);
    for (int i = tt; i < p.n; i += kTeam) {
        tok[i] = i < nl ? __ldcg(&sw.T_tok[p.n + i]) : -1; par[i] = i < nl ? __ldcg(&sw.T_par[p.n + i]) : -1;
        phat[i] = i < nl ? __ldcg(&sw.T_phat[p.n + i]) : -1.0;
    }
}

}  // namespace ot

// ------------------------------------------------------------------------------------------------
// C ABI
// ------------------------------------------------------------------------------------------------
struct opt_tree_ctx {
    opt_tree_config cfg;
    ot::Workspace ws;
    void* base;
    size_t bytes;
    int device;
    int sms;
    int grid;              // resident CTAs of the persistent kernels (SMs x occupancy)
    size_t smem;           // dynamic shared memory of one such CTA (cta_smem_bytes(cfg.n))
    int mcap;
    int64_t launches;
    // pinned host staging of opt_tree_step_host: the step's inputs and outputs cross the bus in one
    // copy each and are spread to / gathered from the caller's arrays on the host
    char* hstage;
    size_t in_bytes, out_bytes;     // device ranges [h_root, end of h_base) and [o_token, end of o_next)
};

namespace {

bool valid_cfg(const opt_tree_config* c) {
    return c && c->V >= 1 && c->H >= 1 && c->n >= 1 && c->k >= 1 && c->max_depth >= 1 && c->max_batch >= 1;
}
int supported_cfg(const opt_tree_config* c) {
    if (c->n > OPT_TREE_MAX_N || c->k > OPT_TREE_MAX_K || c->k > c->V) return OPT_TREE_ERR_UNSUPPORTED;
    if ((long long)c->V * 31 + c->max_depth > 2147483647LL) return OPT_TREE_ERR_UNSUPPORTED;
    if (c->max_batch > 32767 || c->max_depth > 65535 || c->H > ot::kMaxTableRows) return OPT_TREE_ERR_UNSUPPORTED;
    if ((c->max_depth < c->n ? c->max_depth : c->n) > ot::kMaxLayers) return OPT_TREE_ERR_UNSUPPORTED;   // the mailbox item's layer field
    return OPT_TREE_OK;
}
ot::Params make_params(const opt_tree_ctx* ctx, const void* table, float delta) {
    const opt_tree_config& c = ctx->cfg;
    ot::Params p;
    p.V = c.V; p.H = c.H; p.n = c.n; p.k = c.k; p.kk = c.k < c.V ? c.k : c.V;
    p.Dcap = c.max_depth < c.n ? c.max_depth : c.n;
    p.max_depth = c.max_depth;
    p.B = 0;
    p.prune = 0;
    p.mcap = ctx->mcap;
    p.grid = ctx->grid;
    p.cstride = (int)ot::cand_stride(c.n, c.k);
    p.by_grid = ot::FixedDiv::by((unsigned)ctx->grid); p.by_H = ot::FixedDiv::by((unsigned)c.H); p.by_k = ot::FixedDiv::by((unsigned)c.k);
    p.delta = delta;
    p.aligned = ((reinterpret_cast<uintptr_t>(table) & 15u) == 0 && (c.V % 8) == 0) ? 1 : 0;
    return p;
}
// Launches a kernel that may be set up while the kernel before it in the stream drains (every kernel of
// this library waits for its predecessor before it touches global memory, see grid_dependency_wait).
template <class... KArgs, class... Args>
void launch_after(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}
// Threads of a verification CTA for (n + 1) * B rows (see kVerifyMany); `some`: rows per SM up to which CTAs of 256 are taken.
int verify_threads(int n, int B, int sms, int some) {
    const long long rows = (long long)(n + 1) * B;
    return rows <= 3ll * sms ? ot::kVerifyFew : (rows <= (long long)some * sms ? ot::kVerifySome : ot::kVerifyMany);
}
template <bool kAligned> auto sampled_variant(int threads) {
    return threads == ot::kVerifyFew ? ot::verify_sampled_kernel<ot::kVerifyFew, kAligned>
                                     : (threads == ot::kVerifySome ? ot::verify_sampled_kernel<ot::kVerifySome, kAligned> : ot::verify_sampled_kernel<ot::kVerifyMany, kAligned>);
}
size_t walk_smem(int n) { return (size_t)(3 * n + 1) * sizeof(int); }
bool bad_tree(const opt_tree_out* t) {
    return !t || !t->token || !t->parent || !t->depth || !t->phat || !t->n_sel || !t->depth_reached || !t->expected_len;
}
int check_launch() { return cudaGetLastError() == cudaSuccess ? OPT_TREE_OK : OPT_TREE_ERR_CUDA; }

// Shared memory of a CTA of the persistent kernels for node budget n (one of two layouts).
bool small_n(int n) { return n <= ot::kSmallN; }
size_t cta_smem_bytes(int n) { return small_n(n) ? sizeof(ot::CtaSmemT<ot::kSmallN>) : sizeof(ot::CtaSmemT<ot::kMaxN>); }

using BuildKernel = void (*)(ot::Workspace, ot::Params, const uint16_t*, opt_tree_out, int32_t*);
using RowKernel = void (*)(ot::Params, const uint16_t*, const int32_t*, int, int32_t*, double*, int*);
// Variants: a form of row each (RowForm), the build's also pruned or not.
constexpr int kForms = ot::kRowForms;
template <int NCAP> BuildKernel build_variant(int form, bool prune) {
    static const BuildKernel kernels[kForms][2] = {
        {ot::build_kernel<false, NCAP, 0>, ot::build_kernel<true, NCAP, 0>}, {ot::build_kernel<false, NCAP, 1>, ot::build_kernel<true, NCAP, 1>},
        {ot::build_kernel<false, NCAP, 2>, ot::build_kernel<true, NCAP, 2>}, {ot::build_kernel<false, NCAP, 3>, ot::build_kernel<true, NCAP, 3>},
        {ot::build_kernel<false, NCAP, 4>, ot::build_kernel<true, NCAP, 4>}};
    return kernels[form][prune ? 1 : 0];
}
BuildKernel build_kernel_for(int n, int form, bool prune) { return small_n(n) ? build_variant<ot::kSmallN>(form, prune) : build_variant<ot::kMaxN>(form, prune); }
RowKernel row_variant(int form) {
    static const RowKernel kernels[kForms] = {ot::row_topk_kernel<0>, ot::row_topk_kernel<1>, ot::row_topk_kernel<2>, ot::row_topk_kernel<3>, ot::row_topk_kernel<4>};
    return kernels[form];
}
using LayersKernel = void (*)(ot::Workspace, ot::Params, const uint16_t*, int, opt_tree_out, int32_t*, int32_t*, int32_t*);
template <int NCAP> LayersKernel layers_variant(int form) {
    static const LayersKernel kernels[kForms] = {ot::layers_kernel<NCAP, 0>, ot::layers_kernel<NCAP, 1>, ot::layers_kernel<NCAP, 2>,
                                                 ot::layers_kernel<NCAP, 3>, ot::layers_kernel<NCAP, 4>};
    return kernels[form];
}
int form_of(const ot::Params& p, bool build) { return ot::row_form(p.aligned != 0, p.V, p.kk, build); }
template <class F> bool allow_smem(F* kernel, size_t bytes) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) == cudaSuccess;
}

// CTAs of the persistent kernels on the current device (one CTA of kThreads per SM as long as its
// shared memory fits); 0 if there is no usable device.
int persistent_grid(int n) {
    int dev = 0, per_sm = 0, sms = 0;
    constexpr int S = ot::kSmallN, L = ot::kMaxN;
    if (cudaGetDevice(&dev) != cudaSuccess) { cudaGetLastError(); return 0; }
    bool ok = true;
    for (int f = 0; f < kForms; ++f) {
        for (int prune = 0; prune < 2; ++prune)
            ok = ok && allow_smem(build_variant<S>(f, prune), sizeof(ot::CtaSmemT<S>)) && allow_smem(build_variant<L>(f, prune), sizeof(ot::CtaSmemT<L>));
        ok = ok && allow_smem(row_variant(f), sizeof(ot::CtaSmem)) && allow_smem(layers_variant<S>(f), sizeof(ot::CtaSmemT<S>)) &&
             allow_smem(layers_variant<L>(f), sizeof(ot::CtaSmemT<L>));
    }
    int least = 1 << 30;                             // the variants share one grid: the smallest occupancy counts
    for (int f = 0; f < kForms && ok; ++f)
        for (int prune = 0; prune < 2 && ok; ++prune) {
            ok = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, build_kernel_for(n, f, prune), ot::kThreads, cta_smem_bytes(n)) == cudaSuccess;
            least = per_sm < least ? per_sm : least;
        }
    if (!ok || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    const int grid = least * sms;
    return grid >= 1 && grid <= ot::kMaxGrid ? grid : 0;
}

}  // namespace

extern "C" {

size_t opt_tree_workspace_bytes(const opt_tree_config* cfg) {
    if (!valid_cfg(cfg) || supported_cfg(cfg) != OPT_TREE_OK) return 0;
    int grid = persistent_grid(cfg->n);
    if (grid == 0) grid = 148;                       // no device here: the size on a B200
    return ot::carve(*cfg, grid, nullptr, nullptr);
}

int opt_tree_create(opt_tree_ctx** out, const opt_tree_config* cfg) {
    if (!out) return OPT_TREE_ERR_INVALID_ARG;
    *out = nullptr;
    if (!valid_cfg(cfg)) return OPT_TREE_ERR_INVALID_ARG;
    int rc = supported_cfg(cfg);
    if (rc != OPT_TREE_OK) return rc;
    opt_tree_ctx* ctx = new (std::nothrow) opt_tree_ctx();
    if (!ctx) return OPT_TREE_ERR_CUDA;
    ctx->cfg = *cfg;
    ctx->launches = 0;
    ctx->grid = persistent_grid(cfg->n);
    ctx->smem = cta_smem_bytes(cfg->n);
    if (ctx->grid == 0) { delete ctx; return OPT_TREE_ERR_CUDA; }
    ctx->mcap = (int)ot::mailbox_capacity(*cfg, ctx->grid);
    ctx->bytes = ot::carve(*cfg, ctx->grid, nullptr, nullptr);
    if ((long long)ctx->mcap * ctx->grid > 0x7FFFFFFFLL) { delete ctx; return OPT_TREE_ERR_UNSUPPORTED; }
    if (cudaGetDevice(&ctx->device) != cudaSuccess ||
        cudaDeviceGetAttribute(&ctx->sms, cudaDevAttrMultiProcessorCount, ctx->device) != cudaSuccess || cudaMalloc(&ctx->base, ctx->bytes) != cudaSuccess) {
        cudaGetLastError();
        delete ctx;
        return OPT_TREE_ERR_CUDA;
    }
    ot::carve(*cfg, ctx->grid, static_cast<char*>(ctx->base), &ctx->ws);
    // (carve lays h_root, h_base out next to each other, and likewise o_token ... o_next)
    ctx->in_bytes = (size_t)(reinterpret_cast<char*>(ctx->ws.h_base + cfg->max_batch) - reinterpret_cast<char*>(ctx->ws.h_root));
    ctx->out_bytes = (size_t)(reinterpret_cast<char*>(ctx->ws.o_next + cfg->max_batch) - reinterpret_cast<char*>(ctx->ws.o_token));
    ctx->hstage = nullptr;
    if (cudaMemset(ctx->base, 0, ctx->bytes) != cudaSuccess ||
        cudaHostAlloc(reinterpret_cast<void**>(&ctx->hstage), ctx->in_bytes + ctx->out_bytes, cudaHostAllocDefault) != cudaSuccess) {
        cudaGetLastError();
        cudaFree(ctx->base);
        delete ctx;
        return OPT_TREE_ERR_CUDA;
    }
    *out = ctx;
    return OPT_TREE_OK;
}

int opt_tree_destroy(opt_tree_ctx* ctx) {
    if (!ctx) return OPT_TREE_ERR_INVALID_ARG;
    if (ctx->hstage) cudaFreeHost(ctx->hstage);
    cudaError_t e = cudaFree(ctx->base);
    delete ctx;
    return e == cudaSuccess ? OPT_TREE_OK : OPT_TREE_ERR_CUDA;
}

static int build_common(opt_tree_ctx* ctx, const void* draft, const int32_t* root_token, int32_t B, float delta,
                        const opt_tree_out* out, int prune, int32_t* rows_read, void* stream) {
    if (!ctx || !draft || !root_token || bad_tree(out) || B < 1 || delta != delta) return OPT_TREE_ERR_INVALID_ARG;
    if (B > ctx->cfg.max_batch) return OPT_TREE_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    ot::Params p = make_params(ctx, draft, delta);
    p.B = B;
    p.prune = prune;
    const long long init_threads = (long long)ctx->grid * ctx->mcap > B ? (long long)ctx->grid * ctx->mcap : B;
    launch_after(ot::init_build_kernel, dim3((unsigned)((init_threads + 255) / 256)), dim3(256), 0, st, ctx->ws, p, root_token);
    launch_after(build_kernel_for(ctx->cfg.n, form_of(p, true), prune != 0), dim3(ctx->grid), dim3(ot::kThreads), ctx->smem, st, ctx->ws, p, static_cast<const uint16_t*>(draft), *out, rows_read);
    ctx->launches += 2;
    return check_launch();
}

int opt_tree_build(opt_tree_ctx* ctx, const void* draft, const int32_t* root_token, int32_t B, float delta,
                   const opt_tree_out* out, void* stream) {
    return build_common(ctx, draft, root_token, B, delta, out, 0, nullptr, stream);
}

int opt_tree_build_pruned(opt_tree_ctx* ctx, const void* draft, const int32_t* root_token, int32_t B, float delta,
                          const opt_tree_out* out, int32_t* rows_read, void* stream) {
    return build_common(ctx, draft, root_token, B, delta, out, 1, rows_read, stream);
}

int opt_tree_mask(opt_tree_ctx* ctx, const opt_tree_out* tree, int32_t B, const int32_t* base_pos, uint64_t* mask,
                  int32_t* position_ids, void* stream) {
    if (!ctx || bad_tree(tree) || !mask || !position_ids || B < 1 || B > ctx->cfg.max_batch) return OPT_TREE_ERR_INVALID_ARG;
    launch_after(ot::mask_kernel, dim3(B), dim3(ot::kSmallThreads), ctx->cfg.n * sizeof(int), static_cast<cudaStream_t>(stream),
                 tree->parent, tree->depth, tree->n_sel, base_pos, ctx->cfg.n, mask, position_ids, ctx->ws.status);
    ctx->launches++;
    return check_launch();
}

int opt_tree_verify(opt_tree_ctx* ctx, const opt_tree_out* tree, const void* target, const int32_t* root_token, int32_t B,
                    int32_t* accept_len, int32_t* accept_tokens, int32_t* accept_nodes, int32_t* next_root, void* stream) {
    if (!ctx || bad_tree(tree) || !target || !root_token || !accept_len || !accept_tokens || !accept_nodes || !next_root ||
        B < 1 || B > ctx->cfg.max_batch)
        return OPT_TREE_ERR_INVALID_ARG;
    const ot::Params p = make_params(ctx, target, 0.0f);
    const int threads = verify_threads(ctx->cfg.n, B, ctx->sms, 8);
    launch_after(threads == ot::kVerifyFew ? ot::verify_kernel<ot::kVerifyFew>
                                           : (threads == ot::kVerifySome ? ot::verify_kernel<ot::kVerifySome> : ot::verify_kernel<ot::kVerifyMany>),
                 dim3(ctx->cfg.n + 1, B), dim3(threads), walk_smem(ctx->cfg.n), static_cast<cudaStream_t>(stream),
                 ctx->ws, p, static_cast<const uint16_t*>(target), root_token, *tree, accept_len, accept_tokens, accept_nodes, next_root);
    ctx->launches++;
    return check_launch();
}

int opt_tree_verify_sampled(opt_tree_ctx* ctx, const opt_tree_out* tree, const void* target, const int32_t* root_token, int32_t B,
                            double tau, uint64_t seed, uint64_t step, int32_t* accept_len, int32_t* accept_tokens,
                            int32_t* accept_nodes, int32_t* next_root, void* stream) {
    if (!ctx || bad_tree(tree) || !target || !root_token || !accept_len || !accept_tokens || !accept_nodes || !next_root ||
        B < 1 || B > ctx->cfg.max_batch || !(tau > 0.0))
        return OPT_TREE_ERR_INVALID_ARG;
    const ot::Params p = make_params(ctx, target, 0.0f);
    const int threads = verify_threads(ctx->cfg.n, B, ctx->sms, 6);
    launch_after(p.aligned ? sampled_variant<true>(threads) : sampled_variant<false>(threads),
                 dim3(ctx->cfg.n + 1, B), dim3(threads), walk_smem(ctx->cfg.n), static_cast<cudaStream_t>(stream),
                 ctx->ws, p, static_cast<const uint16_t*>(target), root_token, *tree, tau, (unsigned long long)seed,
                 (unsigned long long)step, accept_len, accept_tokens, accept_nodes, next_root);
    ctx->launches++;
    return check_launch();
}

int opt_tree_post_verify(opt_tree_ctx* ctx, const opt_tree_out* tree, const uint64_t* mask, const int32_t* accept_len,
                         const int32_t* accept_nodes, int32_t B, uint8_t* dense_mask, int32_t* kv_gather, int32_t* kv_keep,
                         void* stream) {
    if (!ctx || bad_tree(tree) || !mask || !accept_len || !accept_nodes || !dense_mask || !kv_gather || !kv_keep || B < 1 ||
        B > ctx->cfg.max_batch)
        return OPT_TREE_ERR_INVALID_ARG;
    launch_after(ot::post_verify_kernel, dim3(B), dim3(ot::kSmallThreads), 0, static_cast<cudaStream_t>(stream),
                 tree->n_sel, mask, accept_len, accept_nodes, ctx->cfg.n, ctx->cfg.max_depth, dense_mask, kv_gather, kv_keep,
                 ctx->ws.status);
    ctx->launches++;
    return check_launch();
}

int opt_tree_layers_begin(opt_tree_ctx* ctx, int32_t B, void* stream) {
    if (!ctx || B < 1 || B > ctx->cfg.max_batch) return OPT_TREE_ERR_INVALID_ARG;
    ot::Params p = make_params(ctx, nullptr, 0.0f);
    p.B = B;
    const long long blocks = ((long long)B * p.cstride + 255) / 256;
    launch_after(ot::layers_begin_kernel, dim3((unsigned)(blocks < 1024 ? blocks : 1024)), dim3(256), 0, static_cast<cudaStream_t>(stream), ctx->ws, p);
    ctx->launches++;
    return check_launch();
}

int opt_tree_layers_step(opt_tree_ctx* ctx, const void* frontier_logits, int32_t frontier_stride, int32_t B, float delta,
                         const opt_tree_out* out, int32_t* next_tokens, int32_t* next_parent, int32_t* next_count, void* stream) {
    if (!ctx || !frontier_logits || bad_tree(out) || !next_tokens || !next_parent || !next_count || B < 1 ||
        B > ctx->cfg.max_batch || frontier_stride < 1 || frontier_stride > ctx->cfg.n || delta != delta)
        return OPT_TREE_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    ot::Params p = make_params(ctx, frontier_logits, delta);
    p.B = B;
    const int nrows = B * frontier_stride, form = form_of(p, true);
    launch_after(small_n(ctx->cfg.n) ? layers_variant<ot::kSmallN>(form) : layers_variant<ot::kMaxN>(form), dim3(nrows < ctx->grid ? nrows : ctx->grid),
                 dim3(ot::kThreads), ctx->smem, st, ctx->ws, p, static_cast<const uint16_t*>(frontier_logits), frontier_stride, *out,
                 next_tokens, next_parent, next_count);
    ctx->launches++;
    return check_launch();
}

int opt_tree_row_softmax_topk(opt_tree_ctx* ctx, const void* logits, const int32_t* rows, int32_t nrows, int32_t* tok_out,
                              double* prob_out, void* stream) {
    if (!ctx || !logits || !rows || !tok_out || !prob_out || nrows < 0) return OPT_TREE_ERR_INVALID_ARG;
    if (nrows == 0) return OPT_TREE_OK;
    const ot::Params p = make_params(ctx, logits, 0.0f);
    const int grid = nrows < ctx->grid ? nrows : ctx->grid;
    launch_after(row_variant(form_of(p, false)), dim3(grid), dim3(ot::kThreads), sizeof(ot::CtaSmem),
        static_cast<cudaStream_t>(stream), p, static_cast<const uint16_t*>(logits), rows, nrows, tok_out, prob_out, ctx->ws.status);
    ctx->launches++;
    return check_launch();
}

int opt_tree_step_host(opt_tree_ctx* ctx, const void* draft, const void* target, const int32_t* root_host,
                       const int32_t* base_host, int32_t B, float delta, const opt_tree_host_out* ho, void* stream) {
    if (!ctx || !draft || !target || !root_host || !ho || B < 1 || B > ctx->cfg.max_batch) return OPT_TREE_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const ot::Workspace& w = ctx->ws;
    const size_t n = ctx->cfg.n, D = ctx->cfg.max_depth, W = (ctx->cfg.n + 63) / 64, Bz = B;
    // inputs: one copy of the range that holds both device arrays
    char* hin = ctx->hstage;
    char* hout = ctx->hstage + ctx->in_bytes;
    const char* din = reinterpret_cast<const char*>(w.h_root);
    memcpy(hin, root_host, Bz * 4);
    if (base_host) memcpy(hin + (reinterpret_cast<const char*>(w.h_base) - din), base_host, Bz * 4);
    if (cudaMemcpyAsync(w.h_root, hin, ctx->in_bytes, cudaMemcpyHostToDevice, st) != cudaSuccess) return OPT_TREE_ERR_CUDA;
    opt_tree_out t = {w.o_token, w.o_parent, w.o_depth, w.o_phat, w.o_nsel, w.o_dreach, w.o_elen, nullptr};
    int rc = opt_tree_build(ctx, draft, w.h_root, B, delta, &t, stream);
    if (rc == OPT_TREE_OK) rc = opt_tree_mask(ctx, &t, B, base_host ? w.h_base : nullptr, w.o_mask, w.o_pos, stream);
    if (rc == OPT_TREE_OK) rc = opt_tree_verify(ctx, &t, target, w.h_root, B, w.o_alen, w.o_atok, w.o_anode, w.o_next, stream);
    if (rc != OPT_TREE_OK) return rc;
    // outputs: one copy of the range that holds all result arrays, then each to the caller's array
    const char* dout = reinterpret_cast<const char*>(w.o_token);
    if (cudaMemcpyAsync(hout, dout, ctx->out_bytes, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return OPT_TREE_ERR_CUDA;
#define OT_OUT(dst, src, bytes) if (dst) memcpy((dst), hout + (reinterpret_cast<const char*>(src) - dout), (bytes));
    OT_OUT(ho->token, w.o_token, Bz * n * 4) OT_OUT(ho->parent, w.o_parent, Bz * n * 4) OT_OUT(ho->depth, w.o_depth, Bz * n * 4)
    OT_OUT(ho->phat, w.o_phat, Bz * n * 8) OT_OUT(ho->n_sel, w.o_nsel, Bz * 4) OT_OUT(ho->depth_reached, w.o_dreach, Bz * 4)
    OT_OUT(ho->expected_len, w.o_elen, Bz * 8) OT_OUT(ho->mask, w.o_mask, Bz * n * W * 8) OT_OUT(ho->position_ids, w.o_pos, Bz * n * 4)
    OT_OUT(ho->accept_len, w.o_alen, Bz * 4) OT_OUT(ho->accept_tokens, w.o_atok, Bz * (D + 1) * 4)
    OT_OUT(ho->accept_nodes, w.o_anode, Bz * D * 4) OT_OUT(ho->next_root, w.o_next, Bz * 4)
#undef OT_OUT
    return OPT_TREE_OK;
}

int opt_tree_selftest_waits(opt_tree_ctx* ctx, int32_t* result, void* stream) {
    if (!ctx || !result) return OPT_TREE_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (cudaFuncSetAttribute(ot::wait_probe_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(ot::CtaSmem)) != cudaSuccess ||
        cudaMemsetAsync(result, 0, OPT_TREE_SELFTEST_WAITS * sizeof(int32_t), st) != cudaSuccess ||
        cudaMemsetAsync(ctx->ws.o_mask, 0, 2 * sizeof(unsigned long long), st) != cudaSuccess) {    // two words nobody writes meanwhile
        cudaGetLastError();
        return OPT_TREE_ERR_CUDA;
    }
    ot::wait_probe_kernel<<<1, ot::kThreads, sizeof(ot::CtaSmem), st>>>(
        result, reinterpret_cast<const unsigned long long*>(ctx->ws.o_mask), 1ll << 16, 1 << 10);
    ctx->launches++;
    return check_launch();
}

int opt_tree_selftest_selection(opt_tree_ctx* ctx, int32_t rows, int32_t written, int32_t joint, int32_t* result, int32_t* token,
                                int32_t* parent, double* phat, void* stream) {
    if (!ctx || !result || !token || !parent || !phat || rows < 1 || rows > ctx->cfg.n || written < 0 || written > rows || ctx->cfg.max_depth < 2)
        return OPT_TREE_ERR_INVALID_ARG;
    if (joint && 32 + rows * ctx->cfg.k > ot::kStageCap) return OPT_TREE_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    ot::Params p = make_params(ctx, nullptr, 0.0f);
    p.B = 1;
    const bool small = small_n(ctx->cfg.n);
    auto* kernel = small ? ot::selection_probe_kernel<ot::kSmallN> : ot::selection_probe_kernel<ot::kMaxN>;
    if (!allow_smem(kernel, ctx->smem) || cudaMemsetAsync(result, 0, sizeof(int32_t), st) != cudaSuccess) {
        cudaGetLastError();
        return OPT_TREE_ERR_CUDA;
    }
    kernel<<<1, ot::kThreads, ctx->smem, st>>>(ctx->ws, p, rows, written, joint, 1 << 10, result, token, parent, phat);
    ctx->launches++;
    return check_launch();
}

int opt_tree_last_device_status(opt_tree_ctx* ctx, int32_t* status_host) {
    if (!ctx || !status_host) return OPT_TREE_ERR_INVALID_ARG;
    if (cudaDeviceSynchronize() != cudaSuccess) return OPT_TREE_ERR_CUDA;
    if (cudaMemcpy(status_host, ctx->ws.status, 4, cudaMemcpyDeviceToHost) != cudaSuccess) return OPT_TREE_ERR_CUDA;
    if (cudaMemset(ctx->ws.status, 0, 4) != cudaSuccess) return OPT_TREE_ERR_CUDA;
    return OPT_TREE_OK;
}

int64_t opt_tree_launch_count(const opt_tree_ctx* ctx) { return ctx ? ctx->launches : 0; }

const char* opt_tree_strerror(int code) {
    switch (code) {
        case OPT_TREE_OK: return "ok";
        case OPT_TREE_ERR_INVALID_ARG: return "invalid argument";
        case OPT_TREE_ERR_UNSUPPORTED: return "unsupported configuration";
        case OPT_TREE_ERR_CUDA: return "CUDA runtime error";
        case OPT_TREE_ERR_TIMEOUT: return "device-side wait timed out";
        case OPT_TREE_ERR_INTERNAL: return "device-side bounds check failed";
        default: return "unknown error";
    }
}

}  // extern "C"

// ------------------------------------------------------------------------------------------------
// Verification without any allocation (opt_tree_verify_static).
// ------------------------------------------------------------------------------------------------
// The verify kernel needs three pieces of scratch: the target's best token per node, a per-sequence
// arrival counter and a status word.  A context keeps them in memory it got from cudaMalloc; this
// variant keeps them in the array below, which is part of the loaded library image on every GPU.
namespace {

constexpr size_t kStaticG = (size_t)OPT_TREE_STATIC_MAX_BATCH * (OPT_TREE_STATIC_MAX_N + 1);   // ints
constexpr size_t kStaticInts = kStaticG + OPT_TREE_STATIC_MAX_BATCH + 1;
constexpr size_t kStaticBytes = (kStaticInts * sizeof(int32_t) + 255) & ~(size_t)255;

static __device__ __align__(256) unsigned char g_verify_scratch[kStaticBytes];

constexpr int kMaxDevices = 64;
int32_t* g_scratch_addr[kMaxDevices];      // device address of g_verify_scratch on each device, once looked up

// The array's name means nothing to a kernel when used from host code; the device address comes from
// the runtime, once per device, with that device current.  No lock: two threads racing here both
// store the same value.
int static_scratch(int32_t** out) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return OPT_TREE_ERR_CUDA;
    if (!g_scratch_addr[dev]) {
        void* ptr = nullptr;
        if (cudaGetSymbolAddress(&ptr, g_verify_scratch) != cudaSuccess || !ptr) {
            cudaGetLastError();
            return OPT_TREE_ERR_CUDA;
        }
        g_scratch_addr[dev] = static_cast<int32_t*>(ptr);
    }
    *out = g_scratch_addr[dev];
    return OPT_TREE_OK;
}

}  // namespace

extern "C" int opt_tree_verify_static(const opt_tree_config* cfg, const opt_tree_out* tree, const void* target,
                                      const int32_t* root_token, int32_t B, int32_t* accept_len, int32_t* accept_tokens,
                                      int32_t* accept_nodes, int32_t* next_root, int32_t* device_status, void* stream) {
    if (!cfg) return OPT_TREE_ERR_INVALID_ARG;
    opt_tree_config sized = *cfg;
    sized.max_batch = 1;                                     // this entry point does not look at max_batch
    if (!valid_cfg(&sized) || bad_tree(tree) || !target || !root_token || !accept_len || !accept_tokens || !accept_nodes ||
        !next_root || B < 1)
        return OPT_TREE_ERR_INVALID_ARG;
    if (supported_cfg(&sized) != OPT_TREE_OK) return OPT_TREE_ERR_UNSUPPORTED;
    if (B > OPT_TREE_STATIC_MAX_BATCH || cfg->n > OPT_TREE_STATIC_MAX_N) return OPT_TREE_ERR_UNSUPPORTED;
    int32_t* base = nullptr;
    const int rc = static_scratch(&base);
    if (rc != OPT_TREE_OK) return rc;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    ot::Workspace ws;
    memset(&ws, 0, sizeof ws);
    ws.g = base;
    ws.vdone = base + kStaticG;
    ws.status = base + kStaticG + OPT_TREE_STATIC_MAX_BATCH;
    // counters and status start from zero whatever the previous call left behind
    if (cudaMemsetAsync(ws.vdone, 0, (OPT_TREE_STATIC_MAX_BATCH + 1) * sizeof(int32_t), st) != cudaSuccess) return OPT_TREE_ERR_CUDA;
    ot::Params p;
    memset(&p, 0, sizeof p);
    p.V = cfg->V; p.H = cfg->H; p.n = cfg->n; p.k = cfg->k; p.kk = cfg->k < cfg->V ? cfg->k : cfg->V;
    p.max_depth = cfg->max_depth; p.Dcap = cfg->max_depth < cfg->n ? cfg->max_depth : cfg->n;
    p.aligned = ((reinterpret_cast<uintptr_t>(target) & 15u) == 0 && (cfg->V % 8) == 0) ? 1 : 0;
    ot::verify_kernel<ot::kVerifyMany><<<dim3(cfg->n + 1, B), ot::kVerifyMany, walk_smem(cfg->n), st>>>(
        ws, p, static_cast<const uint16_t*>(target), root_token, *tree, accept_len, accept_tokens, accept_nodes, next_root);
    if (cudaGetLastError() != cudaSuccess) return OPT_TREE_ERR_CUDA;
    if (device_status && cudaMemcpyAsync(device_status, ws.status, sizeof(int32_t), cudaMemcpyDeviceToDevice, st) != cudaSuccess)
        return OPT_TREE_ERR_CUDA;
    return OPT_TREE_OK;
}
