// The hot kernel: one decoding step of SAM-Decoding's draft retrieval for a batch of sequences.
//
// One block per sequence slot, of two warps and, up to 1184 slots, a third that reads ahead of them.  Warp 0 advances the slot's match state through the
// STATIC automaton (Transfer, Algorithm 1) for each accepted token; warp 1 extends the slot's own
// DYNAMIC automaton (Expand, Algorithm 3) with the same tokens and keeps its match state, which
// after each Expand is link[last] with length len[link[last]] (the state Transfer would reach on
// the automaton as it was before the token, Section 3.3, made canonical).  Both warps then read
// the first end position of their state, fetch their candidate draft speculatively, and the
// source rule l1 > l2 + l_bias (Section 3.2) picks which one is written out.
//
// Each warp runs one dependent chain of memory reads, so the work is latency-bound, and the code
// is organised around the number of read round trips per step:
//   - everything a step needs to start (64 control words with copies of both match states'
//     records, the count, the first 32 tokens) is read in one round trip;
//   - values are warp-uniform (all lanes read the same 32-byte record: one request); lanes work
//     side by side only where a structure is wide (a 128-byte hash bucket, a window of 32 root-table
//     entries, an edge block, the draft read);
//   - independent reads go out together: a static state's record with its hash bucket, the root-row
//     entries of all tokens of the step, and the dynamic root-table lookups of all tokens of a chunk,
//     one lane per token;
//   - runs of tokens that are new to the sequence while nothing is matched are extended by the lanes
//     in parallel (each such Expand is three independent writes);
//   - runs of tokens that repeat a passage of the sequence and make every Expand clone are extended by
//     the lanes in parallel as well: the states the clones are made from are guessed (position -> state
//     map, or ids two apart), read in one round trip and checked (dyn_repeat_run);
//   - the static match is not advanced token by token: all suffixes of the row are walked side by side, and a
//     match that goes on as the corpus does is taken in one round (static_match.cuh);
//   - steps whose tokens are all at hand (sam_run_steps) run in one launch or two, no slot waiting for another;
//   - a prompt that fills an empty slot is not extended token by token either: its automaton is built at once by all
//     threads of a block (prefill_build.cuh, sam_prefill_kernel);
//   - when the batch is larger than the GPU holds at once, the slots with the most tokens are started
//     first (order_slots_kernel);
//   - from 8192 slots on the two sides of a slot run as separate one-warp blocks (the static side of a slot
//     with few tokens on a single lane), neither waiting for the other, and whichever finishes last writes
//     the slot's outputs (sam_step_split_kernel, further down).
#include "common.h"
#include "once.h"

#include <cstring>

// Operation counters (library built with -DSAM_COUNTERS only): per slot, what its two chains did — the
// moves and insertions Algorithms 1 and 3 count, and the rounds of dependent reads each chain waited for.
// They exist to be compared with the CPU oracle's counters and to put a number on the latency bound;
// the regular build carries none of this.
#ifdef SAM_COUNTERS
__device__ unsigned long long* g_sam_counters = nullptr;     // [slots][SAM_N_COUNTERS]
__device__ int g_sam_counter_slots = 0;
#define SAM_COUNT(x, n) ((x) += (n))
#else
#define SAM_COUNT(x, n) ((void)0)
#endif

namespace {

constexpr unsigned FULL = 0xFFFFFFFFu;

// The sum of v over a warp's lanes up to this one.
__device__ __forceinline__ int sum_upto(int v, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const int t = __shfl_up_sync(FULL, v, o); if (lane >= o) v += t; }
    return v;
}

// counts of one chain of one slot in one step, or in all of a replay (registers; dropped by the compiler in the regular build)
struct ChainCounts { uint32_t rounds, a, b, c, d; };

__device__ __forceinline__ void flush_counts(int slot, int lane, bool is_static, const ChainCounts& k, int m, int steps) {
#ifdef SAM_COUNTERS
    if (g_sam_counters && lane == 0 && slot < g_sam_counter_slots) {
        unsigned long long* o = g_sam_counters + (size_t)slot * SAM_N_COUNTERS;
        if (is_static) {
            o[SAM_CNT_STATIC_ROUNDS] += k.rounds; o[SAM_CNT_STATIC_LINK_MOVES] += k.a; o[SAM_CNT_STATIC_NEXT_MOVES] += k.b;
        } else {
            o[SAM_CNT_DYNAMIC_ROUNDS] += k.rounds; o[SAM_CNT_WALK_INSERTS] += k.a; o[SAM_CNT_CLONES] += k.b;
            o[SAM_CNT_COPIED_EDGES] += k.c; o[SAM_CNT_REDIRECTS] += k.d;
            o[SAM_CNT_TOKENS] += (unsigned)m; o[SAM_CNT_SEQ_STEPS] += (unsigned)steps;
        }
    }
#endif
}
constexpr int MAX_DRAFT_REGS = 4;     // 4 x 32 lanes = 128 draft tokens

}  // namespace

#include "static_match.cuh"
#include "prefill_build.cuh"

namespace {

struct StepArgs {
    SamStaticView S;
    SamBatchView W;
    int32_t has_static;
    const int32_t* new_tokens; int32_t stride; const int32_t* counts; int32_t L;
    int32_t* draft_tokens; int32_t* draft_len; int32_t* match_len; int32_t* source;
    int32_t* state; int32_t* status;
    // optional completion signal for the host-array step: the last block to finish writes done_seq to
    // *done_flag (host-mapped memory) so the host can poll instead of synchronising the stream
    int32_t* done_count; int32_t* done_flag; int32_t done_seq;
    // small host-array steps: where set, slot b's outputs go to row b of this host-mapped buffer, L + 7 words (draft,
    // draft_len, match_len[2], source, state[2], status), each with the step's number beside it (sam_step_host)
    uint2* tagged; uint32_t tag;
    // optional fused greedy verification (Section 2.2): when v_draft is set, new_tokens holds the target
    // model's tokens [B, stride] with stride = previous draft length limit + 1, and each slot's count is
    // derived here: the confirmed prefix of its previous draft plus the target's next token
    const int32_t* v_draft; const int32_t* v_draft_len; const int32_t* v_max_new;
    int32_t* v_counts_out; int32_t* v_accepted_out;
    // optional: block i works on slot order[i] (slots with many tokens first; see order_slots_kernel)
    const int32_t* order;
    // split step (sam_step_split_kernel): blocks [0, n_warp_blocks) run the static side of one slot each (the
    // first *split_count slots of `order`, those with many tokens), the next n_lane_blocks blocks the static
    // side of 32 slots each, the remaining blocks the dynamic side of one slot each
    int32_t n_warp_blocks, n_lane_blocks;
    const int32_t* split_count;
};

// ------------------------------------------------------------------ draft read
// d[r] (lane j of round r) = text[e + 32 r + j] for 32 r + j < dl, else -1.  The window is read as
// aligned 16-byte vectors (nine lanes per 32 tokens) and realigned with shuffles.
// READ: 0 plain loads, 1 read-only path (text that no kernel writes), 2 loads that bypass the L1 (text
// written by another block of the grid that is running).
template <int READ>
__device__ __forceinline__ void gather_draft(const int32_t* text, int64_t e, int dl, int L, int lane,
                                             int32_t d[MAX_DRAFT_REGS]) {
    const int off = (int)(e & 3);
    const int4* v = reinterpret_cast<const int4*>(text + (e - off));
    const int nvec = (off + dl + 3) >> 2;
    const int src = (off + lane) >> 2, comp = (off + lane) & 3;
#pragma unroll
    for (int r = 0; r < MAX_DRAFT_REGS; r++) {
        d[r] = -1;
        if (r * 32 < L) {
            int4 q = make_int4(0, 0, 0, 0);
            const int vi = 8 * r + lane;
            if (lane < 9 && vi < nvec) q = READ == 1 ? __ldg(v + vi) : READ == 2 ? __ldcg(v + vi) : v[vi];
            int x0 = __shfl_sync(FULL, q.x, src), x1 = __shfl_sync(FULL, q.y, src);
            int x2 = __shfl_sync(FULL, q.z, src), x3 = __shfl_sync(FULL, q.w, src);
            int val = comp == 0 ? x0 : comp == 1 ? x1 : comp == 2 ? x2 : x3;
            if (r * 32 + lane < dl) d[r] = val;
        }
    }
}

// A draft ends before the first stop token (the separator between documents of a concatenated
// corpus): returns the shortened length and blanks the lanes from there on.
__device__ __forceinline__ int cut_at_stop(int32_t d[MAX_DRAFT_REGS], int dl, int lane, int32_t stop) {
    if (stop < 0) return dl;
#pragma unroll
    for (int r = 0; r < MAX_DRAFT_REGS; r++) {
        const unsigned hit = __ballot_sync(FULL, r * 32 + lane < dl && d[r] == stop);
        if (hit) { dl = r * 32 + __ffs(hit) - 1; break; }
    }
#pragma unroll
    for (int r = 0; r < MAX_DRAFT_REGS; r++) if (r * 32 + lane >= dl) d[r] = -1;
    return dl;
}

// ------------------------------------------------------------------ dynamic side
struct Dyn {
    unsigned char* pool;
    uint2* root;                 // this slot's root table
    int32_t* text;               // this slot's token text
    uint32_t* pstate;            // this slot's position -> state map (the state each token created)
    int32_t* pool_hdr; int32_t* free_stack; int32_t* slab_owner;
    uint32_t* cb;                // this slot's control block
    uint32_t tab;                // lane i: slab index of state slab i
    uint32_t n_rec_slabs, n_states, blk_cur, blk_end, root_deg, root_bmask;
    int slab_shift, rps_shift, seq, lane, err;
    // Root-table lookups settled ahead of time, one lane per token of the current chunk of 32
    // (root_precompute): pr_state 0 = not known (or stale), 1 = present, 2 = absent.
    uint32_t pr_state, pr_tgt, pr_slot, pr_bucket;
    int cur;                     // lane that holds the answer for the token being processed
    mutable ChainCounts kc;      // rounds, walk-inserts, clones, copied transitions, redirects
};

struct Pre {                     // records read ahead for the clone branch of Expand, kept in shared memory
    bool valid;
    uint32_t q;                  // rec[0..1] is the record of q, rec[2..3] that of link[s2] (if it is not the root)
    const uint4* rec;
};

struct Look {                    // result of looking a token up in a non-root state
    uint32_t len, link, deg, b0, b1, b2, b3;
    uint32_t tgt;                // transition target with its S bit, valid if found
    uint32_t idx;                // 0 / 1 inline slot, or index in the edge block
    bool found;
    uint4* rp;                   // the record
};

__device__ __forceinline__ uint4* rec_ptr(const Dyn& D, uint32_t s) {
    uint32_t slab = __shfl_sync(FULL, D.tab, (int)(s >> D.rps_shift));
    return reinterpret_cast<uint4*>(D.pool + ((size_t)slab << D.slab_shift) +
                                    ((size_t)(s & ((1u << D.rps_shift) - 1)) << 5));
}
__device__ __forceinline__ uint2* blk_ptr(const Dyn& D, uint32_t off) {
    return reinterpret_cast<uint2*>(D.pool + (size_t)off * 128);
}

// (Out of line: it is needed in nine places and seldom runs.)
__device__ __noinline__ int take_slab(int32_t* pool_hdr, int32_t* free_stack, int32_t* slab_owner, int seq) {
    int idx = -1;
    if ((threadIdx.x & 31) == 0) {
        int old = atomicSub(pool_hdr, 1);
        if (old <= 0) atomicAdd(pool_hdr, 1);
        else { idx = free_stack[old - 1]; slab_owner[idx] = seq; }
    }
    return __shfl_sync(FULL, idx, 0);
}
__device__ __forceinline__ int alloc_slab(Dyn& D) { return take_slab(D.pool_hdr, D.free_stack, D.slab_owner, D.seq); }

// make sure state id s has a record to live in
__device__ __forceinline__ void ensure_rec(Dyn& D, uint32_t s) {
    uint32_t si = s >> D.rps_shift;
    if (si < D.n_rec_slabs) return;
    if (si >= SAM_MAX_REC_SLABS) { D.err = SAM_SEQ_CAPACITY; return; }
    int slab = alloc_slab(D);
    if (slab < 0) { D.err = SAM_SEQ_CAPACITY; return; }
    if (D.lane == (int)si) D.tab = (uint32_t)slab;
    if (D.lane == 0) D.cb[CB_SLABTAB + si] = (uint32_t)slab;
    D.n_rec_slabs = si + 1;
}
// State slabs of a slot that has n_rec_slabs of them, up to number `upto` or as many as there are: {this lane's slab, how many now}.
__device__ __noinline__ uint2 take_rec_slabs(int32_t* pool_hdr, int32_t* free_stack, int32_t* slab_owner, int seq, uint32_t* cb,
                                             uint32_t upto, uint32_t n_rec_slabs, uint32_t tab) {
    for (; n_rec_slabs <= upto && n_rec_slabs < SAM_MAX_REC_SLABS; n_rec_slabs++) {
        const int slab = take_slab(pool_hdr, free_stack, slab_owner, seq);
        if (slab < 0) break;
        if ((threadIdx.x & 31) == n_rec_slabs) tab = (uint32_t)slab;
        if ((threadIdx.x & 31) == 0) cb[CB_SLABTAB + n_rec_slabs] = (uint32_t)slab;
    }
    return make_uint2(tab, n_rec_slabs);
}

// Make sure of records for n states from s on, fewer than a slab holds; returns how many there are.  Where the pool has no slab left
// that may be fewer: the tokens before the one that fails are done all the same.
// How that rare case is written matters, since it stands in four places of the chain that a step waits for (us a step):
//   - F::call, a call: the single steps' kernels.  With a loop in each place they spilled on every token's way (sam_step_kernel<false, 0>
//     56/92 bytes stored/loaded, 8/40 now; the split kernel 62/100, 6/8 now): 2000 slots 15.1, now 14.8; 8191 slots 40.0, 39.3;
//     12000 slots 48.1, 47.6; 1000 slots 12.9, 12.6;
//   - in place, all tokens of a run or none: the verified steps' kernel of 80 registers, 1000 slots 18.4 (a call: 19.0);
//   - F::chunks, in place and as many tokens as there are: replays, whose kernels spill nothing (a call: 1 to 2 % slower).
template <class F>
__device__ __forceinline__ uint32_t ensure_recs(Dyn& D, uint32_t s, uint32_t n) {
    const uint32_t upto = (s + n - 1) >> D.rps_shift;
    if (upto < D.n_rec_slabs) return n;
    if (F::call) {
        const uint2 r = take_rec_slabs(D.pool_hdr, D.free_stack, D.slab_owner, D.seq, D.cb, upto, D.n_rec_slabs, D.tab);
        D.tab = r.x; D.n_rec_slabs = r.y;
    } else {
        ensure_rec(D, s);
        if (!D.err) ensure_rec(D, s + n - 1);
        D.err = 0;
    }
    const uint32_t there = D.n_rec_slabs << D.rps_shift;
    if (there <= s) { D.err = SAM_SEQ_CAPACITY; return 0; }
    return min(n, there - s);
}
template <class F>
__device__ __forceinline__ void ensure_next(Dyn& D, uint32_t s) {        // of one state
    if (F::call) ensure_recs<F>(D, s, 1);
    else ensure_rec(D, s);
}
// of a run of r tokens that make `per` states each; returns how many tokens there are records for (all or none in a kernel that neither
// calls nor has steps to end inside the run)
template <class F>
__device__ __forceinline__ int ensure_run(Dyn& D, uint32_t s, int r, int per) {
    if (F::call || F::chunks) return (int)ensure_recs<F>(D, s, (uint32_t)(per * r)) / per;
    ensure_rec(D, s);
    if (!D.err) ensure_rec(D, s + (uint32_t)(per * r) - 1);
    return D.err ? 0 : r;
}

// edge block of `cap` entries; returns its offset in 128-byte units from the pool base
__device__ __forceinline__ uint32_t alloc_block(Dyn& D, uint32_t cap) {
    uint32_t need = cap >> 4, slab_units = 1u << (D.slab_shift - 7);
    if (need > slab_units) { D.err = SAM_SEQ_CAPACITY; return 0; }
    if (D.blk_cur + need > D.blk_end) {
        int slab = alloc_slab(D);
        if (slab < 0) { D.err = SAM_SEQ_CAPACITY; return 0; }
        D.blk_cur = (uint32_t)slab << (D.slab_shift - 7);
        D.blk_end = D.blk_cur + slab_units;
    }
    uint32_t off = D.blk_cur;
    D.blk_cur += need;
    return off;
}

__device__ __forceinline__ Look lookup_state(const Dyn& D, uint32_t p, uint32_t t,
                                             bool have_rec = false, uint4 pa = make_uint4(0, 0, 0, 0),
                                             uint4 pb = make_uint4(0, 0, 0, 0)) {
    uint4 a = pa, b = pb;
    Look r;
    r.rp = rec_ptr(D, p);
    if (!have_rec) { a = r.rp[0]; b = r.rp[1]; SAM_COUNT(D.kc.rounds, 1); }
    r.len = a.x; r.link = a.y; r.deg = a.w; r.b0 = b.x; r.b1 = b.y; r.b2 = b.z; r.b3 = b.w;
    r.found = false; r.tgt = 0; r.idx = 0;
    if (a.w <= 2) {
        if (a.w >= 1 && b.x == t) { r.found = true; r.tgt = b.y; r.idx = 0; }
        else if (a.w == 2 && b.z == t) { r.found = true; r.tgt = b.w; r.idx = 1; }
        return r;
    }
    // 128 entries per round trip, four a lane in two reads that go out together
    const uint4* blk = reinterpret_cast<const uint4*>(blk_ptr(D, b.x));
    for (uint32_t base = 0; base < a.w; base += 128) {
        SAM_COUNT(D.kc.rounds, 1);
        const uint32_t i0 = base + 2u * D.lane, i1 = i0 + 64;
        uint4 e0 = make_uint4(SAM_NONE, 0, SAM_NONE, 0), e1 = e0;
        if (i0 < a.w) e0 = blk[i0 >> 1];
        if (i1 < a.w) e1 = blk[i1 >> 1];
        const bool x0 = e0.x == t, x1 = e1.x == t;                       // (what lies past the last transition is not looked at)
        const bool m0 = x0 || (e0.z == t && i0 + 1 < a.w), m1 = x1 || (e1.z == t && i1 + 1 < a.w);
        const unsigned hit = __ballot_sync(FULL, m0 || m1);
        if (hit) {
            const int src = __ffs(hit) - 1;
            r.found = true;
            r.tgt = __shfl_sync(FULL, m0 ? (x0 ? e0.y : e0.w) : (x1 ? e1.y : e1.w), src);
            r.idx = __shfl_sync(FULL, m0 ? i0 + !x0 : i1 + !x1, src);
            break;
        }
    }
    return r;
}

// add the transition (p, t) -> tgt to a non-root state whose record is in lk
__device__ __forceinline__ void insert_edge(Dyn& D, const Look& lk, uint32_t t, uint32_t tgt) {
    uint4* rp = lk.rp;
    uint32_t* rw = reinterpret_cast<uint32_t*>(rp);
    if (lk.deg < 2) {
        if (D.lane == 0) {
            reinterpret_cast<uint2*>(rp)[2 + lk.deg] = make_uint2(t, tgt);
            rw[3] = lk.deg + 1;
        }
    } else if (lk.deg == 2) {
        uint32_t off = alloc_block(D, SAM_BLOCK_MIN);
        if (D.err) return;
        if (D.lane == 0) {
            uint2* blk = blk_ptr(D, off);
            blk[0] = make_uint2(lk.b0, lk.b1); blk[1] = make_uint2(lk.b2, lk.b3); blk[2] = make_uint2(t, tgt);
            rp[1] = make_uint4(off, SAM_BLOCK_MIN, 0, 0);
            rw[3] = 3;
        }
    } else {
        uint32_t off = lk.b0, cap = lk.b1;
        if (lk.deg < cap) {
            if (D.lane == 0) { blk_ptr(D, off)[lk.deg] = make_uint2(t, tgt); rw[3] = lk.deg + 1; }
        } else {
            uint32_t noff = alloc_block(D, cap * 2);
            if (D.err) return;
            const uint2* ob = blk_ptr(D, off);
            uint2* nb = blk_ptr(D, noff);
            for (uint32_t i = D.lane; i < lk.deg; i += 32) nb[i] = ob[i];
            if (D.lane == 0) {
                nb[lk.deg] = make_uint2(t, tgt);
                rp[1] = make_uint4(noff, cap * 2, 0, 0);
                rw[3] = lk.deg + 1;
            }
        }
    }
    __syncwarp();
}

struct RootLook { uint32_t tgt, slot; bool found; };

// Each lane looks its own token up in the root table by itself: the home bucket (64 bytes, four
// 16-byte reads) settles it when the token is there, or when the bucket still has an empty entry
// (linear probing never skips one).  All tokens of the chunk are looked up in one round trip,
// before any of them is processed; later changes to the table mark the affected answers stale.
__device__ __forceinline__ void root_precompute(Dyn& D, uint32_t tk, bool valid) {
    D.pr_state = 0; D.pr_tgt = 0; D.pr_slot = 0; D.pr_bucket = SAM_NONE;
    if (!valid) return;
    const uint32_t home = sam_hash1(tk) & D.root_bmask;
    const uint4* bk = reinterpret_cast<const uint4*>(D.root + (size_t)home * SAM_ROOT_BUCKET);
    uint4 v[4];
#pragma unroll
    for (int i = 0; i < 4; i++) v[i] = bk[i];
    D.pr_bucket = home;
    int first_empty = -1;
#pragma unroll
    for (int i = 3; i >= 0; i--) {                       // descending, so the lowest index wins
        if (v[i].z == SAM_NONE) first_empty = 2 * i + 1;
        if (v[i].x == SAM_NONE) first_empty = 2 * i;
    }
#pragma unroll
    for (int i = 0; i < 4; i++) {
        if (v[i].x == tk) { D.pr_state = 1; D.pr_tgt = v[i].y; D.pr_slot = home * SAM_ROOT_BUCKET + 2 * i; }
        if (v[i].z == tk) { D.pr_state = 1; D.pr_tgt = v[i].w; D.pr_slot = home * SAM_ROOT_BUCKET + 2 * i + 1; }
    }
    if (D.pr_state == 0 && first_empty >= 0) { D.pr_state = 2; D.pr_slot = home * SAM_ROOT_BUCKET + first_empty; }
}

// A lookup that was not settled ahead of time, 32 entries a round: {found (2: table full), target, slot, rounds}
__device__ __noinline__ uint4 root_probe(const uint2* root, uint32_t bmask, uint32_t t) {
    const uint32_t cap_mask = (bmask + 1) * SAM_ROOT_BUCKET - 1, base = (sam_hash1(t) & bmask) * SAM_ROOT_BUCKET;
    const uint32_t lane = threadIdx.x & 31;
    for (uint32_t off = 0; off <= cap_mask; off += 32) {
        const uint2 e = root[(base + off + lane) & cap_mask];
        const unsigned hit = __ballot_sync(FULL, e.x == t);
        if (hit) {
            const int src = __ffs(hit) - 1;
            return make_uint4(1, __shfl_sync(FULL, e.y, src), (base + off + src) & cap_mask, off / 32 + 1);
        }
        const unsigned empty = __ballot_sync(FULL, e.x == SAM_NONE);
        if (empty) return make_uint4(0, 0, (base + off + (__ffs(empty) - 1)) & cap_mask, off / 32 + 1);
    }
    return make_uint4(2, 0, 0, 0);
}

__device__ __forceinline__ RootLook root_lookup(Dyn& D, uint32_t t) {
    RootLook r; r.found = false; r.tgt = 0; r.slot = 0;
    const uint32_t st = __shfl_sync(FULL, D.pr_state, D.cur);
    if (st != 0) {                                       // settled ahead of time and still current
        r.found = st == 1;
        r.tgt = __shfl_sync(FULL, D.pr_tgt, D.cur);
        r.slot = __shfl_sync(FULL, D.pr_slot, D.cur);
        return r;
    }
    const uint4 x = root_probe(D.root, D.root_bmask, t);
    SAM_COUNT(D.kc.rounds, x.w);
    r.found = x.x == 1; r.tgt = x.y; r.slot = x.z;
    if (x.x == 2) D.err = SAM_SEQ_WALK_LIMIT;             // table full: cannot happen with root_cap >= 2 * distinct tokens
    return r;
}

// new root transition; answers settled ahead of time for the bucket it lands in are no longer current
__device__ __forceinline__ void root_insert(Dyn& D, uint32_t slot, uint32_t t, uint32_t tgt) {
    if (D.lane == 0) D.root[slot] = make_uint2(t, tgt);
    if (D.pr_bucket == slot / SAM_ROOT_BUCKET) D.pr_state = 0;
    __syncwarp();
    D.root_deg++;
}
// change the target of an existing root transition
__device__ __forceinline__ void root_retarget(Dyn& D, uint32_t slot, uint32_t tgt) {
    if (D.lane == 0) D.root[slot].y = tgt;
    if (D.pr_state == 1 && D.pr_slot == slot) D.pr_tgt = tgt;
}

// The redirect loop of Expand's clone branch (Algorithm 3): from state pp up the suffix links, every
// t-transition that leads to q is pointed to the clone cl instead; the walk ends at the first state
// whose t-transition leads elsewhere, or past the root.  If first, (na, nb2) is the record of pp.
__device__ __forceinline__ void redirect_walk(Dyn& D, uint32_t pp, uint32_t t, uint32_t q, uint32_t cl, int guard,
                                              bool first, uint4 na, uint4 nb2) {
    for (;;) {
        if (pp == 0) {
            RootLook r2 = root_lookup(D, t);
            if (D.err) return;
            if (r2.found && (r2.tgt & SAM_IDMASK) == q) { root_retarget(D, r2.slot, cl); SAM_COUNT(D.kc.d, 1); }
            return;
        }
        Look l2k = lookup_state(D, pp, t, first, na, nb2);
        first = false;
        if (!l2k.found) { D.err = SAM_SEQ_WALK_LIMIT; return; }   // every state up the chain has t
        if ((l2k.tgt & SAM_IDMASK) != q) return;
        uint32_t* rw2 = reinterpret_cast<uint32_t*>(l2k.rp);
        if (D.lane == 0) {
            if (l2k.deg <= 2) rw2[5 + 2 * l2k.idx] = cl;
            else blk_ptr(D, l2k.b0)[l2k.idx].y = cl;
        }
        SAM_COUNT(D.kc.d, 1);
        pp = l2k.link;
        if (--guard < 0) { D.err = SAM_SEQ_WALK_LIMIT; return; }
    }
}

// Expand (Algorithm 3) for token t, fused with the dynamic matcher's Transfer.
// last: state of the whole text; ntok: text length; (s2, l2): match state = link[last], its length.
// On entry, if have_rec, (pa, pb) is the record of s2 as it stands; on exit have_rec says whether
// (pa, pb) is the record of the new s2 (known without a read when s2 is a fresh clone).
template <class F>
__device__ __forceinline__ void dyn_extend(Dyn& D, uint32_t t, uint32_t& last, uint32_t& ntok,
                                           uint32_t& s2, uint32_t& l2, bool& have_rec, uint4& pa, uint4& pb,
                                           const Pre& pre) {
    bool use_rec = have_rec;
    have_rec = false;
    const uint32_t k = ntok + 1;                       // max_length after this token
    const uint32_t c = D.n_states;
    ensure_next<F>(D, c);
    if (D.err) return;
    D.n_states = c + 1;

    uint32_t p;
    if (last != 0) {
        // `last` has no transition yet; it gets (t -> c), solid, and its record is complete now
        uint4* rl = rec_ptr(D, last);
        if (D.lane == 0) {
            rl[0] = make_uint4(ntok, s2, ntok, 1);
            rl[1] = make_uint4(t, c | SAM_FLAG, 0, 0);
        }
        __syncwarp();
        SAM_COUNT(D.kc.a, 1);
        p = s2;                                        // link[last]
    } else {
        p = 0;                                         // empty automaton: last is the root
    }

    // walk the suffix links from p, adding (t -> c) until a state already has t
    bool found = false, at_root = false;
    uint32_t qt = 0, plen = 0, root_slot = 0;
    Look lk;
    lk.len = lk.link = lk.deg = lk.b0 = lk.b1 = lk.b2 = lk.b3 = lk.tgt = lk.idx = 0; lk.found = false; lk.rp = nullptr;
    int guard = (int)k + 2;
    for (;;) {
        if (p == 0) {
            RootLook rl = root_lookup(D, t);
            if (D.err) return;
            if (rl.found) { found = true; at_root = true; qt = rl.tgt; plen = 0; root_slot = rl.slot; }
            else {
                root_insert(D, rl.slot, t, c | (k == 1 ? SAM_FLAG : 0u));
                SAM_COUNT(D.kc.a, 1);
            }
            break;
        }
        lk = lookup_state(D, p, t, use_rec, pa, pb);
        use_rec = false;
        if (lk.found) { found = true; qt = lk.tgt; plen = lk.len; break; }
        insert_edge(D, lk, t, c);                   // len[p] + 1 < k: not solid
        SAM_COUNT(D.kc.a, 1);
        if (D.err) return;
        p = lk.link;
        if (--guard < 0) { D.err = SAM_SEQ_WALK_LIMIT; return; }
    }

    if (!found) {                                      // walked past the root
        s2 = 0; l2 = 0;
    } else {
        const uint32_t q = qt & SAM_IDMASK;
        if (qt & SAM_FLAG) {                           // len[p] + 1 == len[q]
            s2 = q; l2 = plen + 1;
        } else {
            // clone q as cl with len[p] + 1
            const uint32_t cl = D.n_states;
            ensure_next<F>(D, cl);
            if (D.err) return;
            D.n_states = cl + 1;
            uint4* rq = rec_ptr(D, q);
            // the redirect walk's first read (the record of link[p]) does not depend on q's record:
            // both go out together.  link[p] is neither p, q nor cl, so nothing below changes it.
            const bool ahead = !at_root && lk.link != 0;
            const uint4* rn = rec_ptr(D, ahead ? lk.link : q);
            uint4 qa, qb, na = make_uint4(0, 0, 0, 0), nb2 = make_uint4(0, 0, 0, 0);
            if (pre.valid && pre.q == q) {              // both were read by a run attempt that did not apply
                qa = pre.rec[0]; qb = pre.rec[1];
                if (ahead) { na = pre.rec[2]; nb2 = pre.rec[3]; }
            } else {
                qa = rq[0]; qb = rq[1];
                if (ahead) { na = rn[0]; nb2 = rn[1]; }
                SAM_COUNT(D.kc.rounds, 1);
            }
            SAM_COUNT(D.kc.b, 1); SAM_COUNT(D.kc.c, qa.w); SAM_COUNT(D.kc.d, 1);   // the clone, its copied transitions, p's own redirect
            uint4 nb;
            if (qa.w <= 2) {
                nb = make_uint4(qb.x, qb.y & SAM_IDMASK, qb.z, qb.w & SAM_IDMASK);   // copies are never solid
            } else {
                uint32_t noff = alloc_block(D, qb.y);
                if (D.err) return;
                const uint2* ob = blk_ptr(D, qb.x);
                uint2* nbk = blk_ptr(D, noff);
                for (uint32_t i = D.lane; i < qa.w; i += 32) { uint2 e = ob[i]; e.y &= SAM_IDMASK; nbk[i] = e; }
                nb = make_uint4(noff, qb.y, 0, 0);
            }
            uint4* rc = rec_ptr(D, cl);
            if (D.lane == 0) {
                rc[0] = make_uint4(plen + 1, qa.y, qa.z, qa.w);      // link[q], min_endpos[q], deg[q]
                rc[1] = nb;
            }
            __syncwarp();
            // redirect p and the states above it whose t-transition is q
            if (at_root) {
                root_retarget(D, root_slot, cl | SAM_FLAG);
            } else {
                uint32_t* rw = reinterpret_cast<uint32_t*>(lk.rp);
                if (D.lane == 0) {
                    if (lk.deg <= 2) rw[5 + 2 * lk.idx] = cl | SAM_FLAG;
                    else blk_ptr(D, lk.b0)[lk.idx].y = cl | SAM_FLAG;
                }
                redirect_walk(D, lk.link, t, q, cl, (int)plen + 2, ahead, na, nb2);
                if (D.err) return;
            }
            if (D.lane == 0) reinterpret_cast<uint32_t*>(rq)[1] = cl;        // link[q] = cl
            __syncwarp();
            s2 = cl; l2 = plen + 1;
            have_rec = true;                                                 // cl's record as just written
            pa = make_uint4(plen + 1, qa.y, qa.z, qa.w); pb = nb;
        }
    }
    if (D.lane == 0) { D.text[ntok] = (int32_t)t; D.pstate[ntok] = c; }
    last = c; ntok = k;
}

// A run of tokens that are all new to the sequence, met while nothing is matched (s2 is the root):
// Expand for each of them is the same three writes — the previous state's record with its one
// solid transition, a root transition, the text — and none depends on another, so lanes j..j+r-1
// do one token each at once.  A token qualifies if its root lookup was settled ahead of time as
// "absent" and no earlier token of the run shares its home bucket (so slots and tokens differ).
// The token that ends the run is in it too if the root has it, by a solid transition: Expand for it is the same without the
// root transition, and the match goes on from there.  (256 slots fed by verified drafts, a fifth of whose tokens are of this kind:
// 19.3 -> 18.7 us a step; 300 slots with copied texts 11.9 -> 11.7.  Up to 888 slots, in the kernels of three warps a slot with 96
// registers and more: beyond, where throughput counts, it gives nothing or takes, us a step with / without it: 2000 slots 14.7 / 14.7,
// 4096 28.8 / 28.6, 8192 41.5 / 41.2, 12000 59.1 / 58.7, verified 1000 18.3 / 18.4, 1400 21.0 / 21.0.  Nor in chunks of replayed steps.)
// Returns the number of tokens (0: token j does not qualify); s2, l2: the match after them.
template <class F>
__device__ __forceinline__ int dyn_fresh_run(Dyn& D, uint32_t tk, int j, int cnt, unsigned bucket_peers,
                                             uint32_t& last, uint32_t& ntok, uint32_t& s2, uint32_t& l2, F& emit) {
    const unsigned from_j = ~((1u << j) - 1u);
    const unsigned lt = (1u << D.lane) - 1u;
    const bool first_of_bucket = (bucket_peers & from_j & lt) == 0;
    const unsigned elig = __ballot_sync(FULL, D.pr_state == 2 && first_of_bucket && D.lane >= j && D.lane < cnt);
    const unsigned known = F::seen ? __ballot_sync(FULL, D.pr_state == 1 && (D.pr_tgt & SAM_FLAG) && D.lane < cnt) : 0u;
    const unsigned gap = ~(elig >> j);
    const int fresh = gap ? __ffs(gap) - 1 : 32 - j;          // tokens that are new
    int r = fresh + (F::seen && j + fresh < 32 ? (int)(known >> (j + fresh) & 1u) : 0);
    if (r <= 0) return 0;
    const uint32_t c0 = D.n_states;
    r = ensure_run<F>(D, c0, r, 1);
    if (r == 0) return 0;
    const int idx = D.lane - j;
    const bool mine = idx >= 0 && idx < r, is_new = F::seen ? mine && idx < fresh : mine;
    const uint32_t c = c0 + (uint32_t)idx;
    const uint32_t prev = idx == 0 ? last : c - 1;            // the state this token's transition leaves
    const uint32_t plen = ntok + (uint32_t)idx;               // its length = tokens before this one
    uint4* rp = rec_ptr(D, mine ? prev : 1u);
    if (mine) {
        if (prev != 0) {
            rp[0] = make_uint4(plen, 0, plen, 1);             // link is the root: nothing was matched
            rp[1] = make_uint4(tk, c | SAM_FLAG, 0, 0);
        }
        if (is_new) D.root[D.pr_slot] = make_uint2(tk, c | (plen == 0 ? SAM_FLAG : 0u));
        D.text[plen] = (int32_t)tk;
        D.pstate[plen] = c;
    }
    const int n_new = F::seen ? min(r, fresh) : r;
    const unsigned run = ((n_new >= 32 ? 0u : (1u << n_new)) - 1u) << j;
    if (bucket_peers & run) D.pr_state = 0;                   // those buckets changed
    __syncwarp();
    SAM_COUNT(D.kc.a, r + n_new - (last == 0 ? 1 : 0));        // per token: the previous state's transition (none from the root) and the root's
    emit(is_new, D.lane, 0u, 0u, 0u, plen + 1, c, c + 1);
    if (F::seen && r > n_new) { s2 = __shfl_sync(FULL, D.pr_tgt, j + n_new) & SAM_IDMASK; l2 = 1; }
    D.n_states = c0 + r; D.root_deg += n_new;
    last = c0 + r - 1; ntok += r;
    return r;
}

// A run of tokens that repeat a passage of the sequence and all make Expand clone (Algorithm 3).
// While the match (state s2, length l0, first end position e) is extended by the tokens that followed
// its earliest occurrence, token k of the run reaches q_k, a state with first end position e + 1 + k,
// through a transition that is not solid: a new state c_k, a clone cl_k of q_k with length l0 + k + 1,
// the transition of the previous clone pointed to cl_k, link[q_k] = cl_k.  One Expand after the other
// finds q_k only from q_{k-1}'s record.  Here the q_k are guessed — the states of the prefixes ending at
// e + 1 + k (position -> state map) when the passage occurred once before, ids two apart when q_0 is a
// clone left by an earlier repeat — their records are read in one round trip, one lane per token, and
// checked (q_{k-1}'s transition on token k must lead to the guessed q_k); the lanes then write their
// new states side by side.  Only the redirect walks above each clone (they start at the old link of
// q_{k-1}) run one after the other.  Writing every link[q_k] before the walks gives what one Expand
// after the other gives: a walk of token k follows states shorter than l0 + k, every q_k' with k' > k
// is longer, and what a walk reads ahead (its first record) is checked not to be a q_k.
// On entry (pa, pb) is the record of s2.  Returns the number of tokens taken (0: not such a run; pre
// then offers the records read on the way to the ordinary Expand of token j).
template <class F>
__device__ __forceinline__ int dyn_repeat_run(Dyn& D, uint32_t tk, int j, int cnt, uint32_t& last, uint32_t& ntok,
                                              uint32_t& s2, uint32_t& l2, uint4& pa, uint4& pb, Pre& pre,
                                              uint32_t (*stage)[12], F& emit) {
    pre.valid = false;
    if (pa.w == 0 || pa.w > 2 || cnt - j < 2) return 0;
    const int lane = D.lane;
    const uint32_t t0 = __shfl_sync(FULL, tk, j);
    int idx0; uint32_t qt;
    if (pb.x == t0) { idx0 = 0; qt = pb.y; }
    else if (pa.w == 2 && pb.z == t0) { idx0 = 1; qt = pb.w; }
    else return 0;
    if (qt & SAM_FLAG) return 0;                               // solid: Expand does not clone
    const uint32_t q0 = qt, e = pa.z, l0 = l2, u0 = pa.y;
    const int rmax = min(cnt - j, (int)(ntok - e));            // text[e + k] must exist already
    if (rmax < 2) return 0;
    __syncwarp();

    // first round trip: the text after the earlier occurrence and the states created there; the records of q_0
    // and of link[s2] (what the ordinary Expand of token j would read, should this not be a run)
    const uint32_t tkr = __shfl_sync(FULL, tk, (j + lane) & 31);          // lane k: token k of the run
    const uint32_t tnext = __shfl_sync(FULL, tk, (j + lane + 1) & 31);
    int32_t tx = -1; uint32_t ps = SAM_NONE;
    if (lane < rmax) { tx = D.text[e + lane]; ps = D.pstate[e + lane]; }
    const uint4* rq0 = rec_ptr(D, q0);
    const uint4* ru0 = rec_ptr(D, u0 ? u0 : q0);
    uint4 qa = rq0[0], qb = rq0[1], ua = make_uint4(0, 0, 0, 0), ub = ua;
    if (u0) { ua = ru0[0]; ub = ru0[1]; }
    SAM_COUNT(D.kc.rounds, 1);
    const unsigned same = __ballot_sync(FULL, lane < rmax && (uint32_t)tx == tkr);
    // q_0 may be `last` itself (if token j does not continue the earliest occurrence), whose record is
    // only completed by the Expand of token j: what was read of it is then not used
    if (q0 != last) {
        uint4* keep = reinterpret_cast<uint4*>(&stage[0][0]);
        if (lane == 0) { keep[0] = qa; keep[1] = qb; keep[2] = ua; keep[3] = ub; }
        __syncwarp();
        pre.valid = true; pre.q = q0; pre.rec = keep;
    }
    int r = (~same) ? __ffs(~same) - 1 : 32;
    if (r < 2) return 0;
    // Where the q_k are expected: the states of the prefixes ending there if the passage occurred once
    // before (q_0 is then the prefix state); otherwise q_0 is a clone from an earlier repeat of the
    // passage, and clones made token after token have ids two apart.  Either guess is checked below.
    if (__shfl_sync(FULL, ps, 0) != q0) ps = q0 + 2 * (uint32_t)lane;

    // second round trip: the records of q_1 .. q_{r-1} (states that exist and are complete: not `last`)
    const bool exists = ps < D.n_states && ps != last;
    {
        const bool rd = lane > 0 && lane < r && exists;
        const uint4* rqk = rec_ptr(D, rd ? ps : q0);
        if (rd) { qa = rqk[0]; qb = rqk[1]; }
    }
    // q_k: inline transitions only, first end position e + 1 + k, reached by a transition that is not
    // solid; and, but for the last of the run, its transition on the next token leads to q_{k+1}
    int nidx = -1;
    if (qa.w >= 1 && qa.w <= 2 && qb.x == tnext) nidx = 0;
    else if (qa.w == 2 && qb.z == tnext) nidx = 1;
    const uint32_t ntgt = (nidx == 0 ? qb.y : qb.w) & SAM_IDMASK;
    const uint32_t psn = __shfl_down_sync(FULL, ps, 1);
    const unsigned okm = __ballot_sync(FULL, lane < r && exists && qa.w <= 2 && qa.z == e + 1 + (uint32_t)lane &&
                                                 qa.x > l0 + 1 + (uint32_t)lane);
    const unsigned nxm = __ballot_sync(FULL, nidx >= 0 && ntgt == psn);
    r = min(r, (~okm) ? __ffs(~okm) - 1 : 32);
    r = min(r, ((~nxm) ? __ffs(~nxm) - 1 : 32) + 1);
    if (r < 2) return 0;

    // third round trip: where each redirect walk starts, the old link of q_{k-1} (of s2 for k = 0)
    uint32_t u = __shfl_up_sync(FULL, qa.y, 1);
    if (lane == 0) u = u0;
    {
        const bool rd = lane > 0 && lane < r && u != 0;
        const uint4* ruk = rec_ptr(D, rd ? u : q0);
        if (rd) { ua = ruk[0]; ub = ruk[1]; }
    }
    {   // a walk's first record has been read now, before link[q_k] changes: it must not be one of the
        // q_k (the q_k are told apart by their first end positions e + 1 + k)
        const int kk = (int)ua.z - (int)e - 1;
        const uint32_t cand = __shfl_sync(FULL, ps, kk & 31);
        const unsigned inq = __ballot_sync(FULL, lane < r && u != 0 && kk >= 0 && kk < r && cand == u);
        if (inq) r = min(r, __ffs(inq) - 1);
        if (r < 2) return 0;
    }

    // Most walks end where they begin: at a state (or the root) whose transition leads elsewhere than to q_k.  Earlier walks do not
    // change that: they turn transitions from their own q to their own clone.  In long runs (chunks of replayed steps) lanes say so
    // for all tokens at once where the state's transitions are inline or the root's entry is settled.  (1.5 % there; runs within a
    // step are too short for it, 1 % the other way.)
    unsigned walks = FULL;
    if (F::chunks) {
        const uint32_t known = __shfl_sync(FULL, D.pr_state, (j + lane) & 31), to = __shfl_sync(FULL, D.pr_tgt, (j + lane) & 31);
        bool walk = true;
        if (u == 0) walk = known == 0 || (known == 1 && (to & SAM_IDMASK) == ps);
        else if (ua.w <= 2) {
            const uint32_t at = inline_target(ua, ub, tkr);
            walk = at == SAM_NONE || (at & SAM_IDMASK) == ps;              // (none: the walk reports it)
        }
        walks = __ballot_sync(FULL, walk);
    }

    *reinterpret_cast<uint4*>(&stage[lane][0]) = ua;
    *reinterpret_cast<uint4*>(&stage[lane][4]) = ub;
    *reinterpret_cast<uint4*>(&stage[lane][8]) = make_uint4(tkr, ps, u, 0);

    const uint32_t n0 = D.n_states;                            // c_k = n0 + 2k, cl_k = n0 + 2k + 1
    pre.valid = false;                                         // (its place has been used again)
    r = ensure_run<F>(D, n0, r, 2);
    if (r < 2) return 0;

    // the new states, side by side
    const bool mine = lane < r;
    const uint32_t ck = n0 + 2 * (uint32_t)lane, clk = ck + 1;
    uint4* rprev = rec_ptr(D, mine ? (lane == 0 ? last : ck - 2) : 1u);      // the state whose transition t_k leaves
    uint4* rcl = rec_ptr(D, mine ? clk : 1u);
    uint32_t* rqw = reinterpret_cast<uint32_t*>(rec_ptr(D, mine ? ps : 1u));
    uint32_t* rs2 = reinterpret_cast<uint32_t*>(rec_ptr(D, s2));
    uint4 nb = make_uint4(qb.x, qb.y & SAM_IDMASK, qb.z, qb.w & SAM_IDMASK);  // copies are never solid ...
    if (lane < r - 1) {                                                       // ... until redirected to the next clone
        if (nidx == 0) nb.y = (clk + 2) | SAM_FLAG; else nb.w = (clk + 2) | SAM_FLAG;
    }
    if (mine) {
        rprev[0] = make_uint4(ntok + lane, lane == 0 ? s2 : clk - 2, ntok + lane, 1);
        rprev[1] = make_uint4(tkr, ck | SAM_FLAG, 0, 0);
        rcl[0] = make_uint4(l0 + 1 + lane, qa.y, qa.z, qa.w);
        rcl[1] = nb;
        rqw[1] = clk;                                                         // link[q_k] = cl_k
        D.text[ntok + lane] = (int32_t)tkr;
        D.pstate[ntok + lane] = ck;
        if (lane == 0) rs2[5 + 2 * idx0] = clk | SAM_FLAG;                    // s2's transition on t_0
    }
    __syncwarp();

    // the redirect walks, one after the other; what each needs was left in shared memory by its lane
    for (int k = 0; k < r && !D.err; k++) {
        if (F::chunks && !(walks >> k & 1u)) continue;
        D.cur = j + k;
        const uint4 xa = *reinterpret_cast<const uint4*>(&stage[k][0]);
        const uint4 xb = *reinterpret_cast<const uint4*>(&stage[k][4]);
        const uint4 xc = *reinterpret_cast<const uint4*>(&stage[k][8]);       // token, q_k, start of the walk
        redirect_walk(D, xc.z, xc.x, xc.y, n0 + 2 * (uint32_t)k + 1, (int)(l0 + k) + 2, xc.z != 0, xa, xb);
    }
    if (D.err) return 0;
    SAM_COUNT(D.kc.rounds, 2);
    SAM_COUNT(D.kc.a, r); SAM_COUNT(D.kc.b, r); SAM_COUNT(D.kc.d, r);
    {
        uint32_t copied = mine ? qa.w : 0u;
        for (int o = 16; o; o >>= 1) copied += __shfl_xor_sync(FULL, copied, o);
        SAM_COUNT(D.kc.c, copied);
    }

    emit(mine, (j + lane) & 31, clk, l0 + 1 + (uint32_t)lane, qa.z, ntok + (uint32_t)lane + 1, ck, clk + 1);
    const int lr = r - 1;                                      // the last clone is the new match state
    pa = make_uint4(l0 + (uint32_t)r, __shfl_sync(FULL, qa.y, lr), __shfl_sync(FULL, qa.z, lr), __shfl_sync(FULL, qa.w, lr));
    pb = make_uint4(__shfl_sync(FULL, nb.x, lr), __shfl_sync(FULL, nb.y, lr), __shfl_sync(FULL, nb.z, lr), __shfl_sync(FULL, nb.w, lr));
    D.n_states = n0 + 2 * (uint32_t)r;
    last = n0 + 2 * (uint32_t)lr; s2 = last + 1; l2 = l0 + (uint32_t)r; ntok += (uint32_t)r;
    pre.valid = false;
    return r;
}

// The static match moved over a step's m tokens (tok_first: lane k's token of the first 32), by one warp: the
// state Transfer (Algorithm 1) reaches.  In and out: the state (s, sf, l) and, where l > 0, its record (ra, rb).
// early(): called where the match is in the state of a corpus prefix, so that the draft after m tokens can be requested
// with the first reads; returns true if the match did go on as the corpus does, for all m tokens.
template <class F>
__device__ __forceinline__ bool static_advance(const SamStaticView& S, int lane, int32_t tok_first, const int32_t* toks, int m,
                                               uint32_t& s, uint32_t& sf, int32_t& l, uint4& ra, uint4& rb, int& err, ChainCounts& kc, F early) {
#ifdef SAM_COUNTERS
    ChainCounts tally = {0, 0, 0, 0, 0};                 // the moves Algorithm 1 itself makes over these tokens
    {
        uint32_t ts = s, tsf = sf; int32_t tl = l;
        for (int j = 0; j < m && !err; j++)
            static_transfer(S, ts, tsf, tl, (uint32_t)toks[j], __ldg(S.root_row + toks[j]), lane, err, false, ra, rb, tally);
    }
#endif
    bool follows = false;
    if (m > 32) static_suffix(S, toks, m, lane, s, sf, l, ra, rb, err, kc);
    else if (m > 0) {
        const uint32_t tk = (uint32_t)tok_first;
        uint32_t re = SAM_NONE;
        if (lane < m) re = __ldg(S.root_row + tk);
        SAM_COUNT(kc.rounds, 1);
        int i0 = 0;
        bool have = s != 0, prefix = false;
        if (have) {                                      // the match so far may take the tokens in one round
            prefix = ra.x == ra.z;
            if (prefix) early();
            i0 = static_run(S, s, sf, ra, rb, have, tk, m, lane, kc);
            l += i0;
        }
        if (i0 < m) {
            static_walks(S, tk, re, m, lane, s != 0, i0, have, s, sf, l, ra, rb, err, kc);
        } else {
            if (!have) static_record(S, s, ra, rb);
            follows = prefix;
        }
    }
#ifdef SAM_COUNTERS
    kc.a = tally.a; kc.b = tally.b;
#endif
    return follows;
}

// The static side of one slot's step, run by one warp, then the static words of the control block.  cw holds
// control words 0..31 as read at the start of the step; on entry (ra, rb) is the copy of the match state's record
// kept in the control block, ntok0 the text length before the step.  On exit (s, sf, l) is the match state, and, if
// l > 0 and no error, (ra, rb) its record.  DRAFT: also fetch the draft after the state's first end position into
// d / my_dl (requested early where the address is known early).
template <bool DRAFT>
__device__ __forceinline__ void static_chain(const StepArgs& A, int b, int lane, uint32_t* cb, uint32_t cw, int32_t tok_first,
                                             const int32_t* toks, int m, uint32_t ntok0, uint4& ra, uint4& rb,
                                             uint32_t& s_out, uint32_t& sf_out, int32_t& l_out, int& err,
                                             int32_t d[MAX_DRAFT_REGS], int32_t& my_dl) {
    const int L = A.L;
    ChainCounts kc = {1, 0, 0, 0, 0};                    // one round already: the control words
    uint32_t s = __shfl_sync(FULL, cw, CB_S1), sf = __shfl_sync(FULL, cw, CB_S1FLAG);
    int32_t l = (int32_t)__shfl_sync(FULL, cw, CB_L1);
    int dl2 = 0;
    const bool follows = static_advance(A.S, lane, tok_first, toks, m, s, sf, l, ra, rb, err, kc, [&]() {
        if (DRAFT) {
            const int64_t e2 = (int64_t)ra.z + m, room = A.S.n_tokens - e2;
            dl2 = (int)(room < L ? (room < 0 ? 0 : room) : L);
            gather_draft<1>(A.S.corpus, e2, dl2, L, lane, d);
        }
    });
    l_out = l; s_out = s; sf_out = sf;
    if (l > 0 && !err) SAM_COUNT(kc.rounds, DRAFT && !follows ? 1 : 0);
    flush_counts(b, lane, true, kc, m, m > 0);
    if (DRAFT && l > 0 && !err) {
        if (follows) my_dl = dl2;
        else {
            const int64_t e = (int64_t)ra.z;            // min_endpos
            int64_t room = A.S.n_tokens - e;
            my_dl = (int)(room < L ? (room < 0 ? 0 : room) : L);
            gather_draft<1>(A.S.corpus, e, my_dl, L, lane, d);
        }
        my_dl = cut_at_stop(d, my_dl, lane, A.W.stop_token);
    }
    if (m > 0 && lane == 0 && !err) {
        cb[CB_S1] = s; cb[CB_L1] = (uint32_t)l; cb[CB_S1FLAG] = sf; cb[CB_NTOK_S] = ntok0 + (uint32_t)m;
        if (l > 0) { reinterpret_cast<uint4*>(cb + CB_REC1)[0] = ra; reinterpret_cast<uint4*>(cb + CB_REC1)[1] = rb; }
    }
}

// The copy of a match state's record that the control block keeps (its words 32.. are in cw2).
__device__ __forceinline__ void kept_record(uint32_t cw2, int word, uint4& ra, uint4& rb) {
    const int r = word - 32;
    ra.x = __shfl_sync(FULL, cw2, r + 0); ra.y = __shfl_sync(FULL, cw2, r + 1);
    ra.z = __shfl_sync(FULL, cw2, r + 2); ra.w = __shfl_sync(FULL, cw2, r + 3);
    rb.x = __shfl_sync(FULL, cw2, r + 4); rb.y = __shfl_sync(FULL, cw2, r + 5);
    rb.z = __shfl_sync(FULL, cw2, r + 6); rb.w = __shfl_sync(FULL, cw2, r + 7);
}

// The dynamic side of one slot: its automaton and its matcher, kept by one warp for as long as it works on the slot.
struct DynChain {
    Dyn D;
    uint32_t last, ntok, s2, l2;
    bool have;                   // (ra, rb) is the record of s2
    uint4 ra, rb;
};

// cw / cw2 are the slot's 64 control words as read at the start (lane i holds words i and 32 + i); (ra, rb) of X
// is the copy of the match state's record kept there.
__device__ __forceinline__ void dyn_open(const SamBatchView& W, int b, int lane, uint32_t* cb, uint32_t cw, uint32_t cw2, DynChain& X) {
    Dyn& D = X.D;
    D.pool = W.pool;
    D.root = W.root_tab + (size_t)b * W.root_cap;
    D.text = W.text + (size_t)b * W.text_stride;
    D.pstate = W.pstate + (size_t)b * W.text_stride;
    D.pool_hdr = W.pool_hdr; D.free_stack = W.free_stack; D.slab_owner = W.slab_owner;
    D.cb = cb;
    {   // slab table entry i is control word 16 + i
        uint32_t lo = __shfl_sync(FULL, cw, (lane + 16) & 31), hi = __shfl_sync(FULL, cw2, (lane + 16) & 31);
        D.tab = lane < 16 ? lo : hi;
    }
    D.n_rec_slabs = __shfl_sync(FULL, cw, CB_NRECSLABS);
    D.n_states = __shfl_sync(FULL, cw, CB_NSTATES);
    D.blk_cur = __shfl_sync(FULL, cw, CB_BLK_CUR);
    D.blk_end = __shfl_sync(FULL, cw, CB_BLK_END);
    D.root_deg = __shfl_sync(FULL, cw, CB_ROOTDEG);
    D.root_bmask = (uint32_t)(W.root_cap / SAM_ROOT_BUCKET) - 1;
    D.slab_shift = W.slab_shift; D.rps_shift = W.slab_shift - 5;
    D.seq = b; D.lane = lane; D.err = 0;
    D.pr_state = 0; D.pr_tgt = 0; D.pr_slot = 0; D.pr_bucket = SAM_NONE; D.cur = 0;
    D.kc = ChainCounts{1, 0, 0, 0, 0};                   // one round already: the control words
    X.last = __shfl_sync(FULL, cw, CB_LAST); X.ntok = __shfl_sync(FULL, cw, CB_NTOK);
    X.s2 = __shfl_sync(FULL, cw, CB_S2); X.l2 = __shfl_sync(FULL, cw, CB_L2);
    X.have = X.s2 != 0;
    if (D.n_states == 0) D.n_states = 1;            // the root exists implicitly (no record is read for it)
}

// Expand (fused with the dynamic matcher's Transfer) for each of up to 32 tokens, one in each lane.  emit is called by the whole
// warp whenever tokens are done, with what holds after them: (whether this lane has one, the lane that held its token, s2, l2,
// first end position of s2, text length, state of the whole text, number of states); ends: the tokens for which it is wanted.
// seen: runs of new tokens take the known one behind them (dyn_fresh_run).  call, chunks: ensure_recs.
template <bool SEEN, bool CALL>
struct NoEmit {
    static constexpr bool chunks = false, seen = SEEN, call = CALL;
    static constexpr unsigned ends = 0;
    __device__ __forceinline__ void operator()(bool, int, uint32_t, uint32_t, uint32_t, uint32_t, uint32_t, uint32_t) const {}
};
template <class F>
__device__ __forceinline__ void dyn_emit(DynChain& X, int j, F& emit) {    // after token j
    if (X.l2 > 0 && !X.have) { const uint4* rs = rec_ptr(X.D, X.s2); X.ra = rs[0]; X.rb = rs[1]; X.have = true; SAM_COUNT(X.D.kc.rounds, 1); }
    emit(X.D.lane == j, X.D.lane, X.s2, X.l2, X.ra.z, X.ntok, X.last, X.D.n_states);
}
template <class F>
__device__ __forceinline__ void dyn_tokens(DynChain& X, uint32_t tk, int cnt, uint32_t (*sh_run)[12], F& emit) {
    Dyn& D = X.D;
    root_precompute(D, tk, D.lane < cnt);           // most walks end in the root table
    SAM_COUNT(D.kc.rounds, 1);
    const unsigned bucket_peers = __match_any_sync(FULL, D.pr_bucket);
    int j = 0;
    while (j < cnt && !D.err) {
        if (X.s2 == 0) {
            const int r = dyn_fresh_run(D, tk, j, cnt, bucket_peers, X.last, X.ntok, X.s2, X.l2, emit);
            if (r > 0) {
                j += r;
                X.have = false;
                continue;
            }
            if (D.err) break;
        }
        Pre pre;
        pre.valid = false;
        if (X.s2 != 0 && X.have) {
            const int r = dyn_repeat_run(D, tk, j, cnt, X.last, X.ntok, X.s2, X.l2, X.ra, X.rb, pre, sh_run, emit);
            if (r > 0) { j += r; continue; }
            if (D.err) break;
        }
        D.cur = j;
        dyn_extend<F>(D, __shfl_sync(FULL, tk, j), X.last, X.ntok, X.s2, X.l2, X.have, X.ra, X.rb, pre);
        if ((emit.ends >> j & 1u) && !D.err) dyn_emit(X, j, emit);
        j++;
    }
}
// The newest state's record, without a transition yet, and the slot's control words.
__device__ __forceinline__ void dyn_close(DynChain& X) {
    uint4* rl = rec_ptr(X.D, X.last);
    uint32_t* cb = X.D.cb;
    if (X.D.lane == 0) {
        rl[0] = make_uint4(X.ntok, X.s2, X.ntok, 0);
        rl[1] = make_uint4(0, 0, 0, 0);
        cb[CB_NTOK] = X.ntok; cb[CB_NSTATES] = X.D.n_states; cb[CB_LAST] = X.last;
        cb[CB_S2] = X.s2; cb[CB_L2] = X.l2; cb[CB_BLK_CUR] = X.D.blk_cur; cb[CB_BLK_END] = X.D.blk_end;
        cb[CB_NRECSLABS] = X.D.n_rec_slabs; cb[CB_ROOTDEG] = X.D.root_deg;
    }
    __syncwarp();
}
// A step's m tokens, then the slot's control words.  On return, unless D.err is set, (ra, rb) is the record of s2 if l2 > 0 (also
// stored in the control block).
template <bool SEEN, bool CALL>
__device__ __forceinline__ void dyn_feed(DynChain& X, int32_t tok_first, const int32_t* toks, int m, uint32_t (*sh_run)[12]) {
    Dyn& D = X.D;
    const int lane = D.lane;
    NoEmit<SEEN, CALL> none;
    for (int base = 0; base < m && !D.err; base += 32) {
        const int i = base + lane;
        uint32_t tk = 0;
        if (i < m) tk = (uint32_t)(base == 0 ? tok_first : toks[i]);
        dyn_tokens(X, tk, min(32, m - base), sh_run, none);
    }
    if (m > 0 && !D.err) dyn_close(X);
    if (X.l2 > 0 && !D.err) SAM_COUNT(D.kc.rounds, 1);   // the draft
    if (X.l2 > 0 && !D.err && m > 0) {                  // the state moved: get its record, keep a copy
        if (!X.have) { const uint4* rs = rec_ptr(D, X.s2); X.ra = rs[0]; X.rb = rs[1]; X.have = true; SAM_COUNT(D.kc.rounds, 1); }
        if (lane == 0) { reinterpret_cast<uint4*>(D.cb + CB_REC2)[0] = X.ra; reinterpret_cast<uint4*>(D.cb + CB_REC2)[1] = X.rb; }
    }
    if (!D.err) flush_counts(D.seq, lane, false, D.kc, m, m > 0);
}

// Called by one thread of a block after the block's outputs are written (and made known to that
// thread by a block barrier where another warp wrote some of them).
// A block orders its output stores (to mapped host memory) before its count with a device-scope fence;
// the block that counts last has thereby observed all the others, and its one system-scope fence — fences
// are cumulative — orders every block's stores before the flag the host polls.  (A system-scope fence in
// every block is what the host waited for: 3.5 us more at 64 blocks, 7 us more at 256.)
__device__ __forceinline__ void signal_done(const StepArgs& A) {
    __threadfence();
    const int prev = atomicAdd(A.done_count, 1);
    if (prev == (int)gridDim.x - 1) {
        *A.done_count = 0;
        __threadfence_system();
        *reinterpret_cast<volatile int32_t*>(A.done_flag) = A.done_seq;
    }
}

// Where a step's outputs go (step `at` of outputs that keep every step).
struct StepOut { int32_t *draft, *draft_len, *match_len, *source, *state, *status; };
__device__ __forceinline__ StepOut step_out(const StepArgs& A, int at) {
    const size_t n = (size_t)at * A.W.batch;
    return {A.draft_tokens + n * A.L, A.draft_len + n, A.match_len + 2 * n, A.source + n, A.state ? A.state + 2 * n : nullptr, A.status + n};
}

__device__ __forceinline__ void write_failed_tagged(const StepArgs& A, int b, int lane, int status) {
    uint2* row = A.tagged + (size_t)b * (A.L + 7);
    __threadfence();                                       // as in step_outputs
    for (int j = lane; j < A.L + 7; j += 32) row[j] = make_uint2(j < A.L ? 0xFFFFFFFFu : j == A.L + 6 ? (uint32_t)status : 0u, A.tag);
}

__device__ __forceinline__ void write_failed_slot(const StepOut& o, int L, int b, int lane, int status) {
    for (int j = lane; j < L; j += 32) o.draft[(size_t)b * L + j] = -1;
    if (lane == 0) {
        o.draft_len[b] = 0; o.match_len[2 * b] = 0; o.match_len[2 * b + 1] = 0; o.source[b] = 0;
        if (o.state) { o.state[2 * b] = 0; o.state[2 * b + 1] = 0; }
        o.status[b] = status;
    }
}

// Choose the source (Section 3.2), read the draft, write the outputs: by a whole warp that has both sides' results
// (match length, state, first end position; ntok: the text's length).  Other blocks of the grid may have written the text.
__device__ __forceinline__ void write_slot(const StepArgs& A, const StepOut& o, int b, int lane, int l1, int s1, int64_t e1,
                                           int l2, int s2, int64_t e2, int64_t ntok) {
    const int L = A.L;
    const bool use_static = A.has_static && l1 > l2 + A.W.l_bias;
    const int lsel = use_static ? l1 : l2;
    const int need = A.W.min_match > 1 ? A.W.min_match : 1;
    const int src = lsel < need ? SAM_SRC_NONE : (use_static ? SAM_SRC_STATIC : SAM_SRC_DYNAMIC);
    int32_t d[MAX_DRAFT_REGS] = {-1, -1, -1, -1};
    int dl = 0;
    if (src != SAM_SRC_NONE) {
        const int64_t e = use_static ? e1 : e2, room = (use_static ? A.S.n_tokens : ntok) - e;
        dl = (int)(room < L ? (room < 0 ? 0 : room) : L);
        gather_draft<2>(use_static ? A.S.corpus : A.W.text + (size_t)b * A.W.text_stride, e, dl, L, lane, d);
        dl = cut_at_stop(d, dl, lane, A.W.stop_token);
    }
#pragma unroll
    for (int r = 0; r < MAX_DRAFT_REGS; r++) {
        const int j = r * 32 + lane;
        if (j < L) o.draft[(size_t)b * L + j] = d[r];
    }
    if (lane == 0) {
        o.draft_len[b] = dl; o.match_len[2 * b] = l1; o.match_len[2 * b + 1] = l2; o.source[b] = src;
        if (o.state) { o.state[2 * b] = s1; o.state[2 * b + 1] = s2; }
        o.status[b] = 0;
    }
}

// A third warp that reads ahead of the dynamic side, for batches that leave the GPU room for it.  It goes through the step's
// tokens as the dynamic side will, from every token on along the transitions of the tokens after it, but only reads: the slot's root-table buckets, records and edge blocks come into the
// SM's L1, where the dynamic side, which reads them one after the other, then finds them (a record from the L2 or beyond takes
// it 520 cycles, an edge block 810).  The dynamic side changes these structures meanwhile, so what is read here may be of
// any age; it is used for addresses only, each checked against the pool, and for no result.
// The same reads made by the dynamic side itself, before its first token, cost what they saved; following the match
// state's suffix links as well gave nothing.  Per step: 4 slots 6.2 -> 5.5 us, 64 slots 6.0 -> 5.5, 1000 slots 18.5 -> 17.0, 256
// slots fed by verified drafts 26.2 -> 21.5.
struct Ahead {
    const unsigned char* pool;
    uint32_t tab, n_states, n_units;      // lane i: slab index of state slab i; states and 128-byte units that may be read
    int slab_shift, lane;
};
__device__ __forceinline__ uint4 ahead_load(const void* p) {
    uint4 v;
    asm volatile("ld.global.ca.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
    return v;
}
// The record of state s of each lane that wants one.
__device__ __forceinline__ void ahead_records(const Ahead& H, bool want, uint32_t s, uint4& a, uint4& b) {
    want = want && s != 0 && s < H.n_states;
    const int rps_shift = H.slab_shift - 5;
    const uint32_t slab = __shfl_sync(FULL, H.tab, want ? (int)(s >> rps_shift) : 0);
    a = b = make_uint4(0, 0, 0, 0);
    if (want) {
        const unsigned char* p = H.pool + ((size_t)slab << H.slab_shift) + ((size_t)(s & ((1u << rps_shift) - 1)) << 5);
        a = ahead_load(p); b = ahead_load(p + 16);
    }
}
// Where each lane's state (record a, b) leads on token t: looked for in all lanes' edge blocks.
__device__ __forceinline__ uint32_t ahead_targets(const Ahead& H, const uint4& a, const uint4& b, uint32_t t) {
    uint32_t q = 0;
    if (a.w >= 1 && a.w <= 2) { if (b.x == t) q = b.y; else if (a.w == 2 && b.z == t) q = b.w; }
    const bool wide = a.w > 2 && a.w <= 512 && b.x + ((a.w + 15) >> 4) <= H.n_units && b.x < H.n_units;
    const unsigned todo = __ballot_sync(FULL, wide);
    for (unsigned w = todo; w; w &= w - 1) {               // every line of every block asked for ...
        const int k = __ffs(w) - 1;
        const uint32_t deg = __shfl_sync(FULL, a.w, k), off = __shfl_sync(FULL, b.x, k);
        if ((uint32_t)H.lane * 16u < deg) asm volatile("prefetch.global.L1 [%0];" ::"l"(H.pool + ((size_t)off + H.lane) * 128));
    }
    for (unsigned w = todo; w; w &= w - 1) {               // ... before any is looked through
        const int k = __ffs(w) - 1;
        const uint32_t deg = __shfl_sync(FULL, a.w, k), off = __shfl_sync(FULL, b.x, k), tk = __shfl_sync(FULL, t, k);
        for (uint32_t base = 0; base < deg; base += 64) {  // two entries a lane
            const uint32_t i = base + 2u * H.lane;
            uint4 e = make_uint4(SAM_NONE, 0, SAM_NONE, 0);
            if (i < deg) e = ahead_load(H.pool + (size_t)off * 128 + (size_t)i * 8);
            const bool first = e.x == tk, second = e.z == tk && i + 1 < deg;
            const unsigned hit = __ballot_sync(FULL, first || second);
            if (hit) {
                const uint32_t v = __shfl_sync(FULL, first ? e.y : e.w, __ffs(hit) - 1);
                if (H.lane == k) q = v;
                break;
            }
        }
    }
    return q & SAM_IDMASK;
}
// A barrier of all three warps; whether x holds for any thread.  (Not the barrier of step_sync: the third warp may come to this
// one before the others have passed that.)
__device__ __forceinline__ bool step_join(bool x) {
    uint32_t r;
    asm volatile("{ .reg .pred p, q; setp.ne.u32 p, %1, 0; bar.red.or.pred q, 2, 96, p; selp.u32 %0, 1, 0, q; }" : "=r"(r) : "r"((uint32_t)x) : "memory");
    return r != 0;
}
// The third warp's part in it, once what it read last has arrived: its vote depends on that (and says nothing).  Out of line,
// so that a step nobody waits for in this way does not wait for those reads.
__device__ __noinline__ void ahead_join(uint32_t x, uint32_t y, uint32_t z) { step_join(x + (y ^ z) == 0xFFFFFFFFu); }

constexpr int AHEAD_MIN_TOKENS = 2, AHEAD_LEVELS = 4;
// join: end with ahead_join.
__device__ __forceinline__ void read_ahead(const SamBatchView& W, int b, int lane, uint32_t cw, uint32_t cw2, int32_t tok_first, int m, bool join) {
    const int n = m < 32 ? m : 32;
    if (n < AHEAD_MIN_TOKENS) { if (join) ahead_join((uint32_t)tok_first, 0, 0); return; }
    Ahead H;
    H.pool = W.pool; H.slab_shift = W.slab_shift; H.lane = lane;
    {
        const uint32_t lo = __shfl_sync(FULL, cw, (lane + 16) & 31), hi = __shfl_sync(FULL, cw2, (lane + 16) & 31);
        H.tab = lane < 16 ? lo : hi;
        if (H.tab >= (uint32_t)W.pool_slabs) H.tab = 0;
    }
    H.n_states = min(__shfl_sync(FULL, cw, CB_NSTATES), __shfl_sync(FULL, cw, CB_NRECSLABS) << (W.slab_shift - 5));
    H.n_units = (uint32_t)W.pool_slabs << (W.slab_shift - 7);
    const uint32_t t = (uint32_t)tok_first;
    // the token's entry in the root table, from its home bucket
    uint32_t u = 0;
    if (lane < n) {
        const uint32_t home = sam_hash1(t) & ((uint32_t)(W.root_cap / SAM_ROOT_BUCKET) - 1u);
        const uint2* bucket = W.root_tab + (size_t)b * W.root_cap + (size_t)home * SAM_ROOT_BUCKET;
#pragma unroll
        for (int i = 0; i < SAM_ROOT_BUCKET / 2; i++) {
            const uint4 e = ahead_load(bucket + 2 * i);
            if (e.x == t) u = e.y & SAM_IDMASK;
            if (e.z == t) u = e.w & SAM_IDMASK;
        }
    }
    // level by level: lane k is at the state of tokens k .. k + level - 1 and looks up token k + level
    uint4 a, bb;
    ahead_records(H, lane < n, u, a, bb);
    for (int level = 1; level <= AHEAD_LEVELS; level++) {
        const uint32_t next = __shfl_sync(FULL, t, (lane + level) & 31);
        if (lane + level >= n) a.w = 0;
        if (!__any_sync(FULL, a.w != 0)) break;
        u = ahead_targets(H, a, bb, next);
        ahead_records(H, u != 0, u, a, bb);
    }
    if (join) ahead_join(t, a.w, bb.w);
}

// Both warps' results are in shared memory: choose the source, write the slot's outputs.  Not failed: both errors are 0.
// PAIRS: to the host, each with the step's number beside it, where A.tagged says so.
template <bool VERIFY, bool PAIRS>
__device__ __forceinline__ void step_outputs(const StepArgs& A, int b, int warp, int lane, uint32_t* cb, const int32_t* sh_l, const int32_t* sh_s,
                                             const int32_t* sh_dl, const int32_t* sh_err, bool failed, const int32_t d[MAX_DRAFT_REGS], int m, int confirmed) {
    const int L = A.L;
    const int any_err = !failed ? 0 : sh_err[0] ? sh_err[0] : sh_err[1];
    const int l1 = sh_l[0], l2v = sh_l[1];
    const bool use_static = A.has_static && l1 > l2v + A.W.l_bias;        // Section 3.2
    const int lsel = use_static ? l1 : l2v;
    const int need = A.W.min_match > 1 ? A.W.min_match : 1;
    const int src = (any_err || lsel < need) ? SAM_SRC_NONE : (use_static ? SAM_SRC_STATIC : SAM_SRC_DYNAMIC);
    const int winner = src == SAM_SRC_DYNAMIC ? 1 : 0;

    if (PAIRS && A.tagged) {
        uint2* row = A.tagged + (size_t)b * (L + 7);
        if (warp == 0) {
            if (any_err && lane == 0) cb[CB_STATUS] = (uint32_t)any_err;
            // The host takes the step for done when it has all words, of which some are this warp's: what the block has changed of
            // the slot is there before them, for whatever stream the batch is used on next.
            __threadfence();
        }
        if (warp == winner) {
#pragma unroll
            for (int r = 0; r < MAX_DRAFT_REGS; r++) {
                const int j = r * 32 + lane;
                if (j < L) row[j] = make_uint2((uint32_t)(src == SAM_SRC_NONE ? -1 : d[r]), A.tag);
            }
        }
        if (warp == 0) {
            const int v = lane == 0 ? (src == SAM_SRC_NONE ? 0 : sh_dl[winner]) : lane == 3 ? src : lane == 6 ? any_err : any_err ? 0 :
                          lane == 1 ? l1 : lane == 2 ? l2v : lane == 4 ? sh_s[0] : sh_s[1];
            if (lane < 7) row[L + lane] = make_uint2((uint32_t)v, A.tag);
        }
        return;
    }
    if (warp == winner) {
#pragma unroll
        for (int r = 0; r < MAX_DRAFT_REGS; r++) {
            int j = r * 32 + lane;
            if (j < L) A.draft_tokens[(size_t)b * L + j] = (src == SAM_SRC_NONE) ? -1 : d[r];
        }
    }
    if (warp == 0 && lane == 0) {
        if (any_err) cb[CB_STATUS] = (uint32_t)any_err;
        A.draft_len[b] = src == SAM_SRC_NONE ? 0 : sh_dl[winner];
        A.match_len[2 * b] = any_err ? 0 : l1;
        A.match_len[2 * b + 1] = any_err ? 0 : l2v;
        A.source[b] = src;
        if (A.state) { A.state[2 * b] = any_err ? 0 : sh_s[0]; A.state[2 * b + 1] = any_err ? 0 : sh_s[1]; }
        A.status[b] = any_err;
        if (VERIFY && A.v_counts_out) A.v_counts_out[b] = m;
        if (VERIFY && A.v_accepted_out) A.v_accepted_out[b] = confirmed;
    }
}

// ------------------------------------------------------------------ the kernel
// The two warps that work on the slot.
__device__ __forceinline__ void step_sync() { asm volatile("bar.sync 1, 64;" ::: "memory"); }
// VERIFY: the accepted tokens are derived from the previous draft and the target's tokens (sam_step_verified).
// AHEAD: a third warp reads ahead of the dynamic side (read_ahead).
// INLINE: the rows and counts came with the launch (sam_step_host).
// SEEN, CALL: dyn_feed's.
template <bool VERIFY, bool AHEAD, bool INLINE, bool SEEN, bool CALL>
__device__ __forceinline__ void step_body(const StepArgs& A, const int32_t* new_tokens, const int32_t* counts) {
    // Programmatic dependent launch: this grid may be scheduled while the previous kernel of the stream
    // is still finishing.  Nothing is read before that kernel has completed and flushed; the kernel
    // after this one is allowed to get scheduled right away (it waits in the same way).
    if (!A.order) {
        // While the previous kernel of the stream finishes: touch (prefetch, no data is used) the lines this
        // block reads first, so that their address translations and L2 lines are at hand after the wait.
        const int pb_ = blockIdx.x, pl_ = threadIdx.x & 31;
        const char* p0 = reinterpret_cast<const char*>(A.W.ctrl + (size_t)pb_ * SAM_CTRL_WORDS);
        const char* p1 = reinterpret_cast<const char*>(new_tokens + (size_t)pb_ * A.stride);
        const char* p2 = reinterpret_cast<const char*>(VERIFY ? A.v_draft_len + pb_ : counts + pb_);
        const char* pp_ = pl_ == 0 ? p0 : pl_ == 1 ? p0 + 128 : pl_ == 2 ? p1 : p2;
        if (pl_ < (INLINE ? 2 : 4)) asm volatile("prefetch.global.L2 [%0];" ::"l"(pp_));
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
    const int b = A.order ? A.order[blockIdx.x] : (int)blockIdx.x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __shared__ int32_t sh_l[2], sh_s[2], sh_dl[2], sh_err[2];
    __shared__ __align__(16) uint32_t sh_run[32][12];   // per-token staging of a repeat run (dynamic warp)

    // Everything the step needs to get going is read in one round trip: the slot's 64 control
    // words (state, slab table, copies of the two match states' records), its count, and the
    // first 32 tokens of its row (read before the count is known; unused lanes are ignored).
    uint32_t* cb = A.W.ctrl + (size_t)b * SAM_CTRL_WORDS;
    const int32_t* toks = new_tokens + (size_t)b * A.stride;
    const uint32_t cw = cb[lane];                       // control words 0..31
    const uint32_t cw2 = cb[32 + lane];                 // control words 32..63
    int32_t tok_first = 0;
    if (lane < A.stride) tok_first = toks[lane];
    int m, confirmed = 0;
    if (VERIFY) {
        // x_accept = the draft tokens the target reproduces, then the target's own next token
        const int Lp = A.stride - 1;
        int dl = A.v_draft_len[b];
        dl = dl < 0 ? 0 : (dl > Lp ? Lp : dl);
        const int32_t* dr = A.v_draft + (size_t)b * Lp;
        int a = dl;
        for (int base = 0; base < dl; base += 32) {
            const int j = base + lane;
            const bool differs = j < dl && dr[j] != toks[j];
            const unsigned bad = __ballot_sync(FULL, differs);
            if (bad) { a = base + __ffs(bad) - 1; break; }
        }
        m = a + 1;
        if (A.v_max_new) { int cap = A.v_max_new[b]; cap = cap < 0 ? 0 : cap; m = m < cap ? m : cap; }
        confirmed = a < m ? a : m;
    } else {
        m = counts[b];
    }
    int status = (int)__shfl_sync(FULL, cw, CB_STATUS);
    const uint32_t ntok0 = __shfl_sync(FULL, cw, CB_NTOK);
    const int L = A.L;
    const bool host = AHEAD && !VERIFY && (A.tagged != nullptr || A.done_flag != nullptr);
    if (AHEAD && warp == 2) {
        // A host-array step's caller goes on before this kernel has ended, but not before this warp's reads have: of the caller's
        // arrays, which kernels may read in place, and of the batch's memory.
        if (status == 0 && m <= A.stride) read_ahead(A.W, b, lane, cw, cw2, tok_first, m, host);
        else if (host) ahead_join((uint32_t)tok_first, 0, 0);
        return;
    }
    step_sync();              // both warps hold the slot's state as it was before either writes any of it

    // what sam_prefill_kernel, launched before this one where a step may have prompts, has done of the slot
    const bool built = !VERIFY && !INLINE && (uint32_t)status == SAM_STEP_BUILT;
    if (!VERIFY && !INLINE && status < 0) {
        if (threadIdx.x == 0) cb[CB_STATUS] = 0;
        if ((uint32_t)status == SAM_STEP_DONE) {
            if (host) step_join(false);
            if (threadIdx.x == 0 && A.done_flag) signal_done(A);
            return;
        }
        status = 0;
    }

    // validate the whole step before any state changes (both warps reach the same verdict)
    bool fresh_fail = false;
    if (status == 0 && !built) {
        if (m < 0 || m > A.stride) status = SAM_SEQ_BAD_COUNT;
        else if ((int64_t)ntok0 + m > A.W.max_seq_len) status = SAM_SEQ_CAPACITY;
        else {
            const int vocab = A.has_static ? A.S.vocab : A.W.vocab;
            bool bad = false;
            for (int base = 0; base < m; base += 32) {
                int i = base + lane;
                if (i < m) { int t = base == 0 ? tok_first : toks[i]; bad |= (t < 0 || t >= vocab); }
            }
            if (__any_sync(FULL, bad)) status = SAM_SEQ_BAD_TOKEN;
        }
        fresh_fail = status != 0;
    }
    if (status != 0) {
        if (host) step_join(false);
        if (warp == 0) {
            if (fresh_fail && lane == 0) cb[CB_STATUS] = (uint32_t)status;
            if (AHEAD && !VERIFY && A.tagged) write_failed_tagged(A, b, lane, status);
            else write_failed_slot(step_out(A, 0), L, b, lane, status);
            if (lane == 0) {
                if (VERIFY && A.v_counts_out) A.v_counts_out[b] = m;
                if (VERIFY && A.v_accepted_out) A.v_accepted_out[b] = confirmed;
            }
            __syncwarp();
            if (!VERIFY && A.done_flag && lane == 0) signal_done(A);
        }
        return;
    }

    uint4 ra, rb;             // this warp's copy of its match state's record
    kept_record(cw2, warp == 0 ? CB_REC1 : CB_REC2, ra, rb);

    int32_t d[MAX_DRAFT_REGS] = {-1, -1, -1, -1};
    int32_t my_l = 0, my_s = 0, my_dl = 0;
    int err = 0;

    if (warp == 0) {
        // ---------------- static automaton: Transfer per token ----------------
        if (A.has_static) {
            uint32_t s, sf; int32_t l;
            static_chain<true>(A, b, lane, cb, cw, tok_first, toks, m, built ? 0u : ntok0, ra, rb, s, sf, l, err, d, my_dl);
            my_l = l; my_s = (int32_t)s;
        }
    } else {
        // ---------------- dynamic automaton: Expand per token ----------------
        DynChain X;
        X.ra = ra; X.rb = rb;
        dyn_open(A.W, b, lane, cb, cw, cw2, X);
        dyn_feed<SEEN, CALL>(X, tok_first, toks, built ? 0 : m, sh_run);
        err = X.D.err; my_l = (int32_t)X.l2; my_s = (int32_t)X.s2;
        if (X.l2 > 0 && !err) {
            const int64_t e = (int64_t)X.ra.z;                  // min_endpos
            int64_t room = (int64_t)X.ntok - e;
            my_dl = (int)(room < L ? (room < 0 ? 0 : room) : L);
            gather_draft<0>(A.W.text + (size_t)b * A.W.text_stride, e, my_dl, L, lane, d);
            my_dl = cut_at_stop(d, my_dl, lane, A.W.stop_token);
        }
    }

    if (lane == 0) { sh_l[warp] = my_l; sh_s[warp] = my_s; sh_dl[warp] = my_dl; sh_err[warp] = err; }
    bool failed = true;
    if (AHEAD && !VERIFY && A.tagged) failed = step_join(err != 0); else step_sync();
    step_outputs<VERIFY, AHEAD && !VERIFY>(A, b, warp, lane, cb, sh_l, sh_s, sh_dl, sh_err, failed, d, m, confirmed);
    if (!VERIFY && A.done_flag) {
        if (AHEAD) step_join(false); else step_sync();
        if (threadIdx.x == 0) signal_done(A);
    }
}

// AHEAD: blocks of three warps an SM has to hold, 0 for blocks of two.  Registers come in quarters of an SM: 5 blocks (740
// slots) have 120 a thread and spill nothing, 6 (888) have 96, 8 (1184) have 80 and spill 192 bytes.  Prompt-copying
// slots, us a step with 5 / 6 / 8 blocks: 740 slots 14.6 / 15.0 / -, 880 slots - / 15.5 / 16.4, 1000 slots (in two
// waves: 20.5 / 18.5) 17.0, 1180 slots with two warps a slot 19.2, with three 17.4.
template <bool VERIFY, int AHEAD>
__global__ void __launch_bounds__(AHEAD ? 96 : 64, AHEAD ? AHEAD : 10) sam_step_kernel(const __grid_constant__ StepArgs A) {
    step_body<VERIFY, AHEAD != 0, false, AHEAD == 5 || AHEAD == 6, !(VERIFY && AHEAD == 8)>(A, A.new_tokens, A.counts);
}

// A host-array step whose rows and counts fit the launch's arguments: reading them from host memory, in the kernel's first
// round, costs 1.1 us for 4 slots and 3.2 us for 64 (many small requests on the bus), carrying them with the launch nothing.
// (With 32 KB of arguments, for 250 slots, it costs 3 us more than it saves.)
constexpr int SAM_INLINE_WORDS = 896;                    // within 4 KB of arguments
struct StepArgsInline { StepArgs A; int32_t in[SAM_INLINE_WORDS]; };                // rows, then counts
__global__ void __launch_bounds__(96, 5) sam_step_inline_kernel(const __grid_constant__ StepArgsInline I) {
    step_body<false, true, true, true, true>(I.A, I.in, I.in + (size_t)I.A.W.batch * I.A.stride);
}

// Larger ones: the rows and counts are brought over in whole lines by this kernel, launched ahead of the step's.
__global__ void __launch_bounds__(128) fetch_inputs_kernel(const int32_t* rows, const int32_t* counts, int32_t* to, size_t n_rows, size_t n_counts) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
    const size_t t = sam_grid_index(blockIdx.x, blockDim.x, threadIdx.x), all = sam_grid_size(gridDim.x, blockDim.x);
#pragma unroll
    for (int k = 0; k < 2; k++) {
        const int32_t* from = k ? counts : rows;
        int32_t* dst = k ? to + n_rows : to;
        const size_t n = k ? n_counts : n_rows;
        size_t done = 0;
        if (((reinterpret_cast<uintptr_t>(from) | reinterpret_cast<uintptr_t>(dst)) & 15) == 0) {
            for (size_t i = t; i < n / 4; i += all) reinterpret_cast<int4*>(dst)[i] = reinterpret_cast<const int4*>(from)[i];
            done = n & ~(size_t)3;
        }
        for (size_t i = done + t; i < n; i += all) dst[i] = from[i];
    }
}

// ------------------------------------------------------------------ prompts
// Launched ahead of the step kernel when the step's rows are long enough to hold prompts.  An empty slot that is given
// SAM_PREFILL_MIN tokens or more has its automaton built here (prefill_build.cuh); the slot's status tells the step kernel,
// which follows and does the rest of the slots.
//   STATIC: a block per slot.  Warp 0 finds the slot's static match meanwhile, and the slot is done here, outputs included: for
//   batches that leave the GPU room, where the step waits for the slowest slot.
//   Otherwise the step kernel does all but the build, and the build's blocks, without the static side's registers, are resident
//   five to an SM instead of three (4096 prompts of 1024 tokens).  There are as many blocks as are resident at once, and they share
//   out the slots with prompts: those that order_slots_kernel has listed, or, in batches that are not ordered, what they find in the counts.
//   (A block per slot costs an ordinary step of 1000 slots with rows of 8192 tokens 3 us.)
// From how many tokens (SAM_PREFILL_MIN): a step with one such prompt takes 18 us, reset included, one Expand after the other 0.3 to 0.5
// us a token.
__device__ __forceinline__ bool is_prompt(const StepArgs& A, int m) {
    return m >= SAM_PREFILL_MIN && m <= A.stride && m <= PB_MAX && m <= A.W.max_seq_len;
}
// The prompt's tokens to shared memory and to the slot's text (the text of an empty slot is nobody's); whether all of them are
// in the vocabulary (if not, the step kernel reports it).  Run by the whole block.
__device__ __forceinline__ bool load_prompt(const StepArgs& A, int b, int m, uint32_t* tok) {
    const int32_t* toks = A.new_tokens + (size_t)b * A.stride;
    int32_t* text = A.W.text + (size_t)b * A.W.text_stride;
    const int vocab = A.has_static ? A.S.vocab : A.W.vocab;
    bool bad = false;
    for (int j = threadIdx.x; j < m; j += blockDim.x) {
        const int t = toks[j];
        tok[j] = (uint32_t)t; text[j] = t;
        bad |= t < 0 || t >= vocab;
    }
    return !__syncthreads_or(bad);
}
// The list of prompts of a batch that is ordered: how many, how many have been taken beyond one for each block, the slots.
__host__ __device__ __forceinline__ int32_t* prompt_list(const SamBatchView& W) { return W.order + 3 * (size_t)W.batch + SAM_ORDER_WORDS; }

// Which prompts a block builds, one after the other, kept by its first thread in shared memory:
//   - those that order_slots_kernel has listed: the blockIdx.x-th, then whichever is next;
//   - in batches that are not ordered, those among every gridDim.x-th slot (with 740 blocks, at most three), or,
//   - where rows are so wide that only few blocks are resident, every gridDim.x-th of those that a look at all counts finds.
constexpr int PROMPT_SHARE = 128;                          // (more than 18944 slots, not ordered: the others' prompts go token by token)
struct PromptTake { int32_t share[PROMPT_SHARE]; int turn, found, slot; };
template <bool LOOK>
__device__ __forceinline__ void prompts_begin(const StepArgs& A, PromptTake& T) {
    if (threadIdx.x == 0) T.turn = T.found = 0;
    if (!LOOK || A.order) return;
    const int B = A.W.batch, lane = threadIdx.x & 31;
    bool any = false;
#pragma unroll 4
    for (int i = threadIdx.x; i < B; i += blockDim.x) any |= is_prompt(A, A.counts[i]);
    if (!__syncthreads_or(any) || threadIdx.x >= 32) return;
    int rank = 0, mine = 0;
#pragma unroll 4
    for (int base = 0; base < B; base += 32) {
        const bool is = base + lane < B && is_prompt(A, A.counts[base + lane]);
        const unsigned mask = __ballot_sync(FULL, is);
        const int r = rank + __popc(mask & ((1u << lane) - 1u)), k = r / (int)gridDim.x;
        if (is && r % (int)gridDim.x == (int)blockIdx.x && k < PROMPT_SHARE) { T.share[k] = base + lane; mine = k + 1; }
        rank += __popc(mask);
    }
    mine = __reduce_max_sync(FULL, mine);
    if (lane == 0) T.found = mine;
    __syncwarp();
}
// The next one's slot, -1 if there is none; by the first thread.
template <bool LOOK>
__device__ __forceinline__ int prompts_next(const StepArgs& A, PromptTake& T) {
    if (A.order) {
        int32_t* list = prompt_list(A.W);
        int at = blockIdx.x;
        if (T.turn++ > 0) at = (int)gridDim.x + atomicAdd(list + 1, 1);
        return at < list[0] ? list[2 + at] : -1;
    }
    if constexpr (LOOK) return T.turn < T.found ? T.share[T.turn++] : -1;
    else
        for (;;) {
            const int b = (int)blockIdx.x + T.turn++ * (int)gridDim.x;
            if (b >= A.W.batch) return -1;
            if (is_prompt(A, A.counts[b])) return b;
        }
}

template <bool STATIC, int THREADS, int BLOCKS>
__global__ void __launch_bounds__(THREADS, BLOCKS) sam_prefill_kernel(const __grid_constant__ StepArgs A) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
    extern __shared__ __align__(16) unsigned char pb_smem[];
    __shared__ PbShared sh;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (!STATIC) {
        constexpr bool LOOK = THREADS > 256;
        __shared__ PromptTake take;
        prompts_begin<LOOK>(A, take);
        for (;;) {
            if (threadIdx.x == 0) take.slot = prompts_next<LOOK>(A, take);
            __syncthreads();
            if (take.slot < 0) break;
            {
                const int b = take.slot, m = A.counts[b];
                uint32_t* cb = A.W.ctrl + (size_t)b * SAM_CTRL_WORDS;
                if (is_prompt(A, m) && cb[CB_STATUS] == 0 && cb[CB_NTOK] == 0 && load_prompt(A, b, m, pb_arrays(pb_smem, pb_size(m)).tok)) {
                    PbResult r;
                    pb_build(A.W, b, cb, m, pb_smem, sh, (int)threadIdx.x, (int)blockDim.x, r);
                    if (threadIdx.x == 0) A.W.ctrl[(size_t)take.slot * SAM_CTRL_WORDS + CB_STATUS] = r.err ? (uint32_t)r.err : SAM_STEP_BUILT;
                }
            }
            __syncthreads();
        }
        return;
    }
    __shared__ int32_t sh_l[2], sh_s[2], sh_dl[2], sh_err[2];
    const int b = blockIdx.x;
    uint32_t* cb = A.W.ctrl + (size_t)b * SAM_CTRL_WORDS;
    const int m = A.counts[b];
    const uint32_t cw = cb[lane];
    if (!is_prompt(A, m)) return;
    if (__shfl_sync(FULL, cw, CB_STATUS) != 0 || __shfl_sync(FULL, cw, CB_NTOK) != 0) return;
    const int32_t* toks = A.new_tokens + (size_t)b * A.stride;
    const int32_t* text = A.W.text + (size_t)b * A.W.text_stride;
    if (!load_prompt(A, b, m, pb_arrays(pb_smem, pb_size(m)).tok)) return;
    int32_t d[MAX_DRAFT_REGS] = {-1, -1, -1, -1};
    int32_t my_l = 0, my_s = 0, my_dl = 0;
    int err = 0;
    if (warp == 0) {
        if (A.has_static) {
            uint32_t s, sf; int32_t l;
            uint4 ra = make_uint4(0, 0, 0, 0), rb = ra;
            static_chain<true>(A, b, lane, cb, 0u, 0, toks, m, 0u, ra, rb, s, sf, l, err, d, my_dl);
            my_l = l; my_s = (int32_t)s;
        }
    } else {
        PbResult r;
        pb_build(A.W, b, cb, m, pb_smem, sh, (int)threadIdx.x - 32, (int)blockDim.x - 32, r);
        if (warp > 1) return;
        err = r.err; my_l = r.l2; my_s = r.s2;
        if (r.l2 > 0) {
            my_dl = min(m - r.e2, A.L);
            gather_draft<0>(text, r.e2, my_dl, A.L, lane, d);
            my_dl = cut_at_stop(d, my_dl, lane, A.W.stop_token);
        }
    }
    if (lane == 0) { sh_l[warp] = my_l; sh_s[warp] = my_s; sh_dl[warp] = my_dl; sh_err[warp] = err; }
    asm volatile("bar.sync 2, 64;" ::: "memory");
    step_outputs<false, false>(A, b, warp, lane, cb, sh_l, sh_s, sh_dl, sh_err, true, d, m, 0);
    if (threadIdx.x == 0 && sh_err[0] == 0 && sh_err[1] == 0) cb[CB_STATUS] = SAM_STEP_DONE;     // (a failed slot is reported again)
}

// ------------------------------------------------------------------ the split step (large batches)
// With more slots than the GPU holds blocks of the kernel above, throughput is set by how many chains are
// resident, and a block of two warps holds two warps' worth of registers for as long as its slower chain
// runs.  The split step gives the two sides of a slot to different blocks (of one warp) of one grid:
//   - the dynamic side keeps its warp per slot (DynChain);
//   - the static side of a slot with few tokens needs no cooperation between lanes (a state is one 32-byte
//     record, a hash bucket eight 16-byte entries), so one LANE carries it: a warp advances 32 slots, each
//     round of reads serving 32 chains (static_lanes);
//   - the static side of a slot with many tokens is what a step waits for, so it keeps a warp of its own
//     and everything that shortens the chain (static_chain: suffixes side by side, prefix states).
// The slots come sorted by token count (order_slots_kernel), which also says how many of them have "many".
// Neither side waits for the other.  Each writes its result to the slot's control block and then counts
// itself in CB_ARRIVE; the side that finds the other already counted (an odd count) reads both results,
// chooses the source, reads the draft and writes the slot's outputs.  Stores are ordered before the
// count by a device-scope fence, and what the other side wrote is read with loads that bypass the L1.
// A slot that fails its validation, or whose dynamic side runs into an error, is reported by the dynamic
// side alone before it counts itself; the static side validates on its own (it keeps the text length in
// CB_NTOK_S because CB_NTOK may change under it) and never commits a state for a step that is refused.

// How many sides of the slot have counted themselves, read with acquire semantics: if the count is odd the
// other side is done and everything it wrote may be read from here on (with loads that bypass the L1).
__device__ __forceinline__ uint32_t arrive_look(const uint32_t* cb) {
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(cb + CB_ARRIVE) : "memory");
    return v;
}

// Count this warp's side of slot `cb` as finished; true if the other side had finished before.
// A side that finds the other one done already (an acquiring look, one read) has no reader for what it wrote
// in this kernel: it counts itself without waiting for its stores.  Otherwise its stores are ordered before
// the count by a device-scope fence — the wait for them to be acknowledged is what that costs — and the
// count's old value decides.
__device__ __forceinline__ bool arrive_warp(uint32_t* cb, int lane) {
    const uint32_t seen = arrive_look(cb);                 // every lane looks for itself (one request)
    if (__all_sync(FULL, (seen & 1u) != 0)) {
        if (lane == 0) atomicAdd(cb + CB_ARRIVE, 1u);
        return true;
    }
    __threadfence();                                       // every lane's own stores ...
    __syncwarp();
    unsigned old = 0;
    if (lane == 0) { __threadfence(); old = atomicAdd(cb + CB_ARRIVE, 1u); }   // ... and, cumulatively, all of them before the count
    old = __shfl_sync(FULL, old, 0);
    if (old & 1u) __threadfence();                         // the other side's stores before this warp's reads of them
    return (old & 1u) != 0;
}

// Both sides of slot b are done.  Run by a whole warp.
__device__ __forceinline__ void split_epilogue(const StepArgs& A, int b, int lane) {
    uint32_t* cb = A.W.ctrl + (size_t)b * SAM_CTRL_WORDS;
    const uint32_t cw = __ldcg(cb + lane), cw2 = __ldcg(cb + 32 + lane);
    const uint32_t status = __shfl_sync(FULL, cw, CB_STATUS);
    if (status == SAM_STEP_BUILT) { if (lane == 0) cb[CB_STATUS] = 0; } // (both sides have seen it)
    else if (status != 0) return;                                       // reported by the dynamic side
    const int err_s = (int)__shfl_sync(FULL, cw, CB_ERR_S);
    const StepOut o = step_out(A, 0);
    if (err_s) {
        write_failed_slot(o, A.L, b, lane, err_s);
        if (lane == 0) cb[CB_STATUS] = (uint32_t)err_s;
        return;
    }
    write_slot(A, o, b, lane, (int)__shfl_sync(FULL, cw, CB_L1), (int)__shfl_sync(FULL, cw, CB_S1), (int64_t)__shfl_sync(FULL, cw2, CB_REC1 + 2 - 32),
                  (int)__shfl_sync(FULL, cw, CB_L2), (int)__shfl_sync(FULL, cw, CB_S2), (int64_t)__shfl_sync(FULL, cw2, CB_REC2 + 2 - 32),
                  (int64_t)__shfl_sync(FULL, cw, CB_NTOK));
}

// The same for the slots of the lanes of a static_lanes warp that found their dynamic side done (`second`).
// Each such lane knows its own side's result (l1, s1, e1, err_s) and reads the other's from its control block;
// the drafts are then read by the whole warp, row after row — lane k reads token k of every pending row, all
// rows' reads issued together — and written the same way.
__device__ __forceinline__ void split_epilogue_lanes(const StepArgs& A, bool second, int b, int lane,
                                                     int l1, int s1, int64_t e1, int err_s) {
    const unsigned pending0 = __ballot_sync(FULL, second);
    if (!pending0) return;
    uint32_t* cb = A.W.ctrl + (size_t)b * SAM_CTRL_WORDS;
    const int L = A.L;
    int l2 = 0, s2 = 0, src = SAM_SRC_NONE, dl = 0, status = 0;
    int64_t e = 0;
    const int32_t* text = A.S.corpus;
    bool mine = second;
    if (second) {
        const uint32_t st = __ldcg(cb + CB_STATUS);
        l2 = (int)__ldcg(cb + CB_L2); s2 = (int)__ldcg(cb + CB_S2);
        const int64_t ntok = (int64_t)__ldcg(cb + CB_NTOK), e2 = (int64_t)__ldcg(cb + CB_REC2 + 2);
        if (st == SAM_STEP_BUILT) {                                      // both sides are the other warp's
            l1 = (int)__ldcg(cb + CB_L1); s1 = (int)__ldcg(cb + CB_S1); e1 = (int64_t)__ldcg(cb + CB_REC1 + 2);
            err_s = (int)__ldcg(cb + CB_ERR_S);
            cb[CB_STATUS] = 0;
        }
        if (st != 0 && st != SAM_STEP_BUILT) mine = false;               // reported by the dynamic side
        else if (err_s) { status = err_s; l1 = l2 = 0; s1 = s2 = 0; cb[CB_STATUS] = (uint32_t)err_s; }
        else {
            const bool use_static = l1 > l2 + A.W.l_bias;               // Section 3.2
            const int lsel = use_static ? l1 : l2;
            const int need = A.W.min_match > 1 ? A.W.min_match : 1;
            src = lsel < need ? SAM_SRC_NONE : (use_static ? SAM_SRC_STATIC : SAM_SRC_DYNAMIC);
            if (!use_static) text = A.W.text + (size_t)b * A.W.text_stride;
            e = use_static ? e1 : e2;
            const int64_t room = (use_static ? A.S.n_tokens : ntok) - e;
            dl = src == SAM_SRC_NONE ? 0 : (int)(room < L ? (room < 0 ? 0 : room) : L);
        }
    }
    const unsigned pending = __ballot_sync(FULL, mine);
    const int32_t* src_ptr = text + e;
    int32_t* row = A.draft_tokens + (size_t)b * L;
    const int32_t stop = A.W.stop_token;
    int cut = dl;                                                        // this lane's row ends here
    for (int base = 0; base < L; base += 32) {
        int32_t v[32];
#pragma unroll
        for (int i = 0; i < 32; i++) {                                   // row i, token base + lane
            const int32_t* p_i = reinterpret_cast<const int32_t*>(__shfl_sync(FULL, (unsigned long long)src_ptr, i));
            const int dl_i = __shfl_sync(FULL, dl, i);
            v[i] = -1;
            if (base + lane < dl_i) v[i] = __ldcg(p_i + base + lane);
        }
#pragma unroll
        for (int i = 0; i < 32; i++) {
            int cut_i = __shfl_sync(FULL, cut, i);
            const unsigned hit = __ballot_sync(FULL, stop >= 0 && v[i] == stop && base + lane < cut_i);
            if (hit) cut_i = base + __ffs(hit) - 1;                      // a draft ends before the first stop token
            if (lane == i) cut = cut_i;
            int32_t* row_i = reinterpret_cast<int32_t*>(__shfl_sync(FULL, (unsigned long long)row, i));
            if (((pending >> i) & 1u) && base + lane < L) row_i[base + lane] = base + lane < cut_i ? v[i] : -1;
        }
    }
    if (mine) {
        A.draft_len[b] = cut; A.match_len[2 * b] = l1; A.match_len[2 * b + 1] = l2; A.source[b] = src;
        if (A.state) { A.state[2 * b] = s1; A.state[2 * b + 1] = s2; }
        A.status[b] = status;
    }
}

// The static side of 32 slots, one per lane: Transfer (Algorithm 1) for each of the slot's tokens.
// Every pass of the loop is one round of reads for all lanes that still have tokens: the record of the
// lane's state, the home bucket of (state, token) when the state has hashed transitions, the root-row
// entry of the token (used when the walk reaches the root in this pass) and the slot's next token.
__device__ __forceinline__ void static_lanes(const StepArgs& A, int w, int lane) {
    const SamStaticView& S = A.S;
    const int idx = A.W.batch - 1 - (w * 32 + lane);      // from the end of the sorted order: the fewest tokens first
    const int ob = A.order[idx > 0 ? idx : 0];            // (read together with the count below)
    const int first = min(*A.split_count, A.n_warp_blocks);   // the slots before this one have a warp of their own
    const bool live = idx >= first;
    if (!__any_sync(FULL, live)) return;
    const int b = live ? ob : 0;
    uint32_t* cb = A.W.ctrl + (size_t)b * SAM_CTRL_WORDS;
    const int32_t* toks = A.new_tokens + (size_t)b * A.stride;
    uint32_t status = 0, s = 0, sf = 0, ntok_s = 0;
    int32_t l = 0, t = 0;
    int m = 0;
    uint4 ra = make_uint4(0, 0, 0, 0), rb = ra;
    if (live) {
        status = cb[CB_STATUS]; s = cb[CB_S1]; l = (int32_t)cb[CB_L1]; sf = cb[CB_S1FLAG]; ntok_s = cb[CB_NTOK_S];
        ra = *reinterpret_cast<const uint4*>(cb + CB_REC1); rb = *reinterpret_cast<const uint4*>(cb + CB_REC1 + 4);
        m = A.counts[b];
        t = toks[0];
    }
    // the same checks, in the same order, as the dynamic side makes (bad count, capacity, then the tokens
    // one by one as they come up): a refused step leaves the static state as it was
    bool run = live && status == 0 && m >= 0 && m <= A.stride && (int64_t)ntok_s + m <= A.W.max_seq_len;
    bool active = run && m > 0;
    if (active && (t < 0 || t >= S.vocab)) { active = false; run = false; }
    bool have = s != 0;                                  // (ra, rb) is the record of s
    bool need_len = false;
    int j = 0, err = 0;
    int guard = l + 2 * m + 4;                           // at most l + m link moves in all (Appendix A.3)
    [[maybe_unused]] ChainCounts kc = {2, 0, 0, 0, 0};   // two rounds already: the slot's index, its control words
    while (__any_sync(FULL, active)) {
        if (active) SAM_COUNT(kc.rounds, 1);
        // One round of reads for every lane, none of them under a branch (lanes that took different branches
        // would otherwise wait for their reads one group after the other): a lane that does not need a line
        // reads one that every such lane shares (record 0, bucket 0, its own first token).
        const bool at_root = s == 0;
        const bool want_rec = active && !at_root && !have;
        const bool want_bucket = active && !at_root && sf != 0;
        uint32_t home = want_bucket ? sam_hash2(s, (uint32_t)t) & S.hash_mask : 0u;
        const uint32_t re = __ldg(S.root_row + (active ? t : 0));
        const int32_t tn = toks[(active && j + 1 < m) ? j + 1 : 0];
        const size_t ri = want_rec ? (size_t)s : 0;
        uint4 a = __ldg(S.rec + 2 * ri), bb = __ldg(S.rec + 2 * ri + 1);
        uint4 ent[SAM_HASH_BUCKET];
#pragma unroll
        for (int e = 0; e < SAM_HASH_BUCKET; e++) ent[e] = __ldg(S.hash + (size_t)home * SAM_HASH_BUCKET + e);
        if (have) { a = ra; bb = rb; }
        if (active) {
            have = false;
            bool advance = false;
            if (at_root) {                                // at the root the match length is 0
                if (re != SAM_NONE) { s = re & SAM_IDMASK; sf = re >> 31; l = 1; SAM_COUNT(kc.b, 1); } else l = 0;
                advance = true;
            } else {
                if (need_len) { l = (int32_t)a.x; need_len = false; }
                uint32_t tgt = SAM_NONE;
                if (a.w >= 1 && bb.x == (uint32_t)t) tgt = bb.y;
                else if (a.w >= 2 && bb.z == (uint32_t)t) tgt = bb.w;
                else if (a.w > 2) {
                    if (!sf) {                            // (every reference to a state with hashed transitions carries the flag)
                        home = sam_hash2(s, (uint32_t)t) & S.hash_mask;
#pragma unroll
                        for (int e = 0; e < SAM_HASH_BUCKET; e++) ent[e] = __ldg(S.hash + (size_t)home * SAM_HASH_BUCKET + e);
                    }
                    for (int probe = 1;; probe++) {
                        bool empty = false;
#pragma unroll
                        for (int e = 0; e < SAM_HASH_BUCKET; e++) {
                            if (ent[e].x == s && ent[e].y == (uint32_t)t) tgt = ent[e].z;
                            empty |= ent[e].x == SAM_NONE;
                        }
                        if (tgt != SAM_NONE || empty || probe >= S.hash_max_probe) break;
                        home = (home + 1) & S.hash_mask;
#pragma unroll
                        for (int e = 0; e < SAM_HASH_BUCKET; e++) ent[e] = __ldg(S.hash + (size_t)home * SAM_HASH_BUCKET + e);
                    }
                }
                if (tgt != SAM_NONE) { s = tgt & SAM_IDMASK; sf = tgt >> 31; l += 1; advance = true; SAM_COUNT(kc.b, 1); }
                else {                                    // s <- link(s), l <- len(link(s))
                    SAM_COUNT(kc.a, 1);
                    s = a.y & SAM_IDMASK; sf = a.y >> 31;
                    if (s == 0) {                         // the root either has the token or not: known already
                        if (re != SAM_NONE) { s = re & SAM_IDMASK; sf = re >> 31; l = 1; SAM_COUNT(kc.b, 1); } else l = 0;
                        advance = true;
                    } else need_len = true;
                    if (--guard < 0) { err = SAM_SEQ_WALK_LIMIT; active = false; }
                }
            }
            if (advance && active) {
                if (++j < m) {
                    t = tn;
                    if (t < 0 || t >= S.vocab) { active = false; run = false; }
                } else active = false;
            }
        }
    }
    int64_t e1 = (int64_t)ra.z;
    if (run && m > 0 && !err) {
        if (l > 0) {                                      // the state moved: read its record, keep a copy
            ra = __ldg(S.rec + 2 * (size_t)s); rb = __ldg(S.rec + 2 * (size_t)s + 1);
            *reinterpret_cast<uint4*>(cb + CB_REC1) = ra; *reinterpret_cast<uint4*>(cb + CB_REC1 + 4) = rb;
            e1 = (int64_t)ra.z;
        }
        cb[CB_S1] = s; cb[CB_L1] = (uint32_t)l; cb[CB_S1FLAG] = sf; cb[CB_NTOK_S] = ntok_s + (uint32_t)m;
    }
    if (live && err) cb[CB_ERR_S] = (uint32_t)err;
#ifdef SAM_COUNTERS
    if (g_sam_counters && run && b < g_sam_counter_slots) {
        unsigned long long* o = g_sam_counters + (size_t)b * SAM_N_COUNTERS;
        o[SAM_CNT_STATIC_ROUNDS] += kc.rounds + (l > 0 && m > 0 ? 1u : 0u);
        o[SAM_CNT_STATIC_LINK_MOVES] += kc.a; o[SAM_CNT_STATIC_NEXT_MOVES] += kc.b;
    }
#endif
    bool second = false;
    if (live) {
        if (arrive_look(cb) & 1u) { atomicAdd(cb + CB_ARRIVE, 1u); second = true; }
        else {
            __threadfence();
            second = (atomicAdd(cb + CB_ARRIVE, 1u) & 1u) != 0;
            if (second) __threadfence();
        }
    }
    split_epilogue_lanes(A, second, b, lane, l, (int32_t)s, e1, err);
}

// The dynamic side of one slot (one warp), including everything that reports a slot as failed.  Of a slot whose prompt
// has been built it does the static side as well (true: nothing else is left of its own side), for which the lanes of
// static_lanes would be slow; the static side's blocks see the slot's status and only count themselves.
__device__ __forceinline__ bool dynamic_slot(const StepArgs& A, int b, int lane, uint32_t (*sh_run)[12]) {
    uint32_t* cb = A.W.ctrl + (size_t)b * SAM_CTRL_WORDS;
    const int32_t* toks = A.new_tokens + (size_t)b * A.stride;
    const uint32_t cw = cb[lane];
    const uint32_t cw2 = cb[32 + lane];
    int32_t tok_first = 0;
    if (lane < A.stride) tok_first = toks[lane];
    const int m = A.counts[b];
    int status = (int)__shfl_sync(FULL, cw, CB_STATUS);
    if ((uint32_t)status == SAM_STEP_BUILT) return true;
    const uint32_t ntok0 = __shfl_sync(FULL, cw, CB_NTOK);
    bool fresh_fail = false;
    if (status == 0) {                                   // validate the whole step before any state changes
        if (m < 0 || m > A.stride) status = SAM_SEQ_BAD_COUNT;
        else if ((int64_t)ntok0 + m > A.W.max_seq_len) status = SAM_SEQ_CAPACITY;
        else {
            bool bad = false;
            for (int base = 0; base < m; base += 32) {
                const int i = base + lane;
                if (i < m) { const int tt = base == 0 ? tok_first : toks[i]; bad |= (tt < 0 || tt >= A.S.vocab); }
            }
            if (__any_sync(FULL, bad)) status = SAM_SEQ_BAD_TOKEN;
        }
        fresh_fail = status != 0;
    }
    int err = 0;
    if (status == 0) {
        DynChain X;
        kept_record(cw2, CB_REC2, X.ra, X.rb);
        dyn_open(A.W, b, lane, cb, cw, cw2, X);
        dyn_feed<false, true>(X, tok_first, toks, m, sh_run);
        err = X.D.err;
        if (err) { status = err; fresh_fail = true; }
    }
    if (status != 0) {
        if (fresh_fail && lane == 0) cb[CB_STATUS] = (uint32_t)status;
        write_failed_slot(step_out(A, 0), A.L, b, lane, status);
        arrive_warp(cb, lane);
        return false;
    }
    if (arrive_warp(cb, lane)) split_epilogue(A, b, lane);
    return false;
}

// The static side of one slot with a warp of its own.  built: of a slot whose prompt has been built and checked.
__device__ __forceinline__ void static_slot(const StepArgs& A, int b, int lane, bool built) {
    uint32_t* cb = A.W.ctrl + (size_t)b * SAM_CTRL_WORDS;
    const int32_t* toks = A.new_tokens + (size_t)b * A.stride;
    const uint32_t cw = cb[lane];
    const uint32_t cw2 = cb[32 + lane];
    int32_t tok_first = 0;
    if (lane < A.stride) tok_first = toks[lane];
    const int m = A.counts[b];
    const uint32_t ntok_s = __shfl_sync(FULL, cw, CB_NTOK_S);
    bool run = __shfl_sync(FULL, cw, CB_STATUS) == (built ? SAM_STEP_BUILT : 0u) && m >= 0 && m <= A.stride && (int64_t)ntok_s + m <= A.W.max_seq_len;
    if (run && !built) {                                 // the dynamic side reports a refused step; this side only keeps out
        bool bad = false;
        for (int base = 0; base < m; base += 32) {
            const int i = base + lane;
            if (i < m) { const int tt = base == 0 ? tok_first : toks[i]; bad |= (tt < 0 || tt >= A.S.vocab); }
        }
        run = !__any_sync(FULL, bad);
    }
    if (run) {
        uint4 ra, rb;
        kept_record(cw2, CB_REC1, ra, rb);
        uint32_t s, sf; int32_t l, dl = 0;
        int32_t d[MAX_DRAFT_REGS];
        int err = 0;
        static_chain<false>(A, b, lane, cb, cw, tok_first, toks, m, ntok_s, ra, rb, s, sf, l, err, d, dl);
        if (err && lane == 0) cb[CB_ERR_S] = (uint32_t)err;
    }
    if (arrive_warp(cb, lane)) split_epilogue(A, b, lane);
}

__global__ void __launch_bounds__(32) sam_step_split_kernel(const __grid_constant__ StepArgs A) {
    {   // while the previous kernel of the stream finishes: a dynamic-side block touches (prefetch, no data is
        // used) the lines it reads first
        const int pi = (int)blockIdx.x - A.n_warp_blocks - A.n_lane_blocks, pl = (int)threadIdx.x;
        if (pi >= 0 && pl < 4) {
            const char* p0 = reinterpret_cast<const char*>(A.W.ctrl + (size_t)pi * SAM_CTRL_WORDS);
            const char* p1 = reinterpret_cast<const char*>(A.new_tokens + (size_t)pi * A.stride);
            const char* p2 = reinterpret_cast<const char*>(A.counts + pi);
            const char* pp = pl == 0 ? p0 : pl == 1 ? p0 + 128 : pl == 2 ? p1 : p2;
            asm volatile("prefetch.global.L2 [%0];" ::"l"(pp));
        }
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
    __shared__ __align__(16) uint32_t sh_run[32][12];   // per-token staging of a repeat run (dynamic side)
    const int lane = threadIdx.x;
    const int i = (int)blockIdx.x;
    int b = -1;                                          // the slot whose static side this warp does
    bool built = false;
    if (i < A.n_warp_blocks) {
        // slots whose static side gets a warp: the first n_big of the sorted order (read together with order[])
        const int ob = A.order[i];
        if (i < min(*A.split_count, A.n_warp_blocks)) b = ob;
    } else if (i < A.n_warp_blocks + A.n_lane_blocks) {
        static_lanes(A, i - A.n_warp_blocks, lane);
    } else {
        // the dynamic side's time hardly depends on the token count: slots in their own order, one read less
        const int db = i - A.n_warp_blocks - A.n_lane_blocks;
        built = dynamic_slot(A, db, lane, sh_run);
        if (built) b = db;
    }
    if (b >= 0) static_slot(A, b, lane, built);
}

// ------------------------------------------------------------------ many steps in one launch
// sam_run_steps has every step's tokens at hand and slots never meet, so a slot goes through all its steps without waiting
// for the slowest slot of each, its two sides without waiting for each other (a warp each), and both through the tokens of as many
// steps as fit 32 lanes at a time: what a step costs beside its tokens (the round that looks them all up in the root table, the
// control words, runs of tokens cut short, the static match's rounds) is then paid once for some nine steps of 3.3 tokens.
// Both sides leave each step's result in the step's own outputs, and sam_run_finish_kernel, which no chain waits for, chooses the
// sources and reads the drafts: 32 rows a warp, eight rows' reads under way together.
// us a step, step after step on each side (static sides on a few lanes, or three warps a slot up to 296 slots) -> so: 200 slots
// 2.35 -> 1.3, 1000 slots 6.1 -> 2.2, 4096 slots 7.1 -> 4.0, 16384 slots 20.1 -> 11.8.
// Bound by the dynamic sides' rounds of reads and how many warps fit (16 an SM with 128 registers, nothing spilled; 20 with 96:
// 4 % slower at 4096 slots).
// What the two sides leave: match_len, state and status as they will be; the static side's first end position (or minus its
// error) in draft_len, the dynamic side's in source, the text length in the first word of the draft.
struct RunArgs {
    StepArgs A;
    int32_t n_steps, keep;       // keep: the outputs have room for every step
    int32_t finish;              // sam_run_block_kernel finishes the rows
};

struct StaticSide { uint32_t s, sf; int32_t l; uint4 ra, rb; };
__device__ __forceinline__ void static_open(uint32_t cw, uint32_t cw2, StaticSide& T) {
    T.s = __shfl_sync(FULL, cw, CB_S1); T.sf = __shfl_sync(FULL, cw, CB_S1FLAG); T.l = (int32_t)__shfl_sync(FULL, cw, CB_L1);
    kept_record(cw2, CB_REC1, T.ra, T.rb);
}
__device__ __forceinline__ void static_close(uint32_t* cb, int lane, uint32_t ntok, const StaticSide& T) {
    if (lane == 0) {
        cb[CB_S1] = T.s; cb[CB_L1] = (uint32_t)T.l; cb[CB_S1FLAG] = T.sf; cb[CB_NTOK_S] = ntok;
        if (T.l > 0) { reinterpret_cast<uint4*>(cb + CB_REC1)[0] = T.ra; reinterpret_cast<uint4*>(cb + CB_REC1)[1] = T.rb; }
    }
}

// A chunk: whole steps (of one with more than 32 tokens a part), planned a chunk ahead so that its tokens are there when it begins.
struct RunChunk {
    int32_t tok, step, own;      // this lane's token and the step it belongs to; if it ends the step: that step and those without tokens after it
    int32_t n_tok, n_steps, lead;         // tokens and steps in it; steps without tokens before the first that has some
    uint32_t starts;             // where steps begin
    int32_t refuse;              // why the step behind it is refused (0: it is not, or there is none)
    int32_t taken;               // tokens of the step behind it that it holds (of a step of more than 32: the first 32)
    int32_t tail;                // a token of that step behind those
};
__device__ __forceinline__ int32_t run_counts(const RunArgs& R, int b, int lane, int i) {
    return i + lane < R.n_steps ? R.A.counts[(size_t)(i + lane) * R.A.W.batch + b] : 0;
}
// WIDE: sam_run_block_kernel's, for few slots, whose steps may be wide: a step that fills a chunk by itself is planned without the scan, and
// one of more than 32 tokens is checked when it begins instead of here, where that waits for the tokens (64 slots, up to 47 tokens a
// step, 5 to 10 % faster).  For many slots it costs registers and gives nothing (4096 slots x 192 steps 1180 -> 1200 us).
// The chunk that begins with step i, of which `taken` tokens are done, whose slot had ntok tokens before it; m: lane k holds the
// count of step i + k.
template <bool WIDE>
__device__ __forceinline__ RunChunk run_plan(const RunArgs& R, int b, int lane, int i, int taken, uint32_t ntok, int m, int32_t* sh_map) {
    const StepArgs& A = R.A;
    RunChunk C;
    C.tok = C.tail = C.taken = C.refuse = 0;
    const int left = R.n_steps - i;
    const bool counted = m >= 0 && m <= A.stride;
    if (!counted) m = 0;
    const int m0 = __shfl_sync(FULL, m, 0), m1 = WIDE ? __shfl_sync(FULL, m, 1) : 0;
    if (WIDE && m0 >= 1 && m0 <= 32 && m0 + m1 > 32 && (int64_t)ntok + m0 <= A.W.max_seq_len) {          // a wide step, alone
        C.n_steps = 1; C.n_tok = m0; C.step = i; C.own = lane == m0 - 1 ? 1 : 0; C.lead = 0; C.starts = 1;
        if (lane < m0) C.tok = A.new_tokens[((size_t)i * A.W.batch + b) * A.stride + lane];
        return C;
    }
    const int upto = sum_upto(m, lane);                    // tokens up to this step's last
    const bool room = (int64_t)ntok + upto <= A.W.max_seq_len;
    const unsigned no = ~__ballot_sync(FULL, lane < left && counted && room && upto <= 32);
    const int n = no ? __ffs(no) - 1 : 32;
    C.n_steps = n;
    C.n_tok = n > 0 ? __shfl_sync(FULL, upto, n - 1) : 0;
    C.refuse = n < 32 ? __shfl_sync(FULL, lane >= left ? 0 : !counted ? SAM_SEQ_BAD_COUNT : !room ? SAM_SEQ_CAPACITY : 0, n & 31) : 0;
    if (n == 0 && left > 0 && C.refuse == 0) {             // a step of more than 32 tokens, checked as a whole
        const int32_t* row = A.new_tokens + ((size_t)i * A.W.batch + b) * A.stride;
        C.step = i; C.own = 0; C.lead = 0; C.starts = 1;
        if (!WIDE && taken == 0) {
            const int vocab = A.has_static ? A.S.vocab : A.W.vocab;
            const int32_t t0 = row[lane], t1 = lane + 32 < m0 ? row[lane + 32] : 0;
            if (__any_sync(FULL, t0 < 0 || t0 >= vocab || t1 < 0 || t1 >= vocab)) { C.refuse = SAM_SEQ_BAD_TOKEN; C.n_tok = 0; return C; }
        }
        C.n_tok = min(32, m0 - taken);
        if (lane < C.n_tok) C.tok = row[taken + lane];
        if (taken + C.n_tok == m0) { C.n_steps = 1; C.own = lane == C.n_tok - 1 ? 1 : 0; }
        else { C.taken = C.n_tok; if (WIDE && lane + 32 < m0) C.tail = row[lane + 32]; }
        return C;
    }
    const bool some = lane < n && m > 0;
    const unsigned filled = __ballot_sync(FULL, some);
    if (some) sh_map[upto - m] = lane;
    C.starts = __reduce_or_sync(FULL, some ? 1u << (upto - m) : 0u);
    C.lead = filled ? __ffs(filled) - 1 : n;
    __syncwarp();
    const unsigned mine = C.starts & (0xFFFFFFFFu >> (31 - lane));
    const int begin = mine ? 31 - __clz(mine) : 0, k = mine ? sh_map[begin] : 0;    // this lane's token: its step's first, and the step
    const int len = __shfl_sync(FULL, m, k);
    C.step = i + k; C.own = 0; C.tok = 0;
    if (lane < C.n_tok) {
        C.tok = A.new_tokens[((size_t)(i + k) * A.W.batch + b) * A.stride + (lane - begin)];
        const unsigned after = filled & ~((2u << k) - 1u);
        if (lane - begin == len - 1) C.own = (after ? __ffs(after) - 1 : n) - k;
    }
    __syncwarp();
    return C;
}

// Its tokens have come: where one is outside the vocabulary the chunk, which begins with step i, ends before that step.
template <bool WIDE>
__device__ __forceinline__ void run_cut(RunChunk& C, int lane, int i, int vocab) {
    const unsigned wrong = __ballot_sync(FULL, (lane < C.n_tok && (C.tok < 0 || C.tok >= vocab)) || (WIDE && (C.tail < 0 || C.tail >= vocab)));
    if (!wrong) return;
    C.taken = 0;
    const int t = __ffs(wrong) - 1;
    C.n_tok = 31 - __clz(C.starts & (0xFFFFFFFFu >> (31 - t)));
    C.n_steps = __shfl_sync(FULL, C.step, t) - i;
    C.refuse = SAM_SEQ_BAD_TOKEN;
    if (lane >= C.n_tok) C.own = 0;
}

// What a slot's results are written with, and (in shared memory) what holds at the end of the last step that is done.
struct RunEmit {
    static constexpr bool chunks = true, seen = false, call = false;
    const RunArgs& R;
    int b, lane;
    int32_t step, own;           // of the chunk (this lane's)
    unsigned ends;
    uint32_t* done;              // text length, states, state of the whole text, s2, l2; the step after it
    __device__ __forceinline__ void write(int first, int n, uint32_t s2, uint32_t l2, uint32_t e2, uint32_t ntok) const {
        const StepArgs& A = R.A;
        for (int i = first; i < first + n; i++) {
            if (!R.keep && i + 1 != R.n_steps) continue;
            const StepOut o = step_out(A, R.keep ? i : 0);
            o.match_len[2 * b + 1] = (int32_t)l2; o.source[b] = (int32_t)e2; o.status[b] = 0;
            o.draft[(size_t)b * A.L] = (int32_t)ntok;
            if (o.state) o.state[2 * b + 1] = (int32_t)s2;
        }
    }
    __device__ __forceinline__ void operator()(bool on, int from, uint32_t s2, uint32_t l2, uint32_t e2, uint32_t ntok, uint32_t last, uint32_t n_states) {
        const int st = __shfl_sync(FULL, step, from);
        int n = __shfl_sync(FULL, own, from);
        if (!on) n = 0;
        const unsigned ending = __ballot_sync(FULL, n > 0);
        if (!ending) return;
        if (n > 0) write(st, n, s2, l2, e2, ntok);
        if (lane == 31 - __clz(ending)) { done[0] = ntok; done[1] = n_states; done[2] = last; done[3] = s2; done[4] = l2; done[5] = (uint32_t)(st + n); }
        __syncwarp();
    }
};

template <bool WIDE>
__device__ __forceinline__ void run_dynamic(const RunArgs& R, int b, int lane, uint32_t (*sh_run)[12], int32_t* sh_map) {
    const StepArgs& A = R.A;
    __shared__ uint32_t done[6];
    uint32_t* cb = A.W.ctrl + (size_t)b * SAM_CTRL_WORDS;
    const uint32_t cw = cb[lane], cw2 = cb[32 + lane];
    int m = run_counts(R, b, lane, 0);
    int status = (int)__shfl_sync(FULL, cw, CB_STATUS);
    const bool fit = status == 0;
    DynChain X;
    kept_record(cw2, CB_REC2, X.ra, X.rb);
    dyn_open(A.W, b, lane, cb, cw, cw2, X);
    const uint32_t ntok0 = X.ntok;
    RunEmit emit{R, b, lane, 0, 0, 0u, done};
    const int vocab = A.has_static ? A.S.vocab : A.W.vocab;
    if (lane == 0) { done[0] = X.ntok; done[1] = X.D.n_states; done[2] = X.last; done[3] = X.s2; done[4] = X.l2; done[5] = 0; }
    __syncwarp();
    int i = 0;
    [[maybe_unused]] int n_fed = 0;                        // steps with tokens
    RunChunk C;
    if (fit) { C = run_plan<WIDE>(R, b, lane, 0, 0, X.ntok, m, sh_map); m = run_counts(R, b, lane, C.n_steps); }
    while (status == 0 && i < R.n_steps) {
        run_cut<WIDE>(C, lane, i, vocab);
        const int next = i + C.n_steps;
        RunChunk N = C;
        if (C.refuse == 0 && next < R.n_steps) {
            N = run_plan<WIDE>(R, b, lane, next, C.taken, X.ntok + (uint32_t)(C.n_tok - C.taken), m, sh_map);
            if (N.n_steps > 0) m = run_counts(R, b, lane, next + N.n_steps);
        }
        if (C.lead > 0) {
            if (lane == 0) { emit.write(i, C.lead, X.s2, X.l2, X.ra.z, X.ntok); done[5] = (uint32_t)(i + C.lead); }
            __syncwarp();
        }
        if (C.n_tok > 0) {
            emit.step = C.step; emit.own = C.own;
            emit.ends = __ballot_sync(FULL, C.own > 0);
            dyn_tokens(X, (uint32_t)C.tok, C.n_tok, sh_run, emit);
            SAM_COUNT(n_fed, __popc(emit.ends));
            status = X.D.err;
            if (status != 0) break;
        }
        i = next;
        status = C.refuse;
        C = N;
    }
    if (status != 0)
        for (int k = (int)done[5] + lane; k < R.n_steps; k += 32) if (R.keep || k + 1 == R.n_steps) step_out(A, R.keep ? k : 0).status[b] = status;
    if (X.D.err) {
        // The slot is left as the last step that was done left it, but for what the tokens after it have made.  The first of them
        // completes the newest state's record; where the pool had no state for it, that is done here, without a transition.
        const uint32_t newest = done[2];
        __syncwarp();
        uint32_t root_deg = X.D.root_deg;                  // without the transitions that tokens after that step have given it
        for (uint32_t at = done[0]; at < X.ntok; at++) {
            bool seen = false;
            for (uint32_t k = lane; k < at; k += 32) seen |= X.D.text[k] == X.D.text[at];
            if (!__any_sync(FULL, seen)) root_deg--;
        }
        uint4* rl = rec_ptr(X.D, newest);
        const uint4* rs = rec_ptr(X.D, done[3]);
        if (lane == 0) {
            if (newest != 0 && X.D.n_states == done[1]) { rl[0] = make_uint4(done[0], done[3], done[0], 0); rl[1] = make_uint4(0, 0, 0, 0); }
            if (done[4] > 0) { reinterpret_cast<uint4*>(cb + CB_REC2)[0] = rs[0]; reinterpret_cast<uint4*>(cb + CB_REC2)[1] = rs[1]; }
            cb[CB_NTOK] = done[0]; cb[CB_NSTATES] = done[1]; cb[CB_LAST] = newest; cb[CB_S2] = done[3]; cb[CB_L2] = done[4];
            cb[CB_BLK_CUR] = X.D.blk_cur; cb[CB_BLK_END] = X.D.blk_end; cb[CB_NRECSLABS] = X.D.n_rec_slabs; cb[CB_ROOTDEG] = root_deg;
        }
    } else if (X.ntok != ntok0) {
        SAM_COUNT(X.D.kc.rounds, 1);                       // (the first tokens)
        flush_counts(b, lane, false, X.D.kc, (int)(X.ntok - ntok0), n_fed);
        dyn_close(X);
        if (X.l2 > 0 && lane == 0) { reinterpret_cast<uint4*>(cb + CB_REC2)[0] = X.ra; reinterpret_cast<uint4*>(cb + CB_REC2)[1] = X.rb; }
    }
}

// The static side of a slot, a chunk of whole steps at a time: the longest suffix that occurs in the corpus, at the end of each step.
//   - All suffixes that begin in the chunk are walked side by side from the root, one lane each, a token a round.  Where
//     the text is new to the corpus they end after two or three tokens, and a chunk of nine steps is done in as many rounds.
//   - One lane is the chain instead, a match that follows suffix links (Algorithm 1): at first the match so far.  It lives until what
//     is left of it begins at token `base` or later, where the walks are.
//   - A match that goes on along a passage of the corpus takes its tokens in one round (static_follow).  A walk that has done
//     so is the chain from then on, and the walks that began before its end are part of it.
// What holds at the end of a step is what the earliest suffix that reaches it says: a walk leaves its result when the record that it
// goes on from is there; walks that began earlier come there later, except that the chain may be ahead: up to `base` and as far as
// it has come (`sure`) only it has a say.
struct RunResult { uint32_t s; int32_t l, e1; };

// A run of transitions of a match in state s (record a, b), taken in one round by the whole warp, as static_run takes it; n: tokens
// that may be taken, lane k's is tkl.  Returns how many were; out (lane k): the result after k + 1 of them.
__device__ __forceinline__ int static_follow(const SamStaticView& S, uint32_t s, const uint4& a, const uint4& b, int32_t l, uint32_t tkl, int n, int lane,
                                             uint32_t& ref, RunResult& out) {
    out.l = l + 1 + lane; out.s = 0; out.e1 = 0; ref = 0;
    const uint32_t g = inline_target(a, b, __shfl_sync(FULL, tkl, 0));
    bool ok = false;
    if (a.x == a.z) {                                      // the state of a corpus prefix: the tokens are the corpus' own, or not
        const int64_t e = (int64_t)a.z;
        int32_t cx = -2;
        if (lane < n && e + lane < S.n_tokens) { cx = __ldg(S.corpus + e + lane); ref = __ldg(S.pstate + e + lane); }
        ok = lane < n && (uint32_t)cx == tkl;
        out.s = ref & SAM_IDMASK; out.e1 = (int32_t)a.z + 1 + lane;
    } else if (g != SAM_NONE) {                            // ids a constant apart are guessed: lane k reads the (k + 1)-th of them
        const uint32_t d = (g & SAM_IDMASK) - s;
        if (d != 1 && d != 2) return 0;
        const uint32_t id = s + d * (uint32_t)(lane + 1);
        uint4 ka = make_uint4(0, 0, 0, 0), kb = ka;
        if (lane < n && (int64_t)id < S.n_states) static_record(S, id, ka, kb);
        const uint32_t nx = inline_target(ka, kb, __shfl_down_sync(FULL, tkl, 1));         // on the next token
        const uint32_t from = __shfl_up_sync(FULL, nx, 1);
        ref = lane == 0 ? g : from;                        // the transition that leads to this lane's state
        ok = lane < n && ref != SAM_NONE && (ref & SAM_IDMASK) == id;
        out.s = id; out.e1 = (int32_t)ka.z;
    }
    const unsigned no = ~__ballot_sync(FULL, ok);
    return no ? __ffs(no) - 1 : 32;
}

// One chunk: tk, n: its tokens; ends: the last tokens of its steps; T: the match, moved over the chunk (have: T's record is there; it
// is on return, if T.l > 0).  res[k]: the result after token k, for the k in ends.  Returns for how many tokens the results hold: all n,
// or, with err, as many as the match had taken when its links went on for too long.
__device__ __forceinline__ int static_chunk(const SamStaticView& S, uint32_t tk, int n, unsigned ends, int lane, StaticSide& T, RunResult* res, int& err, ChainCounts& kc) {
    uint32_t re = SAM_NONE;
    if (lane < n) re = __ldg(S.root_row + tk);
    res[lane] = RunResult{0u, 0, 0};
    __syncwarp();
    int base = 0, sure = 0;
    bool chain = T.s != 0 && lane == 0;
    bool alive = chain || (lane < n && re != SAM_NONE), have = false, need_len = false;
    bool came = true;                                      // by a transition, not by a link
    uint32_t cs = re & SAM_IDMASK, csf = re >> 31;
    int32_t cl = 1;
    int pos = lane + 1;                                    // tokens taken
    uint4 a = T.ra, b = T.rb;
    if (chain) { cs = T.s; csf = T.sf; cl = T.l; pos = 0; have = true; }
    int guard = T.l + 2 * n + 4;                           // link moves of the chain
    SAM_COUNT(kc.rounds, 1);
    for (;;) {
        const unsigned arrived = __ballot_sync(FULL, alive && pos == n);
        if (arrived && lane > __ffs(arrived) - 1) alive = false;          // an earlier suffix reaches the end
        bool go = alive && (pos < n || !have);
        if (!__any_sync(FULL, go)) break;
        SAM_COUNT(kc.rounds, 1);
        const uint32_t t = __shfl_sync(FULL, tk, pos & 31);
        const bool want_bucket = go && pos < n && csf;
        uint32_t home = 0;
        uint4 ent[SAM_HASH_BUCKET];
        if (want_bucket) {
            home = sam_hash2(cs, t) & S.hash_mask;
#pragma unroll
            for (int e = 0; e < SAM_HASH_BUCKET; e++) ent[e] = __ldg(S.hash + (size_t)home * SAM_HASH_BUCKET + e);
        }
        const bool fresh = go && !have;
        if (fresh) static_record(S, cs, a, b);
        if (go) {
            have = true;
            if (need_len) { cl = (int32_t)a.x; need_len = false; }
            if (chain && pos - cl >= max(base, 1)) alive = false;        // begins where the walks do
        }
        go = go && alive && pos < n;
        if (fresh && alive && came && pos > 0 && (ends >> (pos - 1) & 1u) && (chain || pos > sure)) res[pos - 1] = RunResult{cs, cl, (int32_t)a.z};
        uint32_t tgt = SAM_NONE;
        if (go) tgt = inline_target(a, b, t);
        // the earliest suffix there is, along the corpus as far as it goes
        const unsigned live = __ballot_sync(FULL, alive), apart = (tgt & SAM_IDMASK) - cs;
        const bool may = go && (chain || cl >= 3) && (a.x == a.z ? tgt != SAM_NONE || csf : tgt != SAM_NONE && (apart == 1 || apart == 2));
        if (live && __shfl_sync(FULL, may, __ffs(live) - 1)) {
            const int c = __ffs(live) - 1, p0 = __shfl_sync(FULL, pos, c);
            SAM_COUNT(kc.rounds, 1);
            uint32_t ref;
            RunResult out;
            const int r = static_follow(S, __shfl_sync(FULL, cs, c), shfl4(a, c), shfl4(b, c), __shfl_sync(FULL, cl, c),
                                        __shfl_sync(FULL, tk, (p0 + lane) & 31), n - p0, lane, ref, out);
            if (r > 0) {
                __syncwarp();                              // (walks that are ahead may just have left theirs where this one's count)
                if (lane < r && (ends >> (p0 + lane) & 1u)) res[p0 + lane] = out;
                base = sure = p0 + r;
                const uint32_t to = __shfl_sync(FULL, ref, r - 1);
                if (lane == c) { chain = came = true; cs = to & SAM_IDMASK; csf = to >> 31; cl += r; pos = base; have = go = false; }
                else if (lane < base) alive = go = false;
            }
        }
        if (go) {
            if (tgt == SAM_NONE && want_bucket) {          // (every reference to a state with hashed transitions carries the flag)
                for (int probe = 1;; probe++) {
                    bool empty = false;
#pragma unroll
                    for (int e = 0; e < SAM_HASH_BUCKET; e++) {
                        if (ent[e].x == cs && ent[e].y == t) tgt = ent[e].z;
                        empty |= ent[e].x == SAM_NONE;
                    }
                    if (tgt != SAM_NONE || empty || probe >= S.hash_max_probe) break;
                    home = (home + 1) & S.hash_mask;
#pragma unroll
                    for (int e = 0; e < SAM_HASH_BUCKET; e++) ent[e] = __ldg(S.hash + (size_t)home * SAM_HASH_BUCKET + e);
                }
            }
            have = came = false;
            if (tgt != SAM_NONE) { cs = tgt & SAM_IDMASK; csf = tgt >> 31; cl++; pos++; came = true; }
            else if (!chain) alive = false;
            else {                                         // s <- link(s), l <- len(link(s))
                cs = a.y & SAM_IDMASK; csf = a.y >> 31;
                if (cs != 0) need_len = true;
                else if (pos == 0 && re != SAM_NONE) { cs = re & SAM_IDMASK; csf = re >> 31; cl = 1; pos = 1; came = true; }
                else alive = false;
                if (--guard < 0) { err = SAM_SEQ_WALK_LIMIT; alive = false; }
            }
        }
        const unsigned ahead = __ballot_sync(FULL, alive && chain);
        if (ahead) { const int c = __ffs(ahead) - 1; sure = max(sure, __shfl_sync(FULL, need_len ? 0 : pos, c)); }
        __syncwarp();
    }
    const unsigned failed = __ballot_sync(FULL, err != 0);
    if (failed) { err = SAM_SEQ_WALK_LIMIT; n = __shfl_sync(FULL, pos, __ffs(failed) - 1); }
    const unsigned left = __ballot_sync(FULL, alive);
    if (!left) { T.s = 0; T.sf = 0; T.l = 0; return n; }
    const int first = __ffs(left) - 1;
    T.s = __shfl_sync(FULL, cs, first); T.sf = __shfl_sync(FULL, csf, first); T.l = __shfl_sync(FULL, cl, first);
    T.ra = shfl4(a, first); T.rb = shfl4(b, first);
    return n;
}

template <bool WIDE>
__device__ __forceinline__ void run_static(const RunArgs& R, int b, int lane, int32_t* sh_map, RunResult* res) {
    const StepArgs& A = R.A;
    uint32_t* cb = A.W.ctrl + (size_t)b * SAM_CTRL_WORDS;
    const uint32_t cw = cb[lane], cw2 = cb[32 + lane];
    int m = run_counts(R, b, lane, 0);
    if (__shfl_sync(FULL, cw, CB_STATUS) != 0) return;
    uint32_t ntok = __shfl_sync(FULL, cw, CB_NTOK_S);
    StaticSide T;
    static_open(cw, cw2, T);
    auto write = [&](int first, int n, uint32_t s, int32_t l, int32_t e1) {
        for (int i = first; i < first + n; i++) {
            if (!R.keep && i + 1 != R.n_steps) continue;
            const StepOut o = step_out(A, R.keep ? i : 0);
            o.match_len[2 * b] = l; o.draft_len[b] = l > 0 ? e1 : 0;
            if (o.state) o.state[2 * b] = (int32_t)s;
        }
    };
    int i = 0, err = 0;
    [[maybe_unused]] ChainCounts kc = {2, 0, 0, 0, 0};       // two rounds already: the control words and counts, the first tokens
    RunChunk C = run_plan<WIDE>(R, b, lane, 0, 0, ntok, m, sh_map);
    m = run_counts(R, b, lane, C.n_steps);
    while (i < R.n_steps) {
        run_cut<WIDE>(C, lane, i, A.S.vocab);
        const int next = i + C.n_steps;
        RunChunk N = C;
        if (C.refuse == 0 && next < R.n_steps) {
            N = run_plan<WIDE>(R, b, lane, next, C.taken, ntok + (uint32_t)(C.n_tok - C.taken), m, sh_map);
            if (N.n_steps > 0) m = run_counts(R, b, lane, next + N.n_steps);
        }
        if (C.lead > 0 && lane == 0) write(i, C.lead, T.s, T.l, (int32_t)T.ra.z);
        if (C.n_tok > 0) {
#ifdef SAM_COUNTERS
            {                                              // the moves Algorithm 1 itself makes over these tokens
                uint32_t ts = T.s, tsf = T.sf; int32_t tl = T.l;
                const uint32_t rounds = kc.rounds;
                for (int j = 0; j < C.n_tok && !err; j++) {
                    const uint32_t t = (uint32_t)__shfl_sync(FULL, C.tok, j);
                    static_transfer(A.S, ts, tsf, tl, t, __ldg(A.S.root_row + t), lane, err, false, T.ra, T.rb, kc);
                }
                kc.rounds = rounds; err = 0;
            }
#endif
            const int held = static_chunk(A.S, (uint32_t)C.tok, C.n_tok, __ballot_sync(FULL, C.own > 0), lane, T, res, err, kc);
            __syncwarp();
            const bool mine = C.own > 0 && lane < held;
            if (mine) write(C.step, C.own, res[lane].s, res[lane].l, res[lane].e1);
            __syncwarp();
            if (err) { i = max(i + C.lead, (int)__reduce_max_sync(FULL, mine ? (uint32_t)(C.step + C.own) : 0u)); break; }     // the step that fails
        }
        ntok += (uint32_t)C.n_tok;
        i = next;
        if (C.refuse) break;
        C = N;
    }
    if (err)
        for (int k = i + lane; k < R.n_steps; k += 32) if (R.keep || k + 1 == R.n_steps) step_out(A, R.keep ? k : 0).draft_len[b] = -err;
    static_close(cb, lane, ntok, T);
    flush_counts(b, lane, true, kc, 0, 0);
}

// Blocks of one warp: the dynamic side of each slot, then, with a static automaton, the static side of each slot.
__global__ void __launch_bounds__(32, 16) sam_run_split_kernel(const __grid_constant__ RunArgs R) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
    __shared__ __align__(16) uint32_t sh_run[32][12];
    __shared__ int32_t sh_map[32];
    const int lane = threadIdx.x, B = R.A.W.batch;
    if ((int)blockIdx.x < B) run_dynamic<false>(R, (int)blockIdx.x, lane, sh_run, sh_map);
    else run_static<false>(R, (int)blockIdx.x - B, lane, sh_map, reinterpret_cast<RunResult*>(&sh_run[0][0]));
    // (the slot's status is the finish kernel's to write: its other side may begin after this)
}

constexpr int FINISH_ROWS = 8;                             // rows whose reads a warp has under way together
// n <= 32 rows of the outputs from r0 on, `apart` from one another, by a warp.
__device__ __forceinline__ void run_finish(const RunArgs& R, int64_t r0, int64_t apart, int n, int lane) {
    const StepArgs& A = R.A;
    const int L = A.L;
    const int64_t rows = (int64_t)A.W.batch * (R.keep ? R.n_steps : 1);
    const int64_t r = r0 + lane * apart;
    const bool live = lane < n;
    int src = SAM_SRC_NONE, dl = 0;
    const int32_t* from = A.S.corpus;
    if (live) {                                            // this lane's row
        const int b = (int)(r % A.W.batch);
        int status = A.status[r], l1 = 0, s1 = 0, e1 = 0;
        int l2 = A.match_len[2 * r + 1];
        const int e2 = A.source[r], ntok = A.draft_tokens[r * L];
        if (A.has_static) {
            l1 = A.match_len[2 * r]; e1 = A.draft_len[r];
            if (status == 0 && e1 < 0) status = -e1;       // the static side's error, reported from here on
        }
        if (status != 0 && r + A.W.batch >= rows) A.W.ctrl[(size_t)b * SAM_CTRL_WORDS + CB_STATUS] = (uint32_t)status;
        if (status != 0) {
            l1 = l2 = 0;
            A.status[r] = status;
            if (A.state) { A.state[2 * r] = 0; A.state[2 * r + 1] = 0; }
            A.match_len[2 * r + 1] = 0;
        } else {
            const bool use_static = A.has_static && l1 > l2 + A.W.l_bias;           // Section 3.2
            const int lsel = use_static ? l1 : l2;
            const int need = A.W.min_match > 1 ? A.W.min_match : 1;
            src = lsel < need ? SAM_SRC_NONE : (use_static ? SAM_SRC_STATIC : SAM_SRC_DYNAMIC);
            if (src != SAM_SRC_NONE) {
                const int64_t e = use_static ? e1 : e2, room = (use_static ? A.S.n_tokens : (int64_t)ntok) - e;
                dl = (int)(room < L ? (room < 0 ? 0 : room) : L);
                from = (use_static ? A.S.corpus : A.W.text + (size_t)b * A.W.text_stride) + e;
            }
            if (!A.has_static && A.state) A.state[2 * r] = s1;
        }
        if (!A.has_static || status != 0) A.match_len[2 * r] = l1;
        A.source[r] = src;
    }
    __syncwarp();                                          // (every lane has read its row's first word)
    const int32_t stop = A.W.stop_token;
    int cut = dl;
    for (int base = 0; base < L; base += 32)
        for (int k0 = 0; k0 < n; k0 += FINISH_ROWS) {
            int32_t v[FINISH_ROWS];
#pragma unroll
            for (int k = 0; k < FINISH_ROWS; k++) {
                const int32_t* p = reinterpret_cast<const int32_t*>(__shfl_sync(FULL, (unsigned long long)from, (k0 + k) & 31));
                const int d = __shfl_sync(FULL, dl, (k0 + k) & 31);
                v[k] = -1;
                if (base + lane < d) v[k] = p[base + lane];
            }
#pragma unroll
            for (int k = 0; k < FINISH_ROWS; k++) {
                int c = __shfl_sync(FULL, cut, (k0 + k) & 31);
                if (stop >= 0) {                           // a draft ends before the first stop token
                    const unsigned hit = __ballot_sync(FULL, v[k] == stop && base + lane < c);
                    if (hit) c = base + __ffs(hit) - 1;
                    if (lane == k0 + k) cut = c;
                }
                if (k0 + k < n && base + lane < L) A.draft_tokens[(r0 + (k0 + k) * apart) * L + base + lane] = base + lane < c ? v[k] : -1;
            }
        }
    if (live) A.draft_len[r] = cut;
}
__global__ void __launch_bounds__(128) sam_run_finish_kernel(const __grid_constant__ RunArgs R) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
    const int64_t rows = (int64_t)R.A.W.batch * (R.keep ? R.n_steps : 1);
    const int64_t r0 = ((int64_t)blockIdx.x * 4 + (threadIdx.x >> 5)) * 32;
    if (r0 < rows) run_finish(R, r0, 1, (int)(rows - r0 < 32 ? rows - r0 : 32), threadIdx.x & 31);
}

// Up to two slots an SM: the two sides of a slot are the warps of a block, which have the SM's L1 to themselves (the other kernel asks
// for half of it as shared memory; 1 to 296 slots with 24 tokens a step 5 to 10 % faster), and few rows are finished by the block
// itself: calls of two steps 2.4 (one slot) to 4.4 us (200 slots) shorter, of four 1.0 to 4.7.
__global__ void __launch_bounds__(64, 8) sam_run_block_kernel(const __grid_constant__ RunArgs R) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
    __shared__ __align__(16) uint32_t sh_run[32][12];
    __shared__ RunResult res[32];
    __shared__ int32_t sh_map[2][32];
    const int lane = threadIdx.x & 31, side = threadIdx.x >> 5, b = blockIdx.x, B = R.A.W.batch;
    if (lane < R.n_steps)                                  // (which tokens are read first depends on the counts)
        asm volatile("prefetch.global.L1 [%0];" ::"l"(R.A.new_tokens + ((size_t)lane * B + b) * R.A.stride));
    if (side == 0) run_dynamic<true>(R, b, lane, sh_run, sh_map[0]);
    else if (R.A.has_static) run_static<true>(R, b, lane, sh_map[1], res);
    if (!R.finish) return;
    __syncthreads();
    const int n = R.keep ? R.n_steps : 1;
    for (int i = 32 * side; i < n; i += 64) run_finish(R, (int64_t)i * B + b, B, min(32, n - i), lane);
}

// A batch larger than the GPU holds at once runs in waves, and a step is as long as its last block: a
// slot with many tokens that starts in the last wave ends late.  This kernel sorts the slots by their
// token count, largest first (a counting sort in shared memory), so that block i of the step kernel takes
// slot order[i] and the long slots start in the first wave.  It reads only the step's counts, so it runs
// while the step before is still going; it ends with griddepcontrol.wait, so that its own completion —
// all the next step kernel waits for — implies that of the step before.
// The counts may still be changing while this kernel reads them (when the kernel before it on the stream
// is the one that writes them), so each count is read exactly once: the key taken from it is kept in
// `keys` and used for both passes.  order[] is therefore a permutation of the slots whatever was read;
// a count read too early only costs the intended launch order, never a result (the step kernel reads the
// counts itself, after its own dependency wait).
constexpr int SAM_ORDER_KEYS = 64;
constexpr int SAM_ORDER_THREADS = 1024;
// (SPLIT: the instance launched ahead of the split step; it is given that kernel's split between L1 and shared
// memory, because kernels that want different ones do not share an SM.)
template <bool SPLIT>
__global__ void __launch_bounds__(SAM_ORDER_THREADS) order_slots_kernel(const int32_t* counts, int32_t B, int32_t* order,
                                                                        int32_t* keys, int32_t big_m, int32_t* n_big, int32_t* list) {
    asm volatile("griddepcontrol.launch_dependents;");
    __shared__ int hist[SAM_ORDER_KEYS];
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    for (int k = threadIdx.x; k < SAM_ORDER_KEYS; k += blockDim.x) hist[k] = 0;
    __syncthreads();
    // Four slots per thread and round, so that four reads are under way at a time; the lanes of a warp that
    // hold the same key count themselves with one addition (the counts cluster on a few small values).
    constexpr int U = 4;
    for (int base = 0; base < B; base += U * SAM_ORDER_THREADS) {
        int key[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int i = base + u * SAM_ORDER_THREADS + (int)threadIdx.x;
            key[u] = -1;
            if (i < B) {
                const int m = *reinterpret_cast<const volatile int32_t*>(counts + i);
                key[u] = m < 0 ? 0 : (m >= SAM_ORDER_KEYS ? SAM_ORDER_KEYS - 1 : m);
            }
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int i = base + u * SAM_ORDER_THREADS + (int)threadIdx.x;
            if (i < B) keys[i] = key[u];                     // read back by this same thread below
            const unsigned peers = __match_any_sync(FULL, key[u]);
            if (key[u] >= 0 && (peers & lt) == 0) atomicAdd(&hist[key[u]], __popc(peers));
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {                                  // hist[k] <- first position of key k, keys descending
        int at = 0;
        for (int k = SAM_ORDER_KEYS - 1; k >= 0; k--) {
            const int n = hist[k]; hist[k] = at; at += n;
            if (k == big_m) *n_big = at;                     // slots with at least big_m tokens: the first `at` of order[]
        }
    }
    __syncthreads();
    for (int base = 0; base < B; base += U * SAM_ORDER_THREADS) {
        int key[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int i = base + u * SAM_ORDER_THREADS + (int)threadIdx.x;
            key[u] = i < B ? keys[i] : -1;
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int i = base + u * SAM_ORDER_THREADS + (int)threadIdx.x;
            const unsigned peers = __match_any_sync(FULL, key[u]);
            const int leader = __ffs(peers) - 1;
            int pos = 0;
            if (key[u] >= 0 && lane == leader) pos = atomicAdd(&hist[key[u]], __popc(peers));
            pos = __shfl_sync(FULL, pos, leader) + __popc(peers & lt);
            if (key[u] >= 0 && pos < B) order[pos] = i;      // always true: the keys are those counted above
        }
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (!list) return;
    // Now the counts are final: the slots with prompts, for sam_prefill_kernel, which looks at nothing else.
    __shared__ int n;
    if (threadIdx.x == 0) n = 0;
    __syncthreads();
    for (int base = 0; base < B; base += U * SAM_ORDER_THREADS) {
        int m[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int i = base + u * SAM_ORDER_THREADS + (int)threadIdx.x;
            m[u] = i < B ? __ldcg(counts + i) : 0;
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
            const unsigned mask = __ballot_sync(FULL, m[u] >= SAM_PREFILL_MIN);
            if (!mask) continue;
            int at = 0;
            if (lane == 0) at = atomicAdd(&n, __popc(mask));
            at = __shfl_sync(FULL, at, 0);
            if (m[u] >= SAM_PREFILL_MIN) list[2 + at + __popc(mask & lt)] = base + u * SAM_ORDER_THREADS + (int)threadIdx.x;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) { list[0] = n; list[1] = 0; }
}

// From how many tokens on a slot's static side gets a warp of its own in the split step.  A lane's chain costs
// about 1.3 us per read round against 0.5 us per token for a warp's; up to a few thousand slots a step is as
// long as its slowest slot, beyond that the number of resident warps counts for more.
constexpr int split_big_m(int batch) { return batch >= 8192 ? 8 : 5; }

// The split kernel's blocks are single warps with 1.5 KB of shared memory each: the default split between L1
// and shared memory would hold only a dozen of them per SM.  Once per device.
int split_kernel_setup(int device);

constexpr int SAM_SPLIT_MIN_BATCH = 8192;                    // the split step is used from this many slots on
constexpr int SAM_SMS = 148;
constexpr int SAM_AHEAD_MAX_BATCH = SAM_SMS * 8;             // three warps a slot, all slots resident at once

}  // namespace

namespace {
constexpr int SAM_MAX_DEVICES = 64;
SamOncePerDevice<SAM_MAX_DEVICES> g_split_setup, g_prefill_setup[4];

int split_kernel_setup(int device) {
    if (device < 0 || device >= SAM_MAX_DEVICES) return SAM_ERR_ARG;
    cudaError_t e = (cudaError_t)g_split_setup(device, []() -> int {
        cudaError_t e = cudaFuncSetAttribute(sam_step_split_kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 50);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(order_slots_kernel<true>, cudaFuncAttributePreferredSharedMemoryCarveout, 50);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(sam_run_split_kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 50);
        return (int)e;
    });
    if (e != cudaSuccess) { sam_set_cuda_error(e); return SAM_ERR_CUDA; }
    return SAM_OK;
}
// The build for rows of up to `stride` tokens.  With the static side: a token a thread, as far as threads go, 1024 where a build
// has the SM to itself (fewer slots than SMs, or rows of which the shared memory holds one), otherwise 512, so that the registers
// are enough for two.  (With two tokens a thread 1 x 300 took 25.9 us for 21.0 now, 16 x 1000 41 for 37, and of 256 x 1024 only one
// build fitted an SM: 95 for 78.)  Without: four tokens a thread, registers for as many blocks as the shared memory has room for.
int launch_prefill(const StepArgs& A, int batch, int device, cudaLaunchConfig_t* cfg) {
    using Kernel = void (*)(const StepArgs);
    const Kernel kernels[4] = {sam_prefill_kernel<true, 1024, 1>, sam_prefill_kernel<false, 256, 5>, sam_prefill_kernel<false, 512, 3>,
                               sam_prefill_kernel<false, 1024, 1>};
    int n2 = 64;
    while (n2 < A.stride && n2 < PB_MAX) n2 <<= 1;
    const int most = batch <= SAM_SMS || n2 > 2048 ? 1024 : 512, rows = A.stride < most ? (A.stride + 31) & ~31 : most;
    int k = 0, threads = rows + 32 < most ? rows + 32 : most, blocks = batch;
    if (batch > 2 * SAM_SMS) {
        k = n2 <= 1024 ? 1 : n2 <= 2048 ? 2 : 3;
        threads = n2 / 4 < 128 ? 128 : n2 / 4 > 1024 ? 1024 : n2 / 4;
        const int resident = SAM_SMS * (k == 1 ? (threads < 256 ? 10 : 5) : k == 2 ? 3 : 1);
        if (blocks > resident) blocks = resident;
    }
    if (device < 0 || device >= SAM_MAX_DEVICES) return SAM_ERR_ARG;
    cudaError_t e = (cudaError_t)g_prefill_setup[k](device, [&]() -> int {
        return (int)cudaFuncSetAttribute(kernels[k], cudaFuncAttributeMaxDynamicSharedMemorySize, PB_MAX * PB_BYTES_PER_TOKEN);
    });
    cfg->gridDim = dim3((unsigned)blocks); cfg->blockDim = dim3((unsigned)threads); cfg->dynamicSmemBytes = (size_t)n2 * PB_BYTES_PER_TOKEN;
    if (e == cudaSuccess) e = cudaLaunchKernelEx(cfg, kernels[k], A);
    if (e != cudaSuccess) { sam_set_cuda_error(e); return SAM_ERR_CUDA; }
    return SAM_OK;
}
}  // namespace

int sam_step_launch_count(const sam_batch* b) { return b->view.batch >= SAM_ORDER_MIN_BATCH ? 2 : 1; }

int sam_launch_step(const sam_batch* b, const SamStepIo& io, cudaStream_t stream) {
    SamDeviceGuard guard(b->device);
    if (!guard.ok) return SAM_ERR_CUDA;
    StepArgs A;
    const bool verify = io.v_draft != nullptr;
    A.v_draft = io.v_draft; A.v_draft_len = io.v_draft_len; A.v_max_new = io.v_max_new;
    A.v_counts_out = io.v_counts_out; A.v_accepted_out = io.v_accepted_out;
    A.done_count = b->view.pool_hdr + 4; A.done_flag = io.done_flag; A.done_seq = io.done_seq;
    A.tagged = reinterpret_cast<uint2*>(io.tagged); A.tag = (uint32_t)io.done_seq;
    A.has_static = b->st != nullptr;
    if (b->st) A.S = b->st->view;
    else { A.S = SamStaticView(); A.S.vocab = b->view.vocab; }
    A.W = b->view;
    const int32_t stride = io.stride;
    const int32_t* counts = io.counts;
    A.new_tokens = io.new_tokens; A.stride = stride; A.counts = counts; A.L = io.L;
    A.draft_tokens = io.draft_tokens; A.draft_len = io.draft_len; A.match_len = io.match_len;
    A.source = io.source; A.state = io.state; A.status = io.status;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    A.order = nullptr; A.split_count = nullptr;
    A.n_warp_blocks = A.n_lane_blocks = 0;
    bool prompts = false;
#ifndef SAM_COUNTERS                                       // (the counters count Expand's own operations, one Expand at a time)
    prompts = io.prompts;
#endif
    // (A host-array step is synchronous: nothing runs before it that the ordering kernel could overlap with, so it
    // would cost more than the order saves; its slots are in their own order.)
    if (!verify && !io.from_host && b->view.batch >= SAM_ORDER_MIN_BATCH) {
        int32_t* order = b->view.order + (size_t)(b->order_phase & 1) * b->view.batch;
        cudaLaunchConfig_t oc;
        memset(&oc, 0, sizeof(oc));
        oc.gridDim = dim3(1); oc.blockDim = dim3(SAM_ORDER_THREADS); oc.stream = stream; oc.attrs = attr; oc.numAttrs = 1;
        int32_t* n_big = b->view.order + 3 * (size_t)b->view.batch + 8 * (b->order_phase & 1);
        int32_t* list = prompts ? prompt_list(b->view) : nullptr;
        const bool split = A.has_static && b->view.batch >= SAM_SPLIT_MIN_BATCH;
        if (split) { int rc = split_kernel_setup(b->device); if (rc) return rc; }
        cudaError_t oe = split
            ? cudaLaunchKernelEx(&oc, order_slots_kernel<true>, counts, (int32_t)b->view.batch, order,
                                 b->view.order + 2 * (size_t)b->view.batch, split_big_m(b->view.batch), n_big, list)
            : cudaLaunchKernelEx(&oc, order_slots_kernel<false>, counts, (int32_t)b->view.batch, order,
                                 b->view.order + 2 * (size_t)b->view.batch, split_big_m(b->view.batch), n_big, list);
        A.split_count = n_big;
        b->order_phase ^= 1;
        if (oe != cudaSuccess) { sam_set_cuda_error(oe); return SAM_ERR_CUDA; }
        A.order = order;
    }
    if (prompts) {
        cudaLaunchConfig_t pc;
        memset(&pc, 0, sizeof(pc));
        pc.stream = stream; pc.attrs = attr; pc.numAttrs = 1;
        int rc = launch_prefill(A, b->view.batch, b->device, &pc);
        if (rc) return rc;
    }
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)b->view.batch); cfg.blockDim = dim3(64); cfg.dynamicSmemBytes = 0; cfg.stream = stream;
    cfg.attrs = attr; cfg.numAttrs = 1;
    cudaError_t e;
    if (A.order && A.has_static && b->view.batch >= SAM_SPLIT_MIN_BATCH) {   // the two sides of a slot in different blocks
        int rc = split_kernel_setup(b->device);
        if (rc) return rc;
        A.n_warp_blocks = (b->view.batch + 3) / 4;
        A.n_lane_blocks = (b->view.batch + 31) / 32;
        cfg.gridDim = dim3((unsigned)(b->view.batch + A.n_warp_blocks + A.n_lane_blocks)); cfg.blockDim = dim3(32);
        e = cudaLaunchKernelEx(&cfg, sam_step_split_kernel, A);
    } else {
        const bool ahead = b->view.batch <= SAM_AHEAD_MAX_BATCH;
        if (ahead) cfg.blockDim = dim3(96);
        if (io.inline_rows && ahead && !prompts) {
            const size_t rows = (size_t)b->view.batch * stride;
            StepArgsInline I;
            I.A = A;
            memcpy(I.in, io.inline_rows, rows * 4);
            memcpy(I.in + rows, io.inline_counts, (size_t)b->view.batch * 4);
            e = cudaLaunchKernelEx(&cfg, sam_step_inline_kernel, I);
        } else {
            using Kernel = void (*)(const StepArgs);
            const Kernel kernels[2][4] = {{sam_step_kernel<false, 0>, sam_step_kernel<false, 5>, sam_step_kernel<false, 6>, sam_step_kernel<false, 8>},
                                          {sam_step_kernel<true, 0>, sam_step_kernel<true, 5>, sam_step_kernel<true, 6>, sam_step_kernel<true, 8>}};
            const int B = b->view.batch, k = !ahead ? 0 : B <= SAM_SMS * 5 ? 1 : B <= SAM_SMS * 6 ? 2 : 3;
            e = cudaLaunchKernelEx(&cfg, kernels[verify][k], A);
        }
    }
    if (e != cudaSuccess) { sam_set_cuda_error(e); return SAM_ERR_CUDA; }
    return SAM_OK;
}

// Whether a host-array step's rows and counts, without prompts, can come with the launch.
bool sam_step_is_inline(const sam_batch* b, int32_t stride) {
    return b->view.batch <= SAM_AHEAD_MAX_BATCH && (size_t)b->view.batch * ((size_t)stride + 1) <= (size_t)SAM_INLINE_WORDS;
}

int sam_launch_fetch(const sam_batch* b, const int32_t* rows, const int32_t* counts, int32_t* to, int32_t stride, cudaStream_t stream) {
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    const size_t n = (size_t)b->view.batch * stride, blocks = (n + 511) / 512;      // a 16-byte read a thread
    cfg.gridDim = dim3((unsigned)(blocks < 592 ? blocks : 592)); cfg.blockDim = dim3(128); cfg.stream = stream; cfg.attrs = attr; cfg.numAttrs = 1;
    SAM_CUDA(cudaLaunchKernelEx(&cfg, fetch_inputs_kernel, rows, counts, to, n, (size_t)b->view.batch));
    return SAM_OK;
}

// Up to SAM_RUN_FINISH_MAX times 32 draft tokens of a slot are read by its own block: 64 rows of 16 tokens as fast as by a launch of their
// own (1, 64, 296 slots: 75 / 74, 242 / 245, 171 / 171 us a call with its prompts), 192 rows 160 / 153, 192 of 128 tokens 185 / 148.
constexpr int SAM_RUN_BLOCK_MAX_BATCH = 2 * SAM_SMS, SAM_RUN_FINISH_MAX = 64;
int sam_launch_run(const sam_batch* b, const int32_t* new_tokens, int32_t stride, const int32_t* counts, int32_t n_steps, int32_t L, int32_t keep,
                   int32_t* draft_tokens, int32_t* draft_len, int32_t* match_len, int32_t* source, int32_t* state, int32_t* status,
                   cudaStream_t stream) {
    SamDeviceGuard guard(b->device);
    if (!guard.ok) return SAM_ERR_CUDA;
    RunArgs R;
    memset(&R, 0, sizeof(R));
    StepArgs& A = R.A;
    A.has_static = b->st != nullptr;
    if (b->st) A.S = b->st->view; else A.S.vocab = b->view.vocab;
    A.W = b->view;
    A.new_tokens = new_tokens; A.stride = stride; A.counts = counts; A.L = L;
    A.draft_tokens = draft_tokens; A.draft_len = draft_len; A.match_len = match_len; A.source = source; A.state = state; A.status = status;
    R.n_steps = n_steps; R.keep = keep;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.stream = stream; cfg.attrs = attr; cfg.numAttrs = 1;
    cudaError_t e;
    int rc = split_kernel_setup(b->device);
    if (rc) return rc;
    const int64_t rows = (int64_t)b->view.batch * (keep ? n_steps : 1);
    if (b->view.batch <= SAM_RUN_BLOCK_MAX_BATCH) {
        R.finish = (keep ? n_steps : 1) * ((L + 31) / 32) <= SAM_RUN_FINISH_MAX;
        cfg.gridDim = dim3((unsigned)b->view.batch); cfg.blockDim = dim3(64);
        e = cudaLaunchKernelEx(&cfg, sam_run_block_kernel, R);
    } else {
        cfg.gridDim = dim3((unsigned)b->view.batch * (A.has_static ? 2u : 1u)); cfg.blockDim = dim3(32);
        e = cudaLaunchKernelEx(&cfg, sam_run_split_kernel, R);
    }
    if (R.finish && e == cudaSuccess) return SAM_OK;
    cfg.gridDim = dim3((unsigned)((rows + 127) / 128)); cfg.blockDim = dim3(128);
    if (e == cudaSuccess) e = cudaLaunchKernelEx(&cfg, sam_run_finish_kernel, R);
    if (e != cudaSuccess) { sam_set_cuda_error(e); return SAM_ERR_CUDA; }
    return SAM_OK;
}

// The launches of sam_step for each step where rows may hold prompts (the whole-text build has a kernel of its own), else one or two
// for all.
bool sam_runs_in_one_launch(int32_t stride, int32_t n_steps) { return n_steps > 1 && stride < SAM_PREFILL_MIN; }

extern "C" int sam_counters_available(void) {
#ifdef SAM_COUNTERS
    return 1;
#else
    return 0;
#endif
}

extern "C" int sam_counters_attach(uint64_t* counters_dev, int32_t slots) {
#ifdef SAM_COUNTERS
    if (slots < 0 || (!counters_dev && slots > 0)) return SAM_ERR_ARG;
    unsigned long long* p = reinterpret_cast<unsigned long long*>(counters_dev);
    int n = counters_dev ? slots : 0;
    SAM_CUDA(cudaMemcpyToSymbol(g_sam_counters, &p, sizeof(p)));
    SAM_CUDA(cudaMemcpyToSymbol(g_sam_counter_slots, &n, sizeof(n)));
    return SAM_OK;
#else
    (void)counters_dev; (void)slots;
    return SAM_ERR_UNSUPPORTED;
#endif
}
