// Build the suffix automaton of a whole text at once, by all threads of a block.
//
// Expand (Algorithm 3), run token after token, is a chain of dependent reads: 0.54 us per token for one warp
// (64 slots x 1024 tokens: 550 us, and 5.8 ms for one slot of 8191).  What it ends with is a function of the text alone,
// and all of it can be read off the sorted order of the text's prefixes:
//   - prefixes are sorted by their tokens from the last to the first; A[j] is the end position of the j-th, h[j]
//     the length of the suffix it shares with its predecessor.  Sorting is by prefix doubling: positions are grouped by their
//     token, and each round orders the groups of equal prefixes by four times as many tokens;
//   - the strings that are suffixes of the same set of prefixes form an interval of the sorted order.  An interval is
//     named by the first boundary inside it where h is smallest; its length is that h, its first end position the
//     smallest A in it, its parent the interval at the larger h just outside;
//   - l[p], the longest suffix of prefix p that ends anywhere earlier, is the nearest interval around p that a smaller
//     end position belongs to.  Expand of token p makes state c_p (the whole prefix) and, exactly if no state has that
//     suffix as its longest string yet, one clone: the first p to claim an interval makes it.  State ids follow by
//     counting clones;
//   - suffix links are the parents;
//   - the transitions into a state u (longest string w, link of length k) are those on w's last token from the states
//     along the suffix links of w without that token, down to length k.
// Nothing here depends on a guess: each of these statements is the definition of the automaton of the text.
//
// What bounds it: for short texts the chain of some 40 barriers (1 x 300 tokens 17 us), for long ones one SM's issue slots (8191 tokens, 206 us
// under ncu in the version that was captured, 173 us now: 64 % of them, 3900 instructions of a warp for 32 tokens, a third of the time in
// the sort; everything but the outputs stays
// in shared memory, 28 bytes per token), for many the same (4096 x 1024 tokens: 9.5 tokens a ns), and a step waits for its slowest
// build: 64 x 1024 tokens 34 to 51 us by text, mean 25.
#pragma once
#include "common.h"

namespace {

constexpr int PB_MAX = 8192;               // longest text: 28 bytes per token of shared memory
constexpr int PB_BYTES_PER_TOKEN = 28;
constexpr int PB_LEVELS = 5;               // rank arrays kept for comparing two prefixes
constexpr int PB_COUNTED = 128;            // members of a group up to which they are ordered by counting
constexpr int PB_BLOCK_SLABS = 80;         // slabs the edge blocks of one text can take (at most 64, and a remainder)
constexpr uint32_t PB_ROOT = 0xFFFFu;      // handle of the root; a state is (p << 1 | clone)

struct PbShared {                          // what the threads of one build exchange besides the arrays
    int16_t chunk[PB_MAX / 32];
    uint32_t slab[SAM_MAX_REC_SLABS + PB_BLOCK_SLABS];       // of the records, then of the edge blocks
    uint32_t cls_n[16], cls_base[16];
    int groups[2];                         // counted in rounds in turn: one is cleared while the other is in use
    int rows, placed, clones, root_deg, err, n_rec_slabs;
};

struct PbArrays {
    uint64_t* key; uint16_t* lev; uint16_t* end; uint16_t* A; uint16_t* B; uint32_t* tok;      // while sorting
    uint32_t* tree; uint16_t* rank; uint16_t* canon; uint16_t* enode; uint16_t* parent;
    uint32_t* first; uint16_t* wnode; uint16_t* idc; uint16_t* link; uint16_t* llen; uint32_t* deg; uint16_t* clen;
    int N2;                                // size of the sorted order, a power of two
};

// `tree`: leaves in its upper half.  When they are no longer needed, `link` takes the place of its inner nodes, `deg` that of its
// leaves, `llen` (the lengths of the states that `link` names) that of the tokens, and `clen` (of each position the length of
// `wnode`'s interval, for a position that clones the clone's) that of `rank`.
__device__ __forceinline__ PbArrays pb_arrays(unsigned char* sm, int N2) {
    PbArrays a;
    const size_t n = (size_t)N2;
    a.N2 = N2;
    a.key = (uint64_t*)sm; a.lev = (uint16_t*)(sm + 8 * n); a.end = (uint16_t*)(sm + 18 * n); a.A = (uint16_t*)(sm + 20 * n); a.B = (uint16_t*)(sm + 22 * n);
    a.tok = (uint32_t*)(sm + 24 * n);
    a.tree = (uint32_t*)sm; a.link = (uint16_t*)sm; a.rank = (uint16_t*)(sm + 8 * n); a.canon = (uint16_t*)(sm + 10 * n);
    a.enode = (uint16_t*)(sm + 12 * n); a.parent = (uint16_t*)(sm + 14 * n); a.first = (uint32_t*)(sm + 16 * n);
    a.wnode = (uint16_t*)(sm + 20 * n); a.idc = (uint16_t*)(sm + 22 * n); a.deg = (uint32_t*)(sm + 4 * n); a.llen = (uint16_t*)(sm + 24 * n);
    a.clen = a.rank;
    return a;
}
__device__ __forceinline__ int pb_size(int n) { return n <= 64 ? 64 : 1 << (32 - __clz(n - 1)); }

__device__ __forceinline__ void pb_sync(int nt) { asm volatile("bar.sync 1, %0;" ::"r"(nt) : "memory"); }
__device__ __forceinline__ bool pb_sync_or(int nt, bool x) {
    uint32_t r;
    asm volatile("{ .reg .pred p, q; setp.ne.u32 p, %2, 0; bar.red.or.pred q, 1, %1, p; selp.u32 %0, 1, 0, q; }" : "=r"(r) : "r"(nt), "r"((uint32_t)x) : "memory");
    return r != 0;
}

// The tree over the sorted order: leaf j is h[j] << 16 | A[j], an inner node the two minima of its leaves.
// The levels above 32 nodes of a level of `width` (a power of two), by a warp whose lane k has node at + k in v.
__device__ __forceinline__ void pb_grow(const PbArrays& a, uint32_t v, int width, int at, int lane) {
#pragma unroll
    for (int l = 1; l <= 5; l++) {
        v = __vminu2(v, __shfl_xor_sync(0xFFFFFFFFu, v, 1 << (l - 1)));
        if ((lane & ((1 << l) - 1)) == 0 && lane < width && (width >> l) > 0) a.tree[(width >> l) + ((at + lane) >> l)] = v;
    }
}
// First boundary to the left of sorted position j (inclusive) with h < l; acc: smallest A met, that position's included.
__device__ __forceinline__ int pb_left(const PbArrays& a, int j, uint32_t l, uint32_t& acc) {
    int i = a.N2 + j;
    for (;;) {
        const uint32_t v = a.tree[i];
        if ((v >> 16) < l) {
            while (i < a.N2) {
                const uint32_t r = a.tree[2 * i + 1];
                if ((r >> 16) < l) i = 2 * i + 1;
                else { acc = min(acc, r & 0xFFFFu); i = 2 * i; }
            }
            acc = min(acc, a.tree[i] & 0xFFFFu);
            return i - a.N2;
        }
        acc = min(acc, v & 0xFFFFu);
        while (!(i & 1)) i >>= 1;
        if (i == 1) return 0;                              // (h[0] = 0 ends every search before this)
        i -= 1;
    }
}
// First boundary to the right of sorted position j (exclusive) with h < l, N2 if there is none; acc: smallest A in between.
__device__ __forceinline__ int pb_right(const PbArrays& a, int j, uint32_t l, uint32_t& acc) {
    int i = a.N2 + j + 1;
    if (j + 1 >= a.N2) return a.N2;
    for (;;) {
        const uint32_t v = a.tree[i];
        if ((v >> 16) < l) {
            while (i < a.N2) {
                const uint32_t x = a.tree[2 * i];
                if ((x >> 16) < l) i = 2 * i;
                else { acc = min(acc, x & 0xFFFFu); i = 2 * i + 1; }
            }
            return i - a.N2;
        }
        acc = min(acc, v & 0xFFFFu);
        while (i & 1) i >>= 1;
        if (i == 0) return a.N2;
        i += 1;
    }
}
__device__ __forceinline__ uint32_t pb_h(const PbArrays& a, int j) { return j < a.N2 ? a.tree[a.N2 + j] >> 16 : 0u; }

// The interval that prefix p is alone in the middle of: the larger h on its two sides (0: none but the root).
__device__ __forceinline__ uint32_t pb_leaf(const PbArrays& a, uint32_t p) {
    const int j = a.rank[p];
    const uint32_t hl = pb_h(a, j), hr = pb_h(a, j + 1);
    return max(hl, hr) == 0 ? 0u : a.canon[hl >= hr ? j : j + 1];
}
__device__ __forceinline__ bool pb_clones(const PbArrays& a, uint32_t p) { return (a.wnode[p] & 0x8000u) != 0; }
__device__ __forceinline__ uint32_t pb_len(const PbArrays& a, uint32_t hd) {
    return hd == PB_ROOT ? 0u : (hd & 1) ? a.clen[hd >> 1] : (hd >> 1) + 1;
}
__device__ __forceinline__ uint32_t pb_end(const PbArrays& a, uint32_t hd) { return (hd & 1) ? a.enode[a.wnode[hd >> 1] & 0x7FFF] : hd >> 1; }
__device__ __forceinline__ uint32_t pb_id(const PbArrays& a, uint32_t hd) { return hd == PB_ROOT ? 0u : a.idc[hd >> 1] + (hd & 1); }
__device__ __forceinline__ uint32_t pb_state(const PbArrays& a, uint32_t node) { return node == 0 ? PB_ROOT : a.first[node]; }

// The states that the transitions into state u = (p, clone) come from, but for the root: a stretch of the suffix links' chain from
// the prefix before (for a clone, from what that prefix had in common with an earlier one), from the first state shorter than u
// down to length low (0: the root has one as well).  A link of the chain is two reads that go out together, 40 cycles; reading
// a state's length from its own arrays made it 130.
struct PbChain { uint32_t v, lv, low; };
__device__ __forceinline__ bool pb_more(const PbChain& c) { return c.v != PB_ROOT && c.lv >= c.low; }
__device__ __forceinline__ void pb_next(const PbArrays& a, PbChain& c) {
    const uint32_t n = a.link[c.v], l = a.llen[c.v];
    c.v = l < c.lv ? n : PB_ROOT; c.lv = l;                // (lengths fall along suffix links)
}
// Walk a warp's 32 chains: f(v, on, owner, all) by whole warps, v a state of lane `owner`'s chain where `on`; all: the lanes are
// at the same chain, otherwise each at its own.
// Most chains have one to three states, and each lane goes along its own.  But a build waits for its longest chain, and where
// tokens repeat (a run of one token, or of a few in turn) a chain has a state for each repeat, their handles the same distance
// apart: when few lanes are left, all look at the next 32 states of one chain, as far as that distance holds; where it
// does not, they take what comes one after the other, 16 states at a time.
// (Four states of each lane's chain side by side: 4096 prompts of 1024 tokens 10 % slower, the builds being bound by their instructions.)
constexpr int PB_FEW = 4;                  // lanes left
template <class F>
__device__ __forceinline__ void pb_walk(const PbArrays& a, PbChain& c, int n, int lane, F f) {
    unsigned rest = __ballot_sync(0xFFFFFFFFu, pb_more(c));
    for (int turn = 0; rest; turn++) {
        if (turn >= 4 && __popc(rest) <= PB_FEW) break;
        const bool on = pb_more(c);
        const uint32_t v = c.v;
        if (on) pb_next(a, c);
        f(v, on, lane, false);
        rest = __ballot_sync(0xFFFFFFFFu, pb_more(c));
    }
    for (; rest; rest &= rest - 1) {
        const int owner = __ffs(rest) - 1;
        PbChain x;                                         // the same in all lanes
        x.v = __shfl_sync(0xFFFFFFFFu, c.v, owner); x.lv = __shfl_sync(0xFFFFFFFFu, c.lv, owner); x.low = __shfl_sync(0xFFFFFFFFu, c.low, owner);
        while (pb_more(x)) {
            uint32_t v = x.v + (uint32_t)lane * (a.link[x.v] - x.v);
            const bool in = v < 2u * (uint32_t)n;
            const uint32_t nv = in ? a.link[v] : PB_ROOT, nl = in ? a.llen[v] : 0u;
            uint32_t pv = __shfl_up_sync(0xFFFFFFFFu, nv, 1), pl = __shfl_up_sync(0xFFFFFFFFu, nl, 1);
            if (lane == 0) { pv = x.v; pl = x.lv; }
            const unsigned ok = __ballot_sync(0xFFFFFFFFu, in && pv == v && pl >= x.low && nl < pl);
            const int r = ~ok ? __ffs(~ok) - 1 : 32;
            if (r >= 4) {
                f(v, lane < r, owner, true);
                x.v = __shfl_sync(0xFFFFFFFFu, nv, r - 1); x.lv = __shfl_sync(0xFFFFFFFFu, nl, r - 1);
                continue;
            }
            v = PB_ROOT;
            for (int i = 0; i < 16 && pb_more(x); i++) {
                if (lane == i) v = x.v;
                pb_next(a, x);
            }
            f(v, v != PB_ROOT, owner, true);
        }
        if (lane == owner) c = x;
    }
}
// Where the chain of u's transitions begins.  u: live lanes only.  start: kept beside `first` for a second walk.
__device__ __forceinline__ PbChain pb_chain(const PbArrays& a, bool live, uint32_t u, uint32_t len, int n, int lane) {
    const uint32_t p = u >> 1;
    PbChain c;
    c.v = PB_ROOT; c.lv = 0; c.low = len;
    if (live && len > 1) {
        if (!(u & 1)) { c.v = (p - 1) << 1; c.lv = p; }
        else {
            const uint32_t x = a.wnode[p - 1] & 0x7FFFu;
            c.v = x == 0 ? PB_ROOT : reinterpret_cast<const uint16_t*>(a.first)[2 * x];
            c.lv = a.clen[p - 1];
        }
    }
    pb_walk(a, c, n, lane, [](uint32_t, bool, int, bool) {});        // the states that are not shorter
    if (live) {
        c.low = a.llen[u];
        if (u & 1) reinterpret_cast<uint16_t*>(a.first)[2 * p + 1] = (uint16_t)c.v;
    }
    return c;
}
__device__ __forceinline__ PbChain pb_chain_again(const PbArrays& a, bool live, uint32_t u, uint32_t len) {
    PbChain c;
    c.v = PB_ROOT; c.lv = c.low = 0;
    if (live && len > 1) {
        if (!(u & 1)) { c.v = ((u >> 1) - 1) << 1; c.lv = u >> 1; }
        else { c.v = reinterpret_cast<const uint16_t*>(a.first)[2 * (u >> 1) + 1]; c.lv = pb_len(a, c.v); }
        c.low = a.llen[u];
    }
    return c;
}

// Slabs for a whole prompt, by one warp: all of them or none.  Subtracting and giving back what is too few would do, were it not
// that in between other blocks find the pool short and fail prompts that it has room for.  So the pool's two header words are
// used as one: free slabs below, slabs in the pool above, and added to those the takers that have subtracted and not yet
// settled.  A taker that finds too few gives back and looks again: it fails only where there are too few and nobody is
// unsettled.  (Compare-and-swap alone does as well and lets takers through one round trip after the other: 4096 prompts of 100
// tokens took 2850 us instead of 165.)
constexpr int PB_TAKE_TRIES = 1 << 16;     // looks before giving up; who is unsettled needs one more atomic for it, which waits for nobody
__device__ __forceinline__ int pb_free_slabs(unsigned long long word) { return (int)(uint32_t)word; }
__device__ __forceinline__ uint32_t pb_unsettled(unsigned long long word, int32_t pool_slabs) {
    return (uint32_t)((word - (unsigned long long)(long long)pb_free_slabs(word)) >> 32) - (uint32_t)pool_slabs;
}
// seen: the header words as lane 0 has read them, of any age.
__device__ __forceinline__ uint32_t pb_take_slabs(const SamBatchView& W, unsigned long long seen, int want, int b, uint32_t* out, int lane, int& err) {
    int old = -1;
    if (lane == 0) {
        unsigned long long* hdr = reinterpret_cast<unsigned long long*>(W.pool_hdr);
        const unsigned long long mark = 1ull << 32, n = (unsigned long long)want;
        if (pb_free_slabs(seen) >= want) {
            const unsigned long long was = atomicAdd(hdr, mark - n);
            if (pb_free_slabs(was) >= want) { old = pb_free_slabs(was); atomicAdd(hdr, 0ull - mark); }
            else atomicAdd(hdr, n - mark);
        }
        for (int tries = 0; old < 0 && tries < PB_TAKE_TRIES; tries++) {
            const unsigned long long now = *reinterpret_cast<volatile unsigned long long*>(hdr);
            if (pb_free_slabs(now) >= want) { if (atomicCAS(hdr, now, now - n) == now) old = pb_free_slabs(now); }
            else if (pb_unsettled(now, W.pool_slabs) == 0) break;
        }
    }
    old = __shfl_sync(0xFFFFFFFFu, old, 0);
    if (old < 0) { err = SAM_SEQ_CAPACITY; return 0; }
    for (int i = lane; i < want; i += 32) {
        const int idx = W.free_stack[old - 1 - i];
        W.slab_owner[idx] = b;
        out[i] = (uint32_t)idx;
    }
    return (uint32_t)want;
}

struct PbResult { int32_t s2, l2, e2; int err; };          // e2: first end position of the match state

// The first round: positions grouped by their token, the groups in any order of the tokens (the order in which warps ask for room).
// A: the positions, group after group; rank 0 of `lev`: where a position's group begins.  Returns the number of groups.
// (Counting in a table costs 2 us for 1024 tokens, with a scan of the table for the groups' places 3; sorting keys of three
// tokens cost 10.)
__device__ int pb_group(const PbArrays& a, PbShared& sh, unsigned char* smem, int n, int tid, int nt) {
    const int lane = tid & 31, N2 = a.N2, size = 2 * N2;
    uint32_t* key = reinterpret_cast<uint32_t*>(a.key);                              // [size]: tokens
    uint32_t* cnt = reinterpret_cast<uint32_t*>(smem + 10 * (size_t)N2);             // [size]: positions, then where they begin
    uint16_t* at = reinterpret_cast<uint16_t*>(smem + 18 * (size_t)N2);              // [N2]: a position's table entry
    for (int i = tid; i < size >> 2; i += nt) {
        reinterpret_cast<uint4*>(key)[i] = make_uint4(SAM_NONE, SAM_NONE, SAM_NONE, SAM_NONE);
        reinterpret_cast<uint4*>(cnt)[i] = make_uint4(0, 0, 0, 0);
    }
    if (tid == 0) sh.groups[0] = sh.groups[1] = sh.rows = sh.placed = 0;
    pb_sync(nt);
    for (int p = tid; p < n; p += nt) {
        const uint32_t t = a.tok[p];
        uint32_t h = sam_hash1(t) & (size - 1);
        for (int probe = 0; probe < size; probe++) {       // (at most half full)
            uint32_t old = key[h];
            if (old == SAM_NONE) old = atomicCAS(&key[h], SAM_NONE, t);
            if (old == SAM_NONE || old == t) break;
            h = (h + 1) & (size - 1);
        }
        at[p] = (uint16_t)h;
        a.B[p] = (uint16_t)atomicAdd(&cnt[h], 1u);
    }
    pb_sync(nt);
    for (int p = tid; p - lane < n; p += nt) {             // (whole warps) the first position of each group sees to its place
        const bool first = p < n && a.B[p] == 0;
        const int c = first ? (int)cnt[at[p]] : 0, s = sum_upto(c, lane);
        const unsigned firsts = __ballot_sync(0xFFFFFFFFu, first);
        int base = 0;
        if (lane == 31 && firsts) { base = atomicAdd(&sh.placed, s); atomicAdd(&sh.groups[0], __popc(firsts)); }
        base = __shfl_sync(0xFFFFFFFFu, base, 31);
        if (first) cnt[at[p]] = (uint32_t)(base + s - c);
    }
    pb_sync(nt);
    for (int p = tid; p < n; p += nt) {
        const uint32_t begin = cnt[at[p]];
        a.A[begin + a.B[p]] = (uint16_t)p;
        a.lev[p] = (uint16_t)begin;
    }
    pb_sync(nt);
    return sh.groups[0];
}

// What is common to the rounds of the sort.  A round orders the members of each group of equal prefixes (of `span` tokens) by the
// tokens before those: A -> B, rank -> next.  PB_ALONE in A marks the groups of one, which most positions are in after a round or
// two: they stay where they are.  This is the look at position j: whether it is alone; end: where each group ends.
constexpr uint32_t PB_ALONE = 0x8000u;
__device__ __forceinline__ bool pb_alone(uint16_t* A, const uint16_t* rank, uint16_t* end, int j, int n, uint32_t& p, uint32_t& g, bool& ends) {
    p = A[j];
    ends = false;
    if (p & PB_ALONE) { p &= ~PB_ALONE; return true; }
    g = rank[p];
    ends = j + 1 == n || rank[A[j + 1] & ~PB_ALONE] != g;
    if (ends) {
        end[g] = (uint16_t)(j + 1);
        if (g == (uint32_t)j) { A[j] = (uint16_t)(p | PB_ALONE); return true; }
    }
    return false;
}
// The round's end.  Its counter is read after this barrier and cleared in the next round but one's place, after that round's first
// barrier, when all threads have read it.
__device__ __forceinline__ int pb_groups(PbShared& sh, int turn, int mine, int tid, int nt) {
    mine = __reduce_add_sync(0xFFFFFFFFu, mine);
    if ((tid & 31) == 0) atomicAdd(&sh.groups[turn & 1], mine);
    pb_sync(nt);
    return sh.groups[turn & 1];
}

// A round by counting, for each member, how many of its group come first, by 3 x span tokens.  Returns the number of groups, or 0,
// with nothing ordered, if there are groups so large that two rounds of pb_double take less: 7 us for 1024 tokens, 35 for
// 8191, against 2.2 and 9 for counting small groups.  (Counting groups of 870 of 8191 took 50 us, a bitonic sort of all 47;
// 1000 texts of 1500 tokens, groups of up to 200: 274 us with the sort, 246 with pb_double.)
__device__ int pb_refine(const PbArrays& a, PbShared& sh, uint16_t* A, uint16_t* B, const uint16_t* rank, uint16_t* next, int span, int turn, int n, int tid, int nt) {
    uint32_t alone = 0;                                    // of this thread's positions
    int mine = 0;
    bool large = false;
    for (int j = tid, nth = 0; j < n; j += nt, nth++) {
        uint32_t p, g;
        bool ends;
        if (pb_alone(A, rank, a.end, j, n, p, g, ends)) { alone |= 1u << nth; B[j] = (uint16_t)(p | PB_ALONE); next[p] = (uint16_t)j; mine++; continue; }
        large |= ends && j + 1 - (int)g > PB_COUNTED;
        uint64_t k = 0;
#pragma unroll
        for (int q = 1; q < 4; q++) { const int at = (int)p - q * span; k = k << 16 | (at >= 0 ? (uint32_t)rank[at] + 1u : 0u); }
        a.key[j] = k << 16 | p;
    }
    if (pb_sync_or(nt, large)) return 0;
    if (tid == 0) sh.groups[~turn & 1] = 0;
    for (int j = tid, nth = 0; j < n; j += nt, nth++) {
        if (alone >> nth & 1u) continue;
        const uint64_t k = a.key[j], same = k & ~0xFFFFull;
        const uint32_t p = (uint32_t)k & 0xFFFFu, g = rank[p], e = a.end[g];
        int less = 0, before = 0;                          // the group's that come before this one, and before all equal to it
#pragma unroll 4
        for (uint32_t i = g; i < e; i++) {
            const uint64_t x = a.key[i];
            less += x < k; before += x < same;
        }
        B[g + less] = (uint16_t)p;
        next[p] = (uint16_t)(g + before);
        mine += less == before;
    }
    return pb_groups(sh, turn, mine, tid, nt);
}

// A round that looks at `span` tokens more and does not care how large the groups are.  In the order there is, the prefixes that
// end `span` tokens earlier already lie as the members of each group shall: the i-th of them, q, says where q + span comes in its
// group, after as many as have come by.  In a group of up to PB_FEW_MEMBERS that is counted; a larger group has a row of bits,
// one for each i, and a count before each word of them, 32 groups at a time.
constexpr int PB_FEW_MEMBERS = 64;
__device__ int pb_double(const PbArrays& a, PbShared& sh, uint16_t* A, uint16_t* B, const uint16_t* rank, uint16_t* next, int span, int turn, int n, int tid, int nt) {
    const int lane = tid & 31, w = tid >> 5, nw = nt >> 5, W = a.N2 >> 5;
    uint32_t* key = reinterpret_cast<uint32_t*>(a.key);
    uint32_t* bits = key + a.N2;                           // [32][W]
    uint16_t* before = reinterpret_cast<uint16_t*>(a.tok) + a.N2;                    // [32][W]
    uint16_t* end = a.end;                                 // of a larger group also, one on, its row
    uint32_t alone = 0;
    int mine = 0;
    for (int j = tid, nth = 0; j < n; j += nt, nth++) {
        uint32_t p, g;
        bool ends;
        if (pb_alone(A, rank, end, j, n, p, g, ends)) { alone |= 1u << nth; B[j] = (uint16_t)(p | PB_ALONE); next[p] = (uint16_t)j; mine++; continue; }
        if (ends && j + 1 - (int)g > PB_FEW_MEMBERS) end[g + 1] = (uint16_t)atomicAdd(&sh.rows, 1);
        key[j] = ((int)p >= span ? (uint32_t)rank[p - span] + 1u : 0u) << 16 | p;
    }
    pb_sync(nt);
    if (tid == 0) sh.groups[~turn & 1] = 0;
    for (int j = tid, nth = 0; j < n; j += nt, nth++) {
        if (alone >> nth & 1u) continue;
        const uint32_t k = key[j], same = k & ~0xFFFFu, p = k & 0xFFFFu, g = rank[p], e = end[g];
        if (e - g > PB_FEW_MEMBERS) continue;
        int less = 0, ahead = 0;
#pragma unroll 4
        for (uint32_t i = g; i < e; i++) {
            const uint32_t x = key[i];
            less += x < k; ahead += x < same;
        }
        B[g + less] = (uint16_t)p;
        next[p] = (uint16_t)(g + ahead);
        mine += less == ahead;
    }
    const int rows = sh.rows;
    const uint32_t g0 = rank[span - 1];                    // the group of the one prefix that has `span` tokens: it comes first
    if (rows > 0 && tid == 0 && end[g0] - (int)g0 > PB_FEW_MEMBERS) { B[g0] = (uint16_t)(span - 1); next[span - 1] = (uint16_t)g0; mine++; }
    for (int row0 = 0; row0 < rows; row0 += 32) {
        const int here = min(32, rows - row0);
        for (int i = tid; i < (here * W + 3) >> 2; i += nt) reinterpret_cast<uint4*>(bits)[i] = make_uint4(0, 0, 0, 0);
        pb_sync(nt);
        for (int i = tid; i < n; i += nt) {
            const int p = (A[i] & ~PB_ALONE) + span;
            if (p >= n) continue;
            const uint32_t g = rank[p];
            if (end[g] - (int)g <= PB_FEW_MEMBERS) continue;
            const uint32_t row = end[g + 1] - row0;
            if (row < 32) atomicOr(&bits[row * W + (i >> 5)], 1u << (i & 31));
        }
        pb_sync(nt);
        for (int r = w; r < here; r += nw) {
            int run = 0;
            for (int c = 0; c < W; c += 32) {
                const int v = c + lane < W ? __popc(bits[r * W + c + lane]) : 0;
                const int s = sum_upto(v, lane);
                if (c + lane < W) before[r * W + c + lane] = (uint16_t)(run + s - v);
                run += __shfl_sync(0xFFFFFFFFu, s, 31);
            }
        }
        pb_sync(nt);
        for (int i = tid; i < n; i += nt) {
            const int q = A[i] & ~PB_ALONE, p = q + span;
            if (p >= n) continue;
            const uint32_t g = rank[p];
            if (end[g] - (int)g <= PB_FEW_MEMBERS) continue;
            const uint32_t row = end[g + 1] - row0;
            if (row >= 32) continue;
            const int word = (int)row * W, h = rank[q], first = g == g0 ? 1 : 0;
            const int at = first + before[word + (i >> 5)] + __popc(bits[word + (i >> 5)] & ((1u << (i & 31)) - 1u));
            const int head = first + before[word + (h >> 5)] + __popc(bits[word + (h >> 5)] & ((1u << (h & 31)) - 1u));
            B[g + at] = (uint16_t)p;
            next[p] = (uint16_t)(g + head);
            mine += at == head;
        }
        if (row0 + 32 < rows) pb_sync(nt);
    }
    if (rows > 0 && tid == 0) sh.rows = 0;                 // (all threads have passed a barrier since they read it)
    return pb_groups(sh, turn, mine, tid, nt);
}

// The automaton of a text of n tokens for the empty slot b: every record, transition and table entry Expand would
// leave, and the dynamic words of the slot's control block.  Run by nt threads (tid 0 .. nt - 1, whole warps, barrier 1);
// the result is valid in all of them.  The tokens have been checked and lie in the slot's text and in the `tok` array;
// 1 < n <= PB_MAX.
__device__ void pb_build(const SamBatchView& W, int b, uint32_t* cb, int n, unsigned char* smem,
                         PbShared& sh, int tid, int nt, PbResult& out) {
    const int lane = tid & 31, w = tid >> 5, nw = nt >> 5;
    const int N2 = pb_size(n);
    const PbArrays a = pb_arrays(smem, N2);
    const int32_t* text = W.text + (size_t)b * W.text_stride;

    // ---- sort
    uint16_t *A = a.A, *B = a.B;
    int top = 0, span = 1;                                 // rank level, and the tokens its ranks compare
    int spans[PB_LEVELS];
#pragma unroll
    for (int i = 0; i < PB_LEVELS; i++) spans[i] = 1;
    int groups = pb_group(a, sh, smem, n, tid, nt), turn = 1;
    while (groups < n && span < n) {                       // (ranks of n tokens are all different)
        const uint16_t* r = a.lev + (size_t)top * N2;
        const int to = top < PB_LEVELS - 1 ? top + 1 : top;                          // the last array is used again for longer spans
        uint16_t* next = a.lev + (size_t)to * N2;
        groups = to == top ? 0 : pb_refine(a, sh, A, B, r, next, span, turn, n, tid, nt);
        if (groups == 0) {
            uint16_t* between = reinterpret_cast<uint16_t*>(a.tok);
            groups = pb_double(a, sh, A, B, r, between, span, turn++, n, tid, nt);
            uint16_t* t = A; A = B; B = t;
            if (groups == n || 2 * span >= n) break;       // (where all ranks differ they say nothing of shared suffixes)
            groups = pb_double(a, sh, A, B, between, next, 2 * span, turn, n, tid, nt);
        }
        uint16_t* t = A; A = B; B = t;
        span *= 4;
        turn++;
        top = to;
#pragma unroll
        for (int i = 0; i < PB_LEVELS; i++) if (i == top) spans[i] = span;
    }
    // ---- sorted order, shared suffix lengths
    for (int j = tid; j < N2; j += nt) {
        int x = 0, p = 0xFFFF;
        if (j < n) p = A[j] & ~PB_ALONE;
        if (j > 0 && j < n) {
            const int q = A[j - 1] & ~PB_ALONE;
            int equal = -1;                                // the last level whose ranks are equal: most neighbours differ at the first
#pragma unroll
            for (int i = 0; i < PB_LEVELS; i++) if (equal == i - 1 && i <= top && a.lev[(size_t)i * N2 + p] == a.lev[(size_t)i * N2 + q]) equal = i;
#pragma unroll
            for (int i = PB_LEVELS - 1; i >= 0; i--) {
                if (i <= equal) {
                    const uint16_t* r = a.lev + (size_t)i * N2;
                    while (p - x >= 0 && q - x >= 0 && r[p - x] == r[q - x]) x += spans[i];
                }
            }
        }
        const uint32_t leaf = (uint32_t)x << 16 | (uint32_t)p;
        a.tree[N2 + j] = leaf;
        pb_grow(a, leaf, N2, j - lane, lane);                // (N2 and nt are whole warps)
    }
    pb_sync(nt);
    for (int j = tid; j < n; j += nt) a.rank[A[j] & ~PB_ALONE] = (uint16_t)j;
    if (w == 0)                                              // the other levels, of at most 256 nodes
        for (int width = N2 >> 5; width > 1; width >>= 5) {
            for (int at = 0; at < width; at += 32) pb_grow(a, a.tree[width + at + (lane & (width - 1))], width, at, lane);
            __syncwarp();
        }
    for (int j = tid; j < N2; j += nt) a.first[j] = 0xFFFFFFFFu;
    if (tid == 0) { sh.root_deg = 0; sh.err = 0; }
    if (tid < 16) sh.cls_n[tid] = 0;
    pb_sync(nt);

    // ---- intervals
    for (int j = tid; j < n; j += nt) {
        const uint32_t l = pb_h(a, j);
        uint32_t c = 0;
        if (l > 0) {
            uint32_t e = 0xFFFFu;
            const int i = pb_left(a, j - 1, l + 1, e);
            c = (uint32_t)i;                               // a boundary to the left with the same h: the same interval
            const uint32_t hi = pb_h(a, i);
            if (hi < l) {
                e = min(e, a.tree[N2 + j] & 0xFFFFu);
                const int r = pb_right(a, j, l, e);
                const uint32_t hr = pb_h(a, r);
                a.enode[j] = (uint16_t)e;
                a.parent[j] = (uint16_t)(hi == 0 && hr == 0 ? 0 : hi >= hr ? i : r);
                c = (uint32_t)j;
            }
        }
        a.canon[j] = (uint16_t)c;
    }
    pb_sync(nt);
    for (bool moved = true; moved;) {                      // each boundary to the first of its interval, jumping over jumps
        bool m = false;
        for (int j = tid; j < n; j += nt) {
            const uint32_t was = a.canon[j];
            uint32_t c = was, d = a.canon[c];
            for (int k = 0; k < 3 && c != d; k++) { c = d; d = a.canon[c]; }
            if (c != was) a.canon[j] = (uint16_t)c;
            m |= c != d;
        }
        moved = pb_sync_or(nt, m);
    }
    for (int j = tid; j < n; j += nt) if (j > 0 && a.canon[j] == j) a.parent[j] = a.canon[a.parent[j]];
    pb_sync(nt);

    // ---- longest suffixes that end earlier; who clones
    for (int p = tid; p < n; p += nt) {
        uint32_t x = pb_leaf(a, (uint32_t)p);
        while (x != 0 && a.enode[x] == p) x = a.parent[x]; // (as many rounds in all as there are intervals)
        a.wnode[p] = (uint16_t)x;
        if (x != 0 && a.enode[x] + 1u != pb_h(a, (int)x)) atomicMin(&a.first[x], (uint32_t)p);
    }
    pb_sync(nt);
    const int chunks = (n + 31) >> 5;
    for (int c = w; c < chunks; c += nw) {
        const int p = 32 * c + lane;
        const uint32_t x = p < n ? a.wnode[p] : 0u;
        const bool cl = x != 0 && a.first[x] == (uint32_t)p;
        const unsigned mask = __ballot_sync(0xFFFFFFFFu, cl);
        if (cl) a.wnode[p] = (uint16_t)(x | 0x8000u);
        if (lane == 0) sh.chunk[c] = (int16_t)__popc(mask);
    }
    pb_sync(nt);
    if (w == 0) {                                          // clones before each chunk of 32 tokens
        int run = 0;
        for (int base = 0; base < chunks; base += 32) {
            const int v = base + lane < chunks ? sh.chunk[base + lane] : 0;
            const int s = sum_upto(v, lane);
            if (base + lane < chunks) sh.chunk[base + lane] = (int16_t)(run + s - v);
            run += __shfl_sync(0xFFFFFFFFu, s, 31);
        }
        if (lane == 0) sh.clones = run;
    }
    for (int j = tid; j < n; j += nt)                      // from here on: the handle of the interval's state
        if (j > 0 && a.canon[j] == j) {
            const uint32_t e = a.enode[j];
            a.first[j] = e + 1u == pb_h(a, j) ? e << 1 : a.first[j] << 1 | 1u;
        }
    pb_sync(nt);
    uint32_t* pstate = W.pstate + (size_t)b * W.text_stride;
    if (32 * tid < n) asm volatile("prefetch.global.L1 [%0];" ::"l"(text + 32 * tid));       // for the transitions' tokens
    for (int c = w; c < chunks; c += nw) {
        const int p = 32 * c + lane;
        const bool cl = p < n && pb_clones(a, (uint32_t)p);
        const unsigned mask = __ballot_sync(0xFFFFFFFFu, cl);
        if (p < n) {
            const uint32_t id = (uint32_t)(p + 1 + sh.chunk[c] + __popc(mask & ((1u << lane) - 1u)));
            a.idc[p] = (uint16_t)id;
            pstate[p] = id;
            // suffix links
            uint32_t x = pb_leaf(a, (uint32_t)p);
            if (x != 0 && pb_h(a, (int)x) == (uint32_t)p + 1u) x = a.parent[x];      // the prefix occurs again: the interval is its own
            const uint32_t y = a.wnode[p] & 0x7FFFu, yl = pb_h(a, (int)y);
            a.link[2 * p] = (uint16_t)pb_state(a, x); a.llen[2 * p] = (uint16_t)pb_h(a, (int)x);    // (h[0] is 0)
            a.clen[p] = (uint16_t)yl;                      // (only this thread has read the rank that was there)
            if (cl) {
                const uint32_t up = a.parent[y];
                a.link[2 * p + 1] = (uint16_t)pb_state(a, up); a.llen[2 * p + 1] = (uint16_t)pb_h(a, (int)up);
            }
        }
    }
    // the root's table entries are given out from a bitmap, in place of `canon`, if that is large enough
    uint32_t* taken = reinterpret_cast<uint32_t*>(a.canon);
    const bool bitmap = W.root_cap <= 16 * N2;
    pb_sync(nt);
    if (bitmap) for (int j = tid; j < (N2 >> 1); j += nt) taken[j] = 0;
    uint16_t* clone = a.parent;                            // the positions that clone, one after the other: all states are n + n_clones
    for (int p = tid; p < n; p += nt) {
        a.deg[p] = 0;
        if (pb_clones(a, (uint32_t)p)) clone[a.idc[p] - p - 1] = (uint16_t)p;
    }
    pb_sync(nt);
    const int states = n + sh.clones;
    auto state = [&](int q) { return q < n ? 2u * (uint32_t)q : 2u * clone[q - n] + 1u; };
    auto block_of = [&](uint32_t u) { return (u & 1) ? a.canon + (u >> 1) : reinterpret_cast<uint16_t*>(a.first) + (u & ~1u); };

    // ---- transitions: count them (the root's go to its table at once)
    uint2* root = W.root_tab + (size_t)b * W.root_cap;
    const uint32_t cap_mask = (uint32_t)W.root_cap - 1u, bmask = (uint32_t)(W.root_cap / SAM_ROOT_BUCKET) - 1u;
    for (int q = tid; q - lane < states; q += nt) {        // (whole warps)
        const bool live = q < states;
        const uint32_t u = live ? state(q) : 0u, len = live ? pb_len(a, u) : 0u;
        const bool from_root = live && a.llen[u] == 0;
        uint32_t t = 0;
        if (from_root) t = (uint32_t)text[pb_end(a, u)];
        PbChain c = pb_chain(a, live, u, len, n, lane);
        pb_walk(a, c, n, lane, [&](uint32_t v, bool on, int, bool) {
            if (on) atomicAdd(&a.deg[v >> 1], (v & 1) ? 0x10000u : 1u);
        });
        if (!from_root) continue;
        const uint2 val = make_uint2(t, pb_id(a, u) | (len == 1 ? SAM_FLAG : 0u));
        uint32_t at = (sam_hash1(t) & bmask) * SAM_ROOT_BUCKET;
        for (uint32_t i = 0; i <= cap_mask; i++, at = (at + 1) & cap_mask) {
            if (bitmap) {
                const uint32_t bit = 1u << (at & 31);
                if (!(atomicOr(&taken[at >> 5], bit) & bit)) { root[at] = val; break; }
            } else if (atomicCAS(reinterpret_cast<unsigned long long*>(root + at), (unsigned long long)SAM_NONE,
                                 (unsigned long long)val.y << 32 | val.x) == (unsigned long long)SAM_NONE) break;
        }
        atomicAdd(&sh.root_deg, 1);
    }
    pb_sync(nt);

    // ---- room: records, and edge blocks by size, largest first, so that none crosses a slab
    unsigned long long pool = 0;                           // (read here, where nobody waits for it)
    if (tid == 0) pool = *reinterpret_cast<const volatile unsigned long long*>(W.pool_hdr);
    for (int q = tid; q < states; q += nt) {
        const uint32_t u = state(q), d = a.deg[u >> 1] >> ((u & 1) * 16) & 0xFFFFu;
        if (d > 2) {
            const int k = d <= SAM_BLOCK_MIN ? 0 : 28 - __clz(d - 1);                // 16 << k entries
            *block_of(u) = (uint16_t)atomicAdd(&sh.cls_n[k], 1u);                    // its number among those of its size
            atomicOr(&a.deg[u >> 1], (u & 1) ? 0x80000000u : 0x8000u);               // from here on: it has an edge block
        }
    }
    pb_sync(nt);
    if (w == 0) {
        const int n_rec = ((n + sh.clones) >> (W.slab_shift - 5)) + 1;
        uint32_t units = 0;
        if (lane == 0) for (int k = 15; k >= 0; k--) { sh.cls_base[k] = units; units += sh.cls_n[k] << k; }
        units = __shfl_sync(0xFFFFFFFFu, units, 0);
        const uint32_t slab_units = 1u << (W.slab_shift - 7);
        const int n_blk = (int)((units + slab_units - 1) / slab_units);
        int err = 0;
        if (n_rec > SAM_MAX_REC_SLABS || n_blk > PB_BLOCK_SLABS) err = SAM_SEQ_CAPACITY;
        else pb_take_slabs(W, pool, n_rec + n_blk, b, sh.slab, lane, err);
        __syncwarp();
        if (lane == 0) {
            sh.err = err; sh.n_rec_slabs = n_rec;
            if (!err) {
                const uint32_t last = sh.slab[n_rec + n_blk - 1];
                cb[CB_BLK_CUR] = n_blk ? (last << (W.slab_shift - 7)) + (units - (uint32_t)(n_blk - 1) * slab_units) : 0u;
                cb[CB_BLK_END] = n_blk ? (last + 1u) << (W.slab_shift - 7) : 0u;
            }
        }
    }
    pb_sync(nt);
    if (sh.err) { out.err = sh.err; out.s2 = out.l2 = out.e2 = 0; return; }
    const int rps_shift = W.slab_shift - 5;
    const uint32_t* blk_slab = sh.slab + sh.n_rec_slabs;
    const uint32_t us = W.slab_shift - 7;                  // log2 of the 128-byte units of a slab
    auto record = [&](uint32_t id) {
        return reinterpret_cast<uint4*>(W.pool + ((size_t)sh.slab[id >> rps_shift] << W.slab_shift)) + 2 * (size_t)(id & ((1u << rps_shift) - 1));
    };
    // ---- records
    for (int q = tid; q < states; q += nt) {
        const uint32_t u = state(q), d = a.deg[u >> 1] >> ((u & 1) * 16) & 0x7FFFu;
        uint4 bw = make_uint4(0, 0, 0, 0);
        if (d > 2) {
            const int k = d <= SAM_BLOCK_MIN ? 0 : 28 - __clz(d - 1);
            uint16_t* nth = block_of(u);
            const uint32_t at = sh.cls_base[k] + ((uint32_t)*nth << k);
            *nth = (uint16_t)at;                           // (at most two units for each of 8192 tokens)
            bw = make_uint4((blk_slab[at >> us] << us) + (at & ((1u << us) - 1u)), (uint32_t)SAM_BLOCK_MIN << k, 0, 0);
        }
        uint4* rec = record(pb_id(a, u));
        rec[0] = make_uint4(pb_len(a, u), pb_id(a, a.link[u]), pb_end(a, u) + 1, d);
        rec[1] = bw;
    }
    pb_sync(nt);

    // ---- transitions: write them
    for (int q = tid; q - lane < states; q += nt) {
        const bool live = q < states;
        const uint32_t u = live ? state(q) : 0u;
        const uint32_t t = live ? (uint32_t)text[pb_end(a, u)] : 0u, idu = live ? pb_id(a, u) : 0u, len = live ? pb_len(a, u) : 0u;
        PbChain c = pb_chain_again(a, live, u, len);
        uint32_t to = idu | (c.lv + 1 == len ? SAM_FLAG : 0u);      // (only the first is solid)
        pb_walk(a, c, n, lane, [&](uint32_t v, bool on, int owner, bool all) {
            uint2 edge = make_uint2(t, to);
            if (all) { edge.x = __shfl_sync(0xFFFFFFFFu, t, owner); edge.y = __shfl_sync(0xFFFFFFFFu, to, owner); }
            to = idu;
            if (!on) return;
            const uint32_t h = v >> 1, odd = v & 1, old = atomicSub(&a.deg[h], odd ? 0x10000u : 1u);
            const uint32_t unit = *block_of(v), id = a.idc[h] + odd, was = odd ? old >> 16 : old & 0xFFFFu;
            uint2* at = (was & 0x8000u) ? reinterpret_cast<uint2*>(W.pool + ((((size_t)blk_slab[unit >> us]) << us) + (unit & ((1u << us) - 1u))) * 128)
                                        : reinterpret_cast<uint2*>(record(id) + 1);
            at[(was & 0x7FFFu) - 1u] = edge;
        });
    }
    pb_sync(nt);

    // ---- the slot
    const uint32_t last = (uint32_t)(n - 1) << 1, s2 = a.link[last];
    out.err = 0;
    out.s2 = (int32_t)pb_id(a, s2); out.l2 = (int32_t)pb_len(a, s2);
    out.e2 = s2 == PB_ROOT ? 0 : (int32_t)pb_end(a, s2) + 1;
    if (tid < sh.n_rec_slabs) cb[CB_SLABTAB + tid] = sh.slab[tid];                   // (nt >= SAM_MAX_REC_SLABS)
    if (tid == 0) {
        cb[CB_NTOK] = (uint32_t)n; cb[CB_NSTATES] = (uint32_t)(1 + n + sh.clones); cb[CB_LAST] = pb_id(a, last);
        cb[CB_S2] = (uint32_t)out.s2; cb[CB_L2] = (uint32_t)out.l2;
        cb[CB_NRECSLABS] = (uint32_t)sh.n_rec_slabs; cb[CB_ROOTDEG] = (uint32_t)sh.root_deg;
    }
    if (out.l2 > 0 && tid < 2) reinterpret_cast<uint4*>(cb + CB_REC2)[tid] = record((uint32_t)out.s2)[tid];
}

}  // namespace
