// Build the suffix automaton of a whole text at once, by all threads of a block.
//
// Expand (Algorithm 3), run token after token, is a chain of dependent reads: 0.54 us per token for one warp
// (64 slots x 1024 tokens: 550 us, and 5.8 ms for one slot of 8191).  What it ends with is a function of the text alone,
// and all of it can be read off the sorted order of the text's prefixes:
//   - prefixes are sorted by their tokens from the last to the first; A[j] is the end position of the j-th, h[j]
//     the length of the suffix it shares with its predecessor.  Sorting is by prefix doubling (ranks of 1, 4, 16,
//     ... tokens), so a repeated passage of k tokens costs log4(k) sorts whatever the text is;
//   - l[p], the longest suffix of prefix p that ends anywhere earlier, comes from p's nearest neighbours in
//     sorted order with smaller end positions; e[p] is where that suffix ends first;
//   - Expand of token p makes state c_p (the whole prefix) and, exactly if no state has that suffix as its
//     longest string yet, one clone cl_p with length l[p] and first end position e[p].  A suffix is known by the
//     interval of sorted positions that share it, the interval by the boundary inside it where h is smallest: the
//     first p to claim a boundary makes the clone.  State ids follow by counting clones;
//   - a state's suffix link is the interval around it with the next smaller length;
//   - the transitions into a state u (longest string w, link of length k) are those on w's last token from the states
//     along the suffix links of w without that token, down to length k.
// Nothing here depends on a guess: each of the five statements is the definition of the automaton of the text.
//
// What bounds it: one block's chain of some 60 barriers and shared-memory searches (everything but the outputs
// stays in shared memory, 28 bytes per token).
#pragma once
#include "common.h"

namespace {

constexpr int PB_MAX = 8192;               // longest text: 28 bytes per token of shared memory
constexpr int PB_BYTES_PER_TOKEN = 28;
constexpr int PB_LEVELS = 6;               // rank arrays kept for comparing two prefixes
constexpr int PB_BLOCK_SLABS = 80;         // slabs the edge blocks of one text can take (at most 64, and a remainder)
constexpr uint32_t PB_ROOT = 0xFFFFu;      // handle of the root; a state is (p << 1 | clone)

struct PbShared {                          // what the threads of one build exchange besides the arrays
    int16_t chunk[PB_MAX / 32];
    uint32_t rec_slab[SAM_MAX_REC_SLABS], blk_slab[PB_BLOCK_SLABS];
    uint32_t cls_n[16], cls_base[16];
    int groups, clones, root_deg, err, n_rec_slabs, n_blk_units;
};

struct PbArrays {
    uint64_t* key;                         // sorting; its place is taken by `tree`
    uint16_t* lev; uint16_t* A; uint16_t* H;                       // while sorting
    uint32_t* tree; uint16_t* rank; uint16_t* L; uint16_t* E; uint16_t* idc;
    uint32_t* first; uint16_t* link; uint32_t* deg;
    int N2;                                // size of the sorted order, a power of two
};

__device__ __forceinline__ PbArrays pb_arrays(unsigned char* sm, int N2) {
    PbArrays a;
    const size_t n = (size_t)N2;
    a.N2 = N2;
    a.key = (uint64_t*)sm; a.lev = (uint16_t*)(sm + 8 * n); a.A = (uint16_t*)(sm + 20 * n); a.H = (uint16_t*)(sm + 22 * n);
    a.tree = (uint32_t*)sm; a.rank = (uint16_t*)(sm + 8 * n); a.L = (uint16_t*)(sm + 10 * n); a.E = (uint16_t*)(sm + 12 * n);
    a.idc = (uint16_t*)(sm + 14 * n); a.first = (uint32_t*)(sm + 16 * n); a.link = (uint16_t*)(sm + 20 * n); a.deg = (uint32_t*)(sm + 24 * n);
    return a;
}

__device__ __forceinline__ void pb_sync(int nt) { asm volatile("bar.sync 1, %0;" ::"r"(nt) : "memory"); }

__device__ __forceinline__ uint64_t pb_shfl_xor(uint64_t v, int s) {
    const uint32_t lo = __shfl_xor_sync(0xFFFFFFFFu, (uint32_t)v, s), hi = __shfl_xor_sync(0xFFFFFFFFu, (uint32_t)(v >> 32), s);
    return ((uint64_t)hi << 32) | lo;
}
__device__ __forceinline__ void pb_step(uint64_t& v, int lane, int stride, bool up) {
    const uint64_t o = pb_shfl_xor(v, stride);
    const bool low = (lane & stride) == 0;
    if ((o < v) == (low == up)) v = o;
}

// Bitonic sort of key[0, N2).  Strides below 64 stay in the registers of one warp (two keys a lane).
__device__ void pb_sort(uint64_t* key, int N2, int tid, int nt) {
    const int lane = tid & 31, w = tid >> 5, nw = nt >> 5;
    for (int size = 64; size <= N2; size <<= 1) {
        for (int stride = size >> 1; stride >= 64; stride >>= 1) {
            for (int q = tid; q < (N2 >> 1); q += nt) {
                const int i = ((q & ~(stride - 1)) << 1) | (q & (stride - 1)), k = i + stride;
                const uint64_t x = key[i], y = key[k];
                if ((x > y) == ((i & size) == 0)) { key[i] = y; key[k] = x; }
            }
            pb_sync(nt);
        }
        for (int c = w; c < (N2 >> 6); c += nw) {
            uint64_t x = key[64 * c + lane], y = key[64 * c + 32 + lane];
            if (size == 64) {
#pragma unroll
                for (int sz = 2; sz <= 32; sz <<= 1)
#pragma unroll
                    for (int st = sz >> 1; st; st >>= 1) {
                        pb_step(x, lane, st, sz == 32 ? true : (lane & sz) == 0);
                        pb_step(y, lane, st, sz == 32 ? false : (lane & sz) == 0);
                    }
            }
            const bool up = ((64 * c) & size) == 0;
            if ((x > y) == up) { const uint64_t t = x; x = y; y = t; }
#pragma unroll
            for (int st = 16; st; st >>= 1) { pb_step(x, lane, st, up); pb_step(y, lane, st, up); }
            key[64 * c + lane] = x; key[64 * c + 32 + lane] = y;
        }
        pb_sync(nt);
    }
}

// rank[p] = first sorted position of p's group of equal keys; returns the number of groups.
__device__ int pb_rank(const PbArrays& a, PbShared& sh, uint16_t* rank, int n, int ib, int tid, int nt) {
    const int lane = tid & 31, w = tid >> 5, nw = nt >> 5, chunks = (n + 31) >> 5;
    if (tid == 0) sh.groups = 0;
    pb_sync(nt);
    for (int c = w; c < chunks; c += nw) {
        const int j = 32 * c + lane;
        const bool head = j < n && (j == 0 || (a.key[j] >> ib) != (a.key[j - 1] >> ib));
        const unsigned mask = __ballot_sync(0xFFFFFFFFu, head);
        if (lane == 0) { sh.chunk[c] = mask ? (int16_t)(32 * c + 31 - __clz(mask)) : (int16_t)-1; atomicAdd(&sh.groups, __popc(mask)); }
    }
    pb_sync(nt);
    const uint32_t im = (1u << ib) - 1u;
    for (int c = w; c < chunks; c += nw) {
        const int j = 32 * c + lane;
        const bool head = j < n && (j == 0 || (a.key[j] >> ib) != (a.key[j - 1] >> ib));
        const unsigned mask = __ballot_sync(0xFFFFFFFFu, head);
        int before = 0;                                    // where the group that reaches into this chunk began
        for (int base = c - 1; base >= 0; base -= 32) {
            const int v = base - lane >= 0 ? sh.chunk[base - lane] : -1;
            const unsigned m = __ballot_sync(0xFFFFFFFFu, v >= 0);
            if (m) { before = __shfl_sync(0xFFFFFFFFu, v, __ffs(m) - 1); break; }
        }
        const unsigned mine = mask & (0xFFFFFFFFu >> (31 - lane));
        if (j < n) rank[(uint32_t)a.key[j] & im] = (uint16_t)(mine ? 32 * c + 31 - __clz(mine) : before);
    }
    pb_sync(nt);
    return sh.groups;
}

// The tree over the sorted order: leaf j is h[j] << 16 | A[j], an inner node the two minima of its leaves.
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

// Length of the suffix that p (at sorted position j) shares with its nearest neighbour on one side with a smaller end position.
__device__ __forceinline__ uint32_t pb_earlier_left(const PbArrays& a, int j, uint32_t p) {
    if (j == 0) return 0;
    uint32_t m = pb_h(a, j);
    int i = a.N2 + j - 1;
    while (m) {
        const uint32_t v = a.tree[i];
        if ((v & 0xFFFFu) < p) {
            while (i < a.N2) {
                const uint32_t r = a.tree[2 * i + 1];
                if ((r & 0xFFFFu) < p) i = 2 * i + 1;
                else { m = min(m, r >> 16); i = 2 * i; }
            }
            return m;
        }
        m = min(m, v >> 16);
        while (!(i & 1)) i >>= 1;
        if (i == 1) return 0;
        i -= 1;
    }
    return 0;
}
__device__ __forceinline__ uint32_t pb_earlier_right(const PbArrays& a, int j, uint32_t p) {
    if (j + 1 >= a.N2) return 0;
    uint32_t m = 0xFFFFu;
    int i = a.N2 + j + 1;
    while (m) {
        const uint32_t v = a.tree[i];
        if ((v & 0xFFFFu) < p) {
            while (i < a.N2) {
                const uint32_t x = a.tree[2 * i];
                if ((x & 0xFFFFu) < p) i = 2 * i;
                else { m = min(m, x >> 16); i = 2 * i + 1; }
            }
            return min(m, a.tree[i] >> 16);
        }
        m = min(m, v >> 16);
        while (i & 1) i >>= 1;
        if (i == 0) return 0;
        i += 1;
    }
    return 0;
}

struct PbNode { int lo; uint32_t len, e, up; };            // interval of the strings of length `len` around a prefix: where it
                                                           // begins, its smallest end position, the length of its suffix link
__device__ __forceinline__ PbNode pb_node(const PbArrays& a, int j, uint32_t len) {
    PbNode x;
    uint32_t e = 0xFFFFu;
    x.lo = pb_left(a, j, len, e);
    const int r = pb_right(a, j, len, e);
    x.len = len; x.e = e;
    x.up = max(pb_h(a, x.lo), pb_h(a, r));
    return x;
}
// The boundary that names the interval: the first one inside it where h is as small as `len`.
__device__ __forceinline__ int pb_boundary(const PbArrays& a, int lo, uint32_t len) {
    uint32_t unused = 0xFFFFu;
    return pb_right(a, lo, len + 1, unused);
}
__device__ __forceinline__ uint32_t pb_handle(const PbArrays& a, const PbNode& x) {
    if (x.e + 1 == x.len) return x.e << 1;
    const uint32_t p = a.first[pb_boundary(a, x.lo, x.len)];
    return p == 0xFFFFFFFFu ? PB_ROOT : p << 1 | 1u;       // (every interval has been claimed)
}
__device__ __forceinline__ uint32_t pb_len(const PbArrays& a, uint32_t hd) {
    return hd == PB_ROOT ? 0u : (hd & 1) ? (uint32_t)(a.L[hd >> 1] & 0x7FFF) : (hd >> 1) + 1;
}
__device__ __forceinline__ uint32_t pb_id(const PbArrays& a, uint32_t hd) { return hd == PB_ROOT ? 0u : a.idc[hd >> 1] + (hd & 1); }

// Visit every transition into state u = (p, clone): f(source handle, solid).
template <class F>
__device__ __forceinline__ void pb_into(const PbArrays& a, uint32_t u, F f) {
    const uint32_t p = u >> 1;
    const uint32_t len = pb_len(a, u), low = pb_len(a, a.link[u]);
    uint32_t v = PB_ROOT;
    if (len > 1) {
        if (!(u & 1)) v = (p - 1) << 1;
        else v = pb_handle(a, pb_node(a, a.rank[a.E[p] - 1], len - 1));
    }
    for (uint32_t below = len;;) {
        const uint32_t lv = pb_len(a, v);
        if (lv < low || lv >= below) break;                // (lengths fall along suffix links)
        below = lv;
        f(v, lv + 1 == len);
        if (v == PB_ROOT) break;
        v = a.link[v];
    }
}

__device__ __forceinline__ uint32_t pb_take_slabs(const SamBatchView& W, int want, int b, uint32_t* out, int lane, int& err) {
    // by one warp: all of them with one addition; nothing is taken if they are not all there
    int old = 0;
    if (lane == 0) {
        old = atomicSub(W.pool_hdr, want);
        if (old < want) atomicAdd(W.pool_hdr, want);
    }
    old = __shfl_sync(0xFFFFFFFFu, old, 0);
    if (old < want) { err = SAM_SEQ_CAPACITY; return 0; }
    for (int i = lane; i < want; i += 32) {
        const int idx = W.free_stack[old - 1 - i];
        W.slab_owner[idx] = b;
        out[i] = (uint32_t)idx;
    }
    return (uint32_t)want;
}

struct PbResult { int32_t s2, l2, e2; int err; };

// The automaton of toks[0, n) for the empty slot b: every record, transition and table entry Expand would leave, and the
// dynamic words of the slot's control block.  Run by nt threads (tid 0 .. nt - 1, whole warps, barrier 1); the
// result is valid in all of them.  The tokens have been checked; 1 < n <= PB_MAX.
__device__ void pb_build(const SamBatchView& W, int b, uint32_t* cb, const int32_t* toks, int n, unsigned char* smem,
                         PbShared& sh, int tid, int nt, PbResult& out) {
    const int lane = tid & 31, w = tid >> 5, nw = nt >> 5;
    const int N2 = n <= 64 ? 64 : 1 << (32 - __clz(n - 1));
    const PbArrays a = pb_arrays(smem, N2);
    int32_t* text = W.text + (size_t)b * W.text_stride;
    const int ib = 32 - __clz(n - 1), rb = 32 - __clz(n);  // bits of a position, and of a rank plus one
    const int parts = min(4, (64 - ib) / rb);

    // ---- sort
    for (int j = tid; j < N2; j += nt) {
        uint64_t k = ~0ull;
        if (j < n) { const int32_t t = toks[j]; text[j] = t; k = (uint64_t)(uint32_t)t << ib | (uint32_t)j; }
        a.key[j] = k;
    }
    pb_sync(nt);
    pb_sort(a.key, N2, tid, nt);
    int top = 0, span = 1;                                 // rank level, and the tokens its ranks compare
    int spans[PB_LEVELS];
#pragma unroll
    for (int i = 0; i < PB_LEVELS; i++) spans[i] = 1;
    int groups = pb_rank(a, sh, a.lev, n, ib, tid, nt);
    while (groups < n && span < n) {                       // (ranks of n tokens are all different)
        const uint16_t* r = a.lev + (size_t)top * N2;
        for (int j = tid; j < n; j += nt) {
            uint64_t k = r[j];
            for (int q = 1; q < parts; q++) { const int at = j - q * span; k = k << rb | (at >= 0 ? (uint32_t)r[at] + 1u : 0u); }
            a.key[j] = k << ib | (uint32_t)j;
        }
        for (int j = n + tid; j < N2; j += nt) a.key[j] = ~0ull;
        pb_sync(nt);
        pb_sort(a.key, N2, tid, nt);
        span *= parts;
        if (top < PB_LEVELS - 1) top++;                    // the last array is used again for longer spans
#pragma unroll
        for (int i = 0; i < PB_LEVELS; i++) if (i == top) spans[i] = span;
        groups = pb_rank(a, sh, a.lev + (size_t)top * N2, n, ib, tid, nt);
    }
    // ---- sorted order, shared suffix lengths
    const uint32_t im = (1u << ib) - 1u;
    for (int j = tid; j < n; j += nt) {
        const int p = (int)((uint32_t)a.key[j] & im);
        int x = 0;
        if (j > 0) {
            const int q = (int)((uint32_t)a.key[j - 1] & im);
#pragma unroll
            for (int i = PB_LEVELS - 1; i >= 0; i--) {
                if (i <= top) {
                    const uint16_t* r = a.lev + (size_t)i * N2;
                    while (p - x >= 0 && q - x >= 0 && r[p - x] == r[q - x]) x += spans[i];
                }
            }
        }
        a.A[j] = (uint16_t)p; a.H[j] = (uint16_t)x;
    }
    pb_sync(nt);
    for (int j = tid; j < N2; j += nt) a.tree[N2 + j] = j < n ? (uint32_t)a.H[j] << 16 | a.A[j] : 0xFFFFu;
    pb_sync(nt);
    for (int j = tid; j < n; j += nt) { a.rank[a.A[j]] = (uint16_t)j; }
    for (int width = N2 >> 1; width >= 1; width >>= 1) {
        for (int i = tid; i < width; i += nt) a.tree[width + i] = __vminu2(a.tree[2 * (width + i)], a.tree[2 * (width + i) + 1]);
        if (width > 32) pb_sync(nt); else __syncwarp();      // the last levels are warp 0's alone
    }
    pb_sync(nt);

    // ---- longest suffixes that end earlier; who clones
    for (int j = tid; j < N2; j += nt) a.first[j] = 0xFFFFFFFFu;
    if (tid == 0) { sh.root_deg = 0; sh.err = 0; sh.n_blk_units = 0; }
    if (tid < 16) sh.cls_n[tid] = 0;
    pb_sync(nt);
    for (int p = tid; p < n; p += nt) {
        const int j = a.rank[p];
        const uint32_t l = max(pb_earlier_left(a, j, (uint32_t)p), pb_earlier_right(a, j, (uint32_t)p));
        uint32_t e = 0, r = 0;
        if (l > 0) {
            const PbNode x = pb_node(a, j, l);
            e = x.e;
            if (e + 1 != l) { r = (uint32_t)pb_boundary(a, x.lo, l); atomicMin(&a.first[r], (uint32_t)p); }
        }
        a.L[p] = (uint16_t)l; a.E[p] = (uint16_t)e; a.link[p] = (uint16_t)r;        // (link holds the boundary for now)
        a.deg[p] = 0;
    }
    pb_sync(nt);
    const int chunks = (n + 31) >> 5;
    for (int c = w; c < chunks; c += nw) {
        const int p = 32 * c + lane;
        const bool cl = p < n && a.link[p] != 0 && a.first[a.link[p]] == (uint32_t)p;
        const unsigned mask = __ballot_sync(0xFFFFFFFFu, cl);
        if (cl) a.L[p] |= 0x8000u;
        if (lane == 0) sh.chunk[c] = (int16_t)__popc(mask);
    }
    pb_sync(nt);
    if (w == 0) {                                          // clones before each chunk of 32 tokens
        int run = 0;
        for (int base = 0; base < chunks; base += 32) {
            const int v = base + lane < chunks ? sh.chunk[base + lane] : 0;
            int s = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) { const int t = __shfl_up_sync(0xFFFFFFFFu, s, o); if (lane >= o) s += t; }
            if (base + lane < chunks) sh.chunk[base + lane] = (int16_t)(run + s - v);
            run += __shfl_sync(0xFFFFFFFFu, s, 31);
        }
        const int n_states = 1 + n + run;
        int err = 0;
        const int want = ((n_states - 1) >> (W.slab_shift - 5)) + 1;
        if (want > SAM_MAX_REC_SLABS) err = SAM_SEQ_CAPACITY;
        else pb_take_slabs(W, want, b, sh.rec_slab, lane, err);
        if (lane == 0) { sh.clones = run; sh.n_rec_slabs = want; if (err) sh.err = err; }
    }
    pb_sync(nt);
    if (sh.err) { out.err = sh.err; out.s2 = out.l2 = out.e2 = 0; return; }
    uint32_t* pstate = W.pstate + (size_t)b * W.text_stride;
    for (int c = w; c < chunks; c += nw) {
        const int p = 32 * c + lane;
        const bool cl = p < n && (a.L[p] & 0x8000u);
        const unsigned mask = __ballot_sync(0xFFFFFFFFu, cl);
        if (p < n) {
            const uint32_t id = (uint32_t)(p + 1 + sh.chunk[c] + __popc(mask & ((1u << lane) - 1u)));
            a.idc[p] = (uint16_t)id;
            pstate[p] = id;
        }
    }
    pb_sync(nt);

    // ---- suffix links
    const int rps_shift = W.slab_shift - 5;
    for (int p = tid; p < n; p += nt) {
        const int j = a.rank[p];
        {   // the state of the whole prefix
            PbNode x;
            x.lo = j;
            const uint32_t hr = pb_h(a, j + 1);
            if (hr == (uint32_t)p + 1) x = pb_node(a, j, (uint32_t)p + 1);           // it occurs again
            else x.up = max(pb_h(a, j), hr);
            a.link[2 * p] = (uint16_t)(x.up == 0 ? PB_ROOT : pb_handle(a, pb_node(a, x.lo, x.up)));
        }
        if (a.L[p] & 0x8000u) {
            const PbNode x = pb_node(a, j, a.L[p] & 0x7FFFu);
            a.link[2 * p + 1] = (uint16_t)(x.up == 0 ? PB_ROOT : pb_handle(a, pb_node(a, x.lo, x.up)));
        }
    }
    pb_sync(nt);

    // ---- transitions: count them (the root's go to its table at once)
    uint2* root = W.root_tab + (size_t)b * W.root_cap;
    const uint32_t cap_mask = (uint32_t)W.root_cap - 1u, bmask = (uint32_t)(W.root_cap / SAM_ROOT_BUCKET) - 1u;
    for (int q = tid; q < 2 * n; q += nt) {
        const uint32_t u = (uint32_t)(q < n ? 2 * q : 2 * (q - n) + 1);
        if ((u & 1) && !(a.L[u >> 1] & 0x8000u)) continue;
        pb_into(a, u, [&](uint32_t v, bool solid) {
            if (v != PB_ROOT) { atomicAdd(&a.deg[v >> 1], (v & 1) ? 0x10000u : 1u); return; }
            const uint32_t t = (uint32_t)text[(u & 1) ? a.E[u >> 1] : u >> 1];
            const unsigned long long val = (unsigned long long)(pb_id(a, u) | (solid ? SAM_FLAG : 0u)) << 32 | t;
            uint32_t at = (sam_hash1(t) & bmask) * SAM_ROOT_BUCKET;
            for (uint32_t i = 0; i <= cap_mask; i++, at = (at + 1) & cap_mask)
                if (atomicCAS(reinterpret_cast<unsigned long long*>(root + at), (unsigned long long)SAM_NONE, val) == (unsigned long long)SAM_NONE) break;
            atomicAdd(&sh.root_deg, 1);
        });
    }
    pb_sync(nt);

    // ---- records; edge blocks by size, largest first, so that none crosses a slab
    // (b.x of a record holds the number of its block among those of its size until the blocks have places)
    for (int q = tid; q < 2 * n; q += nt) {
        const uint32_t u = (uint32_t)(q < n ? 2 * q : 2 * (q - n) + 1), p = u >> 1;
        if ((u & 1) && !(a.L[p] & 0x8000u)) continue;
        const uint32_t d = (u & 1) ? a.deg[p] >> 16 : a.deg[p] & 0xFFFFu;
        if (d > 2) {
            const int k = d <= SAM_BLOCK_MIN ? 0 : 28 - __clz(d - 1);                // 16 << k entries
            const uint32_t id = pb_id(a, u);
            uint4* rec = reinterpret_cast<uint4*>(W.pool + ((size_t)sh.rec_slab[id >> rps_shift] << W.slab_shift)) + 2 * (size_t)(id & ((1u << rps_shift) - 1));
            rec[1].x = atomicAdd(&sh.cls_n[k], 1u);
        }
    }
    pb_sync(nt);
    if (w == 0) {
        uint32_t units = 0;
        if (lane == 0) for (int k = 15; k >= 0; k--) { sh.cls_base[k] = units; units += sh.cls_n[k] << k; }
        units = __shfl_sync(0xFFFFFFFFu, units, 0);
        const uint32_t slab_units = 1u << (W.slab_shift - 7);
        const int want = (int)((units + slab_units - 1) / slab_units);
        int err = 0;
        if (want > PB_BLOCK_SLABS) err = SAM_SEQ_CAPACITY;
        else if (want > 0) pb_take_slabs(W, want, b, sh.blk_slab, lane, err);
        __syncwarp();
        if (lane == 0) {
            if (err) sh.err = err;
            else {
                sh.n_blk_units = (int)units;
                cb[CB_BLK_CUR] = want ? (sh.blk_slab[want - 1] << (W.slab_shift - 7)) + (units - (uint32_t)(want - 1) * slab_units) : 0u;
                cb[CB_BLK_END] = want ? (sh.blk_slab[want - 1] + 1u) << (W.slab_shift - 7) : 0u;
            }
        }
    }
    pb_sync(nt);
    // the taken record slabs belong to the slot whatever happens: they go back to the pool at its reset
    if (sh.err) { out.err = sh.err; out.s2 = out.l2 = out.e2 = 0; return; }
    for (int q = tid; q < 2 * n; q += nt) {
        const uint32_t u = (uint32_t)(q < n ? 2 * q : 2 * (q - n) + 1), p = u >> 1;
        if ((u & 1) && !(a.L[p] & 0x8000u)) continue;
        const uint32_t d = (u & 1) ? a.deg[p] >> 16 : a.deg[p] & 0xFFFFu;
        const uint32_t id = pb_id(a, u), e = (u & 1) ? a.E[p] : p;
        uint4* rec = reinterpret_cast<uint4*>(W.pool + ((size_t)sh.rec_slab[id >> rps_shift] << W.slab_shift)) + 2 * (size_t)(id & ((1u << rps_shift) - 1));
        uint4 bw = make_uint4(0, 0, 0, 0);
        if (d > 2) {
            const int k = d <= SAM_BLOCK_MIN ? 0 : 28 - __clz(d - 1);
            const uint32_t at = sh.cls_base[k] + (rec[1].x << k);
            const uint32_t us = W.slab_shift - 7;
            bw = make_uint4((sh.blk_slab[at >> us] << us) + (at & ((1u << us) - 1u)), (uint32_t)SAM_BLOCK_MIN << k, 0, 0);
        }
        rec[0] = make_uint4(pb_len(a, u), pb_id(a, a.link[u]), e + 1, d);
        rec[1] = bw;
    }
    pb_sync(nt);
    for (int p = tid; p < n; p += nt) {                    // bit 15 of a count: the state has an edge block
        const uint32_t v = a.deg[p];
        a.deg[p] = v | ((v & 0xFFFFu) > 2 ? 0x8000u : 0u) | ((v >> 16) > 2 ? 0x80000000u : 0u);
    }
    pb_sync(nt);

    // ---- transitions: write them
    for (int q = tid; q < 2 * n; q += nt) {
        const uint32_t u = (uint32_t)(q < n ? 2 * q : 2 * (q - n) + 1);
        if ((u & 1) && !(a.L[u >> 1] & 0x8000u)) continue;
        const uint32_t t = (uint32_t)text[(u & 1) ? a.E[u >> 1] : u >> 1], idu = pb_id(a, u);
        pb_into(a, u, [&](uint32_t v, bool solid) {
            if (v == PB_ROOT) return;
            const uint32_t was = (v & 1) ? atomicSub(&a.deg[v >> 1], 0x10000u) >> 16 : atomicSub(&a.deg[v >> 1], 1u) & 0xFFFFu;
            const uint32_t k = (was & 0x7FFFu) - 1u, id = pb_id(a, v);
            uint2* rec = reinterpret_cast<uint2*>(W.pool + ((size_t)sh.rec_slab[id >> rps_shift] << W.slab_shift)) + 4 * (size_t)(id & ((1u << rps_shift) - 1));
            uint2* at = (was & 0x8000u) ? reinterpret_cast<uint2*>(W.pool + (size_t)rec[2].x * 128) + k : rec + 2 + k;
            *at = make_uint2(t, idu | (solid ? SAM_FLAG : 0u));
        });
    }
    pb_sync(nt);

    // ---- the slot
    const uint32_t last = (uint32_t)(n - 1) << 1, s2 = a.link[last];
    out.err = 0;
    out.s2 = (int32_t)pb_id(a, s2); out.l2 = (int32_t)pb_len(a, s2);
    out.e2 = s2 == PB_ROOT ? 0 : (int32_t)((s2 & 1) ? a.E[s2 >> 1] : s2 >> 1) + 1;
    if (tid < sh.n_rec_slabs) cb[CB_SLABTAB + tid] = sh.rec_slab[tid];               // (nt >= SAM_MAX_REC_SLABS)
    if (tid == 0) {
        cb[CB_NTOK] = (uint32_t)n; cb[CB_NSTATES] = (uint32_t)(1 + n + sh.clones); cb[CB_LAST] = pb_id(a, last);
        cb[CB_S2] = (uint32_t)out.s2; cb[CB_L2] = (uint32_t)out.l2;
        cb[CB_NRECSLABS] = (uint32_t)sh.n_rec_slabs; cb[CB_ROOTDEG] = (uint32_t)sh.root_deg;
    }
    if (out.l2 > 0 && tid < 2) {
        const uint32_t id = (uint32_t)out.s2;
        const uint4* rec = reinterpret_cast<const uint4*>(W.pool + ((size_t)sh.rec_slab[id >> rps_shift] << W.slab_shift)) + 2 * (size_t)(id & ((1u << rps_shift) - 1));
        reinterpret_cast<uint4*>(cb + CB_REC2)[tid] = rec[tid];
    }
}

}  // namespace
