// Matching on the static automaton.
//
// Transfer (Algorithm 1) run over a step's tokens ends in the state of the longest suffix of (match so far + tokens)
// that occurs in the corpus.  A step reports only that state, and it can be found without visiting the states
// of the tokens in between, each of which costs a dependent read (0.4 us a token for one warp):
//   - a suffix that begins inside the step's tokens is found by walking from the root along transitions only.  One
//     lane per start does so, all lanes reading at once; the walk that reaches the last token from the
//     earliest start is the answer, and most walks end after two or three tokens (static_walks);
//   - the match so far goes on as one more walk, which alone follows suffix links, and only for as long as it covers
//     tokens from before the step (lane 0 of static_walks);
//   - of a long row (a prompt) only the last 8 tokens are walked: if their first start does not reach the end no longer
//     suffix occurs.  If it does, the state's own first occurrence in the corpus is compared with the row leftwards,
//     32 tokens a round: all strings of a state end at the same places, so up to the length of the state's longest
//     string that comparison is the match.  Beyond it, a longer match would have to hold the seam where that string
//     begins, so a few tokens around the seam are walked before anything else is (static_suffix).
#pragma once
#include "common.h"

namespace {

// The two transitions kept in a record: target of t (with its F bit), or SAM_NONE.
__device__ __forceinline__ uint32_t inline_target(const uint4& a, const uint4& b, uint32_t t) {
    if (a.w >= 1 && b.x == t) return b.y;
    if (a.w >= 2 && b.z == t) return b.w;
    return SAM_NONE;
}
__device__ __forceinline__ uint4 shfl4(const uint4& v, int src) {
    return make_uint4(__shfl_sync(FULL, v.x, src), __shfl_sync(FULL, v.y, src), __shfl_sync(FULL, v.z, src), __shfl_sync(FULL, v.w, src));
}
__device__ __forceinline__ void static_record(const SamStaticView& S, uint32_t s, uint4& a, uint4& b) {
    a = __ldg(S.rec + 2 * (size_t)s); b = __ldg(S.rec + 2 * (size_t)s + 1);
}

// Transfer (Algorithm 1) for one token, by a whole warp.  (s, sf, l): state, its F bit, match length;
// root_e is root_row[t]; if have_rec, (pa, pb) is the record of s.
__device__ __forceinline__ void static_transfer(const SamStaticView& S, uint32_t& s, uint32_t& sf, int32_t& l, uint32_t t, uint32_t root_e,
                                                int lane, int& err, bool have_rec, uint4 pa, uint4 pb, ChainCounts& kc) {
    int guard = l + 2;                       // at most l link moves
    bool len_from_rec = false;
    for (;;) {
        if (s == 0) {                        // at the root the match length is 0
            if (root_e != SAM_NONE) { s = root_e & SAM_IDMASK; sf = root_e >> 31; l = 1; SAM_COUNT(kc.b, 1); }
            else l = 0;
            return;
        }
        uint32_t home = sam_hash2(s, t) & S.hash_mask;
        uint4 ent = make_uint4(SAM_NONE, 0, 0, 0);
        if (sf) ent = __ldg(S.hash + (size_t)home * SAM_HASH_BUCKET + (lane & 7));
        uint4 a = pa, b = pb;
        if (!have_rec) { static_record(S, s, a, b); SAM_COUNT(kc.rounds, 1); }
        have_rec = false;
        if (len_from_rec) { l = (int32_t)a.x; len_from_rec = false; }
        uint32_t tgt = inline_target(a, b, t);
        if (tgt == SAM_NONE && a.w > 2) {
            if (!sf) { ent = __ldg(S.hash + (size_t)home * SAM_HASH_BUCKET + (lane & 7)); SAM_COUNT(kc.rounds, 1); }
            for (int probe = 1;; probe++) {
                unsigned hit = __ballot_sync(FULL, ent.x == s && ent.y == t);
                if (hit) { tgt = __shfl_sync(FULL, ent.z, __ffs(hit) - 1); break; }
                unsigned empty = __ballot_sync(FULL, ent.x == SAM_NONE);
                if (empty || probe >= S.hash_max_probe) break;
                home = (home + 1) & S.hash_mask;
                ent = __ldg(S.hash + (size_t)home * SAM_HASH_BUCKET + (lane & 7));
                SAM_COUNT(kc.rounds, 1);
            }
        }
        if (tgt != SAM_NONE) { s = tgt & SAM_IDMASK; sf = tgt >> 31; l += 1; SAM_COUNT(kc.b, 1); return; }
        SAM_COUNT(kc.a, 1);
        s = a.y & SAM_IDMASK; sf = a.y >> 31;            // s <- link(s), l <- len(link(s))
        if (s == 0) l = 0; else len_from_rec = true;
        if (--guard < 0) { err = SAM_SEQ_WALK_LIMIT; return; }
    }
}

// A run of transitions taken in one round of reads, by a whole warp.  The match is in state s (record a, b); lane k holds
// in tkl the token k places on, n of them are there.
//   - s is the state of a whole corpus prefix (len == min_endpos): its transition on the next corpus token is solid, was
//     never redirected and leads to the next prefix's state, so the tokens are compared with the corpus and the
//     state is read from the position -> state array;
//   - otherwise ids a constant one or two apart are guessed (states made token after token along a passage
//     are), and every record on the way is checked to hold the transition.
// Returns how many tokens were taken and moves (s, sf); have: (a, b) is the record of the new s.
__device__ __forceinline__ int static_run(const SamStaticView& S, uint32_t& s, uint32_t& sf, uint4& a, uint4& b, bool& have,
                                          uint32_t tkl, int n, int lane, ChainCounts& kc) {
    const uint32_t t0 = __shfl_sync(FULL, tkl, 0);
    const uint32_t g = inline_target(a, b, t0);
    int r = 0;
    if (a.x == a.z) {
        const int64_t e = (int64_t)a.z;
        int32_t cx = -2; uint32_t px = 0;
        if (lane < n && e + lane < S.n_tokens) { cx = __ldg(S.corpus + e + lane); px = __ldg(S.pstate + e + lane); }
        SAM_COUNT(kc.rounds, 1);
        const unsigned agree = __ballot_sync(FULL, lane < n && (uint32_t)cx == tkl);
        r = (~agree) ? __ffs(~agree) - 1 : 32;
        if (r > 0) {
            const uint32_t ref = __shfl_sync(FULL, px, r - 1);
            s = ref & SAM_IDMASK; sf = ref >> 31; have = false;
        }
    } else if (g != SAM_NONE) {
        const uint32_t d = (g & SAM_IDMASK) - s;
        if (d != 1 && d != 2) return 0;
        const uint32_t id = s + d * (uint32_t)lane;
        uint4 ka = a, kb = b;
        if (lane > 0) {
            ka = make_uint4(0, 0, 0, 0); kb = ka;
            if (lane <= n && (int64_t)id < S.n_states) static_record(S, id, ka, kb);
        }
        SAM_COUNT(kc.rounds, 1);
        const uint32_t nx = inline_target(ka, kb, tkl);
        const unsigned ok = __ballot_sync(FULL, lane < n && nx != SAM_NONE && (nx & SAM_IDMASK) == id + d);
        r = (~ok) ? __ffs(~ok) - 1 : 32;
        if (r > 0) {
            sf = __shfl_sync(FULL, nx, r - 1) >> 31; s += d * (uint32_t)r;
            have = r < 32 && r <= n;
            if (have) { a = shfl4(ka, r); b = shfl4(kb, r); }
        }
    }
    return r;
}

// Transfer for tokens [i, m) of a row of any length, one after the other but for the runs.
__device__ __forceinline__ void static_forward(const SamStaticView& S, const int32_t* toks, int i, int m, uint32_t& s, uint32_t& sf,
                                               int32_t& l, uint4& ra, uint4& rb, bool& have, int lane, int& err, ChainCounts& kc) {
    while (i < m && !err) {
        const int cnt = min(32, m - i);
        uint32_t tk = 0, re = SAM_NONE;
        if (lane < cnt) { tk = (uint32_t)toks[i + lane]; re = __ldg(S.root_row + tk); }
        SAM_COUNT(kc.rounds, 1);
        for (int j = 0; j < cnt && !err;) {
            const uint32_t t = __shfl_sync(FULL, tk, j);
            if (s != 0) {
                if (!have) { static_record(S, s, ra, rb); have = true; SAM_COUNT(kc.rounds, 1); }
                if (cnt - j >= 2 && inline_target(ra, rb, t) != SAM_NONE) {
                    const int r = static_run(S, s, sf, ra, rb, have, __shfl_sync(FULL, tk, (j + lane) & 31), cnt - j, lane, kc);
                    if (r > 0) { l += r; j += r; continue; }
                }
            }
            static_transfer(S, s, sf, l, t, __shfl_sync(FULL, re, j), lane, err, have, ra, rb, kc);
            have = false;
            j++;
        }
        i += cnt;
    }
}

// Walks from every start in a row of w <= 32 tokens (lane k holds token k in tk and its root-row entry in re).  With
// `chain`, lane 0 is not a start but the match so far: state s, length l, i0 tokens of the row already taken,
// have: (ra, rb) is the record of s.  On return (s, sf, l) is the state of the longest suffix found and, if l > 0, (ra, rb)
// its record.
__device__ __forceinline__ void static_walks(const SamStaticView& S, uint32_t tk, uint32_t re, int w, int lane, bool chain, int i0, bool have0,
                                             uint32_t& s, uint32_t& sf, int32_t& l, uint4& ra, uint4& rb, int& err, ChainCounts& kc) {
    bool alive = lane < w && re != SAM_NONE, have = false, need_len = false;
    uint32_t cs = re & SAM_IDMASK, csf = re >> 31;
    int32_t cl = 1;
    int pos = lane + 1;                                   // tokens of the row this walk has taken or begins after
    const bool old = chain && lane == 0;
    if (old) { alive = true; cs = s; csf = sf; cl = l; pos = i0; have = have0; }
    uint4 a = ra, b = rb;
    int guard = l + w + 4;                                // link moves of the match so far
    for (;;) {
        const unsigned done = __ballot_sync(FULL, alive && pos == w);
        if (done && lane > __ffs(done) - 1) alive = false;               // a walk from an earlier start has arrived
        const bool go = alive && (pos < w || !have);
        if (!__any_sync(FULL, go)) break;
        SAM_COUNT(kc.rounds, 1);
        const uint32_t t = __shfl_sync(FULL, tk, pos & 31);
        const bool want_bucket = go && pos < w && csf;
        uint32_t home = 0;
        uint4 ent[SAM_HASH_BUCKET];
        if (want_bucket) {
            home = sam_hash2(cs, t) & S.hash_mask;
#pragma unroll
            for (int e = 0; e < SAM_HASH_BUCKET; e++) ent[e] = __ldg(S.hash + (size_t)home * SAM_HASH_BUCKET + e);
        }
        if (go && !have) static_record(S, cs, a, b);
        if (go) {
            have = true;
            if (need_len) {
                cl = (int32_t)a.x; need_len = false;
                if (cl < pos) alive = false;              // begins inside the row: another lane's walk
            }
            if (alive && pos < w) {
                uint32_t tgt = inline_target(a, b, t);
                if (tgt == SAM_NONE && want_bucket) {     // (every reference to a state with hashed transitions carries the flag)
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
                have = false;
                if (tgt != SAM_NONE) { cs = tgt & SAM_IDMASK; csf = tgt >> 31; cl++; pos++; }
                else if (!old) alive = false;
                else {                                    // the match so far: s <- link(s), l <- len(link(s))
                    cs = a.y & SAM_IDMASK; csf = a.y >> 31;
                    if (cs != 0) need_len = true;
                    else if (pos == 0 && re != SAM_NONE) { cs = re & SAM_IDMASK; csf = re >> 31; cl = 1; pos = 1; }
                    else alive = false;
                    if (--guard < 0) { err = SAM_SEQ_WALK_LIMIT; alive = false; }
                }
            }
        }
    }
    err = __shfl_sync(FULL, err, 0);
    const unsigned done = __ballot_sync(FULL, alive);
    if (!done) { s = 0; sf = 0; l = 0; return; }
    const int first = __ffs(done) - 1;
    s = __shfl_sync(FULL, cs, first); sf = __shfl_sync(FULL, csf, first); l = __shfl_sync(FULL, cl, first);
    ra = shfl4(a, first); rb = shfl4(b, first);
}

// The longest suffix of (match so far + a row of m > 32 tokens) that occurs: (s, sf, l) and, if l > 0, its record.
constexpr int SUFFIX_WINDOW = 8;           // tokens walked first, and on each side of a seam
__device__ __forceinline__ void static_suffix(const SamStaticView& S, const int32_t* toks, int m, int lane, uint32_t& s, uint32_t& sf,
                                              int32_t& l, uint4& ra, uint4& rb, int& err, ChainCounts& kc) {
    const uint32_t s0 = s, sf0 = sf; const int32_t l0 = l;
    const uint4 ra0 = ra, rb0 = rb;
    {
        uint32_t tk = 0, re = SAM_NONE;
        if (lane < SUFFIX_WINDOW) { tk = (uint32_t)toks[m - SUFFIX_WINDOW + lane]; re = __ldg(S.root_row + tk); }
        SAM_COUNT(kc.rounds, 2);
        static_walks(S, tk, re, SUFFIX_WINDOW, lane, false, 0, false, s, sf, l, ra, rb, err, kc);
    }
    if (l < SUFFIX_WINDOW) return;
    for (int turn = 0; !err; turn++) {
        bool ends = false;
        while (!ends) {                                   // the state's first occurrence, leftwards
            const int room = min((int)ra.x, m) - l;
            if (room <= 0) break;
            bool eq = false;
            if (lane < room) eq = __ldg(S.corpus + ((int64_t)ra.z - 1 - l - lane)) == toks[m - 1 - l - lane];
            SAM_COUNT(kc.rounds, 1);
            const unsigned same = __ballot_sync(FULL, eq);
            const int r = (~same) ? __ffs(~same) - 1 : 32;
            l += r;
            ends = r < min(room, 32);
        }
        if (ends || (l >= m && l0 == 0)) return;
        // All of the state's longest string matched (or all of the row): a longer suffix would be another state's, and it
        // would hold the seam between the last token matched and the one before it.
        int c = 0, from = 0;                              // the new match begins at token c and has been taken up to token `from`
        bool have = false;
        const int before = min(SUFFIX_WINDOW, m - l), w = before + SUFFIX_WINDOW;
        if (before > 0 && turn < 12) {
            uint32_t tk = 0, re = SAM_NONE, xs = 0, xsf = 0;
            if (lane < w) { tk = (uint32_t)toks[m - l - before + lane]; re = __ldg(S.root_row + tk); }
            SAM_COUNT(kc.rounds, 2);
            int32_t xl = 0;
            uint4 xa = make_uint4(0, 0, 0, 0), xb = xa;
            static_walks(S, tk, re, w, lane, false, 0, false, xs, xsf, xl, xa, xb, err, kc);
            if (err || xl <= SUFFIX_WINDOW) return;       // nothing that holds the seam occurs
            from = m - l + SUFFIX_WINDOW; c = from - xl;
            s = xs; sf = xsf; l = xl; ra = xa; rb = xb; have = true;
        } else {                                          // (runs of one token and the like: look from further and further to the left)
            c = from = max(0, m - 4 * l);
            s = 0; sf = 0; l = 0;
        }
        const bool whole = c == 0 && l0 > 0;              // it may reach into the match so far
        if (whole) {
            from = 0; s = s0; sf = sf0; l = l0; ra = ra0; rb = rb0; have = true;
        }
        static_forward(S, toks, from, m, s, sf, l, ra, rb, have, lane, err, kc);
        if (l > 0 && !have && !err) { static_record(S, s, ra, rb); SAM_COUNT(kc.rounds, 1); }
        if (whole || l < m - c) return;
    }
}

}  // namespace
