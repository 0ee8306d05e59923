// Tree drafts from the static automaton: best-first expansion over the top-k successors
// (Algorithm 5 of SAM-Decoding, "Drafting via Prim's Algorithm", with the successor frequencies of
// Appendix A.1/A.2).
//
// One warp per slot.  The queue lives in shared memory as plain arrays; an entry holds its path
// probability, its place in the order of pushes, token, parent node, the state's freq and the state's
// successor candidates (its two inline transitions, or its precomputed top-k if its transitions are hashed).
// Because a state's candidates travel with its entry, expanding a popped node needs exactly one round of
// reads: lanes 0..n-1 each fetch one child's freq, record and, if flagged, top-k entry together.
//   - Most nodes are states with one successor that occurs as often as they do: inside a passage the corpus holds once or
//     several times.  Such a stretch is one entry, a path, pushed again with each pop, its tokens those of the corpus.
//     Where the state occurs once the path goes on to the end of the corpus, otherwise over as many states as the
//     automaton's `path` says; the state it ends in is then an ordinary entry whose candidates are read when it is popped.
//   - The entries with the largest probability are popped together as long as they are paths: each goes back to the end
//     of the line with the same probability, so they take turns, and lane t writes the t-th node of up to 32 with one read
//     of the corpus, which the pops after it do not wait for.  Who else has the probability of the first in line is only looked
//     up where that is a path: an entry that is none costs one look through the queue, as if there were no paths.
// us, seeds of 64 slots with k = 4 (one pop and one round of reads for each node): 8 nodes 11.7, 7.8, 8.1 (10.4), 20 nodes 24.2,
// 11.6, 12.6 (18.6 to 20.6), 40 nodes 26.4, 15.8, 15.8 (33 to 35); 4096 slots: 8 nodes 12.2 (14.5), 100 nodes 74 (316).  Bound by the
// pops that are not paths, one after the other, 0.7 to 1.2 us each; a call is as long as its slowest tree, and a tree whose paths
// are all one or two tokens long (24.2) gains nothing by them.
// Probabilities are IEEE float32: quotient freq(child) / freq(state) rounded first,
// then the product with the parent's probability.
#include "common.h"

namespace {

constexpr unsigned FULL = 0xFFFFFFFFu;

struct TreeArgs {
    SamStaticView S;
    const int32_t* states; const int32_t* start_tokens;
    int32_t batch, max_size, k;
    int32_t* tokens; int32_t* parents; float* probs; int32_t* sizes;
};

// Successor candidates of a state, by one lane: (token, target | F) pairs; returns how many.  From the record of a state
// with at most two transitions, in record order ...
__device__ __forceinline__ int inline_candidates(const uint4& a, const uint4& b, uint32_t ctok[SAM_TOPK_MAX], uint32_t ctgt[SAM_TOPK_MAX]) {
    ctok[0] = b.x; ctgt[0] = b.y; ctok[1] = b.z; ctgt[1] = b.w;
    return a.w <= 2u ? (int)a.w : 0;                        // (an unflagged reference to a hashed state cannot happen)
}
// ... or from the top-k table, in top-k order.
__device__ __forceinline__ int load_topk(const SamStaticView& S, uint32_t u, int k, uint32_t ctok[SAM_TOPK_MAX], uint32_t ctgt[SAM_TOPK_MAX],
                                         bool& ordered) {
    ordered = true;
    uint32_t at = sam_hash1(u) & S.topk_mask;
    for (uint32_t probe = 0; probe <= S.topk_mask; probe++) {
        // the whole 64-byte entry in one round of reads; the header decides afterwards
        const uint4 h = __ldg(S.topk + (size_t)at * 4), w1 = __ldg(S.topk + (size_t)at * 4 + 1),
                    w2 = __ldg(S.topk + (size_t)at * 4 + 2), w3 = __ldg(S.topk + (size_t)at * 4 + 3);
        if (h.x == u) {
            // layout: {state, n, 0, 0} {tok0..3} {tok4, tok5, tgt0, tgt1} {tgt2..5}
            ctok[0] = w1.x; ctok[1] = w1.y; ctok[2] = w1.z; ctok[3] = w1.w; ctok[4] = w2.x; ctok[5] = w2.y;
            ctgt[0] = w2.z; ctgt[1] = w2.w; ctgt[2] = w3.x; ctgt[3] = w3.y; ctgt[4] = w3.z; ctgt[5] = w3.w;
            int n = (int)h.y;
            return n < k ? n : k;
        }
        if (h.x == SAM_NONE) return 0;
        at = (at + 1) & S.topk_mask;
    }
    return 0;
}

constexpr int CAND_WORDS = 2 * SAM_TOPK_MAX;                // an entry's candidates: tokens, then targets
constexpr uint32_t ENTRY_ORDERED = 256u, ENTRY_PATH = 512u, ENTRY_ENDS = 1024u, ENTRY_LATE = 2048u;   // flags beside the number of candidates
constexpr int PATH_LEFT = 16;                               // q_n >> PATH_LEFT: nodes left on the path; then, unless it ENDS, the entry
                                                            // is that of its last state (q_cand[0]), LATE: its token is in the corpus at
                                                            // q_tok, its candidates have not been read
constexpr uint32_t PATH_ENDLESS = SAM_PATH_MAX;             // (more than any tree has nodes)
static_assert(PATH_ENDLESS > 128 && PATH_ENDLESS < 1u << (32 - PATH_LEFT), "nodes left fit beside the flags");

__global__ void __launch_bounds__(32) tree_draft_kernel(const __grid_constant__ TreeArgs A) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
    extern __shared__ uint32_t smem[];
    __shared__ int top[32], turn[32];                       // the entries with the largest probability, as found and in order
    const int b = blockIdx.x, lane = threadIdx.x;
    const unsigned lt = (1u << lane) - 1u;
    const int K = A.k, M = A.max_size;
    const int Q = M * K + 1;
    uint32_t* q_key = smem;                                 // bits of the probability, plus one; 0: not in the queue
    uint32_t* q_seq = smem + Q;                             // place in the order of pushes
    uint32_t* q_tok = smem + 2 * Q;                         // of a path: the corpus position of the next node's token
    int32_t* q_par = reinterpret_cast<int32_t*>(smem + 3 * Q);
    uint32_t* q_freq = smem + 4 * Q;
    uint32_t* q_n = smem + 5 * Q;                           // candidates | flags
    uint32_t* q_cand = smem + 6 * Q;                        // [Q][CAND_WORDS]

    int32_t* out_tok = A.tokens + (size_t)b * M;
    int32_t* out_par = A.parents + (size_t)b * M;
    float* out_p = A.probs ? A.probs + (size_t)b * M : nullptr;

    const int32_t s0 = A.states[b];
    int n_out = 0;
    if (s0 > 0 && (int64_t)s0 < A.S.n_states) {
        if (lane == 0) {                                    // the start node: probability 1
            uint32_t ctok[SAM_TOPK_MAX], ctgt[SAM_TOPK_MAX];
            bool ordered = false;
            const uint4 a = __ldg(A.S.rec + 2 * (size_t)s0), r = __ldg(A.S.rec + 2 * (size_t)s0 + 1);
            const int n = a.w > 2u ? load_topk(A.S, (uint32_t)s0, K, ctok, ctgt, ordered) : inline_candidates(a, r, ctok, ctgt);
            q_key[0] = __float_as_uint(1.0f) + 1u; q_seq[0] = 0; q_tok[0] = (uint32_t)A.start_tokens[b]; q_par[0] = -1;
            q_freq[0] = __ldg(A.S.freq + s0); q_n[0] = (uint32_t)n | (ordered ? ENTRY_ORDERED : 0u);
            for (int j = 0; j < SAM_TOPK_MAX; j++) { q_cand[j] = ctok[j]; q_cand[SAM_TOPK_MAX + j] = ctgt[j]; }
        }
        __syncwarp();
        int qn = 1;
        uint32_t seq = 1;
        int32_t late_tok = 0; int late_at = -1;             // a token of the corpus on its way, and the node it is for: the pops after do not wait
        while (n_out < M) {
            // the most probable entry, of equal ones the one pushed first
            uint32_t best = 0, first = 0xFFFFFFFFu;
            int at = 0, ties = 0;
            for (int i = lane; i < qn; i += 32) {
                const uint32_t k = q_key[i], sq = q_seq[i];
                if (k > best) { best = k; first = sq; at = i; ties = 1; }
                else if (k == best) { ties++; if (sq < first) { first = sq; at = i; } }
            }
            const uint32_t key = __reduce_max_sync(FULL, best);
            if (key == 0) break;                            // queue empty
            const float p = __uint_as_float(key - 1u);
            const uint32_t front = __reduce_min_sync(FULL, best == key ? first : 0xFFFFFFFFu);
            at = __shfl_sync(FULL, at, __ffs(__ballot_sync(FULL, best == key && first == front)) - 1);
            const uint32_t nn = q_n[at];
            int group = 1, paths = 0;                       // entries as probable as it; the paths at the head of their line
            if (nn & ENTRY_PATH) {
                group = __reduce_add_sync(FULL, best == key ? ties : 0);
                if (group == 1 || group > 32) {             // (more are too many to sort: the first alone)
                    paths = 1;
                    if (lane == 0) turn[0] = at;
                    __syncwarp();
                } else {
                    int found = 0;
                    for (int base = 0; base < qn; base += 32) {
                        const bool in = base + lane < qn && q_key[base + lane] == key;
                        const unsigned mask = __ballot_sync(FULL, in);
                        if (in) top[found + __popc(mask & lt)] = base + lane;
                        found += __popc(mask);
                    }
                    __syncwarp();
                    int e = 0, rank = 0;
                    uint32_t sq = 0xFFFFFFFFu;
                    if (lane < group) { e = top[lane]; sq = q_seq[e]; }
                    for (int g = 0; g < group; g++) rank += __shfl_sync(FULL, sq, g) < sq;
                    if (lane < group) turn[rank] = e;
                    paths = (int)__reduce_min_sync(FULL, lane < group && !(q_n[e] & ENTRY_PATH) ? (uint32_t)rank : (uint32_t)group);
                    __syncwarp();
                }
            }
            if (paths > 0) {
                // lane t: the t-th pop.  Where other entries stand in line behind the paths, each path is popped once.
                const bool alone = paths == group;
                const int r = lane % paths, i = lane / paths, e = turn[r];
                const int room = (int)(q_n[e] >> PATH_LEFT);
                int count = alone ? 32 : paths;
                count = min(count, M - n_out);
                const int until = room * paths + r;         // the first pop this path cannot serve
                count = (int)__reduce_min_sync(FULL, (uint32_t)(lane < paths ? min(until, count) : count));
                if (late_at >= 0) out_tok[late_at] = late_tok;
                late_at = -1;
                if (lane < count) {
                    late_tok = __ldg(A.S.corpus + q_tok[e] + i); late_at = n_out + lane;
                    out_par[n_out + lane] = i == 0 ? q_par[e] : n_out + lane - paths;
                    if (out_p) out_p[n_out + lane] = p;
                }
                __syncwarp();
                if (lane < paths && lane < count) {         // lane r: path r, popped `c` times
                    const int c = (count - lane + paths - 1) / paths, last = lane + (c - 1) * paths;
                    q_tok[e] += (uint32_t)c; q_par[e] = n_out + last; q_seq[e] = seq + (uint32_t)last;
                    const uint32_t left = q_n[e] - ((uint32_t)c << PATH_LEFT);
                    q_n[e] = left;
                    if ((left >> PATH_LEFT) == 0) {
                        if (left & ENTRY_ENDS) q_key[e] = 0;
                        else q_n[e] = ENTRY_LATE;
                    }
                }
                n_out += count; seq += (uint32_t)count;
                __syncwarp();
                continue;
            }
            const int node = n_out++;
            const uint32_t fs = q_freq[at], tok = q_tok[at];
            if (lane == 0) {
                if (nn & ENTRY_LATE) {
                    if (late_at >= 0) out_tok[late_at] = late_tok;
                    late_tok = __ldg(A.S.corpus + tok); late_at = node;
                } else out_tok[node] = (int32_t)tok;
                out_par[node] = q_par[at];
                if (out_p) out_p[node] = p;
                q_key[at] = 0;
            }
            if (n_out >= M) break;                          // the last node needs no expansion
            // expand: lane j takes candidate j
            int n = (int)(nn & 255u);
            bool ordered = (nn & ENTRY_ORDERED) != 0;
            uint32_t ctok = 0, ctgt = 0, cf = 0;
            uint32_t gtok[SAM_TOPK_MAX], gtgt[SAM_TOPK_MAX];
            if (nn & ENTRY_LATE) {                          // every lane reads the candidates and picks its own
                const uint32_t end = q_cand[(size_t)at * CAND_WORDS], u = end & SAM_IDMASK;
                if (end >> 31) n = load_topk(A.S, u, K, gtok, gtgt, ordered);
                else n = inline_candidates(__ldg(A.S.rec + 2 * (size_t)u), __ldg(A.S.rec + 2 * (size_t)u + 1), gtok, gtgt);
#pragma unroll
                for (int j = 0; j < SAM_TOPK_MAX; j++) if (lane == j && j < n) { ctok = gtok[j]; ctgt = gtgt[j]; }
            } else if (lane < n) {
                ctok = q_cand[(size_t)at * CAND_WORDS + lane]; ctgt = q_cand[(size_t)at * CAND_WORDS + SAM_TOPK_MAX + lane];
            }
            if (n == 0) { __syncwarp(); continue; }
            int cn = 0; bool cord = false;
            uint32_t end1 = 0;                              // first end position
            uint2 path = make_uint2(0, 0);
            if (lane < n) {
                const uint32_t u = ctgt & SAM_IDMASK;
                cf = __ldg(A.S.freq + u);
                if (ctgt >> 31) cn = load_topk(A.S, u, K, gtok, gtgt, cord);
                else {
                    const uint4 ra = __ldg(A.S.rec + 2 * (size_t)u), rb = __ldg(A.S.rec + 2 * (size_t)u + 1);
                    path = __ldg(A.S.path + u);
                    end1 = ra.z;
                    cn = inline_candidates(ra, rb, gtok, gtgt);
                }
            }
            // order two inline candidates by (freq descending, token ascending); keep the first K
            int pos = lane;
            if (!ordered && n == 2) {
                const uint32_t of = __shfl_xor_sync(FULL, cf, 1), ot = __shfl_xor_sync(FULL, ctok, 1);
                if (lane < 2) pos = of > cf || (of == cf && ot < ctok) ? 1 : 0;
            }
            const int keep = n < K ? n : K;
            if (lane < n && pos < keep) {
                const int e = qn + pos;
                uint32_t* to = q_cand + (size_t)e * CAND_WORDS;
                q_key[e] = __float_as_uint(__fmul_rn(p, __fdiv_rn(__uint2float_rn(cf), __uint2float_rn(fs)))) + 1u;
                q_seq[e] = seq + (uint32_t)pos; q_par[e] = node; q_freq[e] = cf;
                if (cf == 1) {
                    const int64_t room = A.S.n_tokens - (int64_t)end1 + 1;
                    q_tok[e] = end1 - 1u;                   // (the token itself is the one before its end position)
                    q_n[e] = ENTRY_PATH | ENTRY_ENDS | (room < (int64_t)PATH_ENDLESS ? (uint32_t)room : PATH_ENDLESS) << PATH_LEFT;
                } else if (path.x > 0) {
                    q_tok[e] = end1 - 1u; to[0] = path.y;
                    q_n[e] = ENTRY_PATH | min(path.x, PATH_ENDLESS) << PATH_LEFT;
                } else {
                    q_tok[e] = ctok; q_n[e] = (uint32_t)cn | (cord ? ENTRY_ORDERED : 0u);
                    for (int j = 0; j < SAM_TOPK_MAX; j++) { to[j] = gtok[j]; to[SAM_TOPK_MAX + j] = gtgt[j]; }
                }
            }
            qn += keep; seq += (uint32_t)keep;
            __syncwarp();
        }
        if (late_at >= 0) out_tok[late_at] = late_tok;
    }
    if (lane == 0) A.sizes[b] = n_out;
    for (int j = n_out + lane; j < M; j += 32) { out_tok[j] = -1; out_par[j] = -1; if (out_p) out_p[j] = 0.f; }
}

}  // namespace

extern "C" int sam_tree_draft(const sam_static_t* st, int32_t batch, const int32_t* states_dev,
                              const int32_t* start_tokens_dev, int32_t max_size, int32_t k,
                              int32_t* tree_tokens_dev, int32_t* tree_parents_dev, float* tree_probs_dev,
                              int32_t* tree_size_dev, void* stream) {
    if (!st || !states_dev || !start_tokens_dev || !tree_tokens_dev || !tree_parents_dev || !tree_size_dev) return SAM_ERR_ARG;
    if (batch < 1 || max_size < 1 || max_size > 128 || k < 1) return SAM_ERR_ARG;
    if (st->info.tree_topk < 1 || k > st->info.tree_topk) return SAM_ERR_ARG;   // built without (enough) tree data
    SamDeviceGuard guard(st->device);
    if (!guard.ok) return SAM_ERR_CUDA;
    TreeArgs A;
    A.S = st->view; A.states = states_dev; A.start_tokens = start_tokens_dev;
    A.batch = batch; A.max_size = max_size; A.k = k;
    A.tokens = tree_tokens_dev; A.parents = tree_parents_dev; A.probs = tree_probs_dev; A.sizes = tree_size_dev;
    const size_t Q = (size_t)max_size * k + 1;
    const size_t smem = Q * (6 + 2 * SAM_TOPK_MAX) * sizeof(uint32_t);
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(tree_draft_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) { sam_set_cuda_error(e); return SAM_ERR_CUDA; }
    }
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)batch); cfg.blockDim = dim3(32); cfg.dynamicSmemBytes = smem; cfg.stream = (cudaStream_t)stream;
    cfg.attrs = attr; cfg.numAttrs = 1;
    SAM_CUDA(cudaLaunchKernelEx(&cfg, tree_draft_kernel, A));
    return SAM_OK;
}
