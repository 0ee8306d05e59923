// Batch objects: workspace layout, slot initialisation and reset, the slab pool's free stack,
// the host-array step, the step replay loop and the inspection calls.
#include "common.h"

#include <atomic>
#include <chrono>
#include <cstring>
#include <new>
#include <vector>

namespace {

constexpr size_t SAM_ZERO_COPY_MAX_BYTES = 4u << 20;     // larger host steps go through two DMA copies
// Outputs of a host step that come back as (word, number) pairs: a fence a slot and no flag, twice the bytes.  us a call as
// pairs / behind the flag: 16 slots (368 words) 15.3 to 16.9 / 16.7 to 17.2, 43 slots (2021 words) 17.9 / 17.9, 44 (2068) 18.0 /
// 17.7, 64 slots of 47 words (3008) 19.5 / 18.5, 87 (4089) 20.5 / 18.8.
constexpr size_t SAM_TAGGED_MAX_WORDS = 2048;
// From how many words of rows on a kernel brings them over ahead of the step's, us a call without / with it: 200 slots (1800
// words) 22.0 / 25.0, 300 (2700) 23.7 / 24.0, 500 (6500) 25.9 / 26.0, 620 (8060) 27.3 / 26.4; 1000 (13000) 39.2 / 36.5.
constexpr size_t SAM_FETCH_MIN_WORDS = 8192;
constexpr size_t SAM_DIRECT_MIN_BYTES = 64u << 10;       // from this size on, page-locked caller arrays are used in place
constexpr int SAM_POLL_LIMIT_US = 2000;                  // how long a host step polls its completion flag

struct WsLayout {
    size_t off_hdr, off_ctrl, off_free, off_owner, off_reset, off_order, off_text, off_pstate, off_root, off_stage, off_pool, total;
    int32_t text_stride, root_cap, slab_shift, pool_slabs, max_host_stride;
    size_t stage_words;
};

inline uint32_t pow2_ceil(uint64_t x) { uint64_t p = 1; while (p < x) p <<= 1; return (uint32_t)p; }

int plan(const sam_batch_opts_t* o, WsLayout* w) {
    if (!o || o->batch < 1 || o->max_seq_len < 1 || o->max_draft_len < 1 || o->max_draft_len > 128 ||
        o->l_bias < 0 || o->min_match < 0 || o->max_host_stride < 0 || o->pool_slabs < 0 ||
        o->stop_token_plus_one < 0 || o->reserved != 0)
        return SAM_ERR_ARG;
    if (o->max_seq_len > (1 << 28) || o->batch > (1 << 24)) return SAM_ERR_LIMIT;
    const int64_t n = o->max_seq_len;
    uint32_t slab = o->slab_bytes ? (uint32_t)o->slab_bytes : pow2_ceil((uint64_t)8 * n);
    if (!o->slab_bytes && slab < 16384) slab = 16384;
    if (slab < 4096 || (slab & (slab - 1)) || slab > (1u << 30)) return SAM_ERR_ARG;
    // a slot's state records (at most 2n+1 of 32 bytes) must fit SAM_MAX_REC_SLABS slabs
    if ((uint64_t)(2 * n + 2) * 32 > (uint64_t)slab * SAM_MAX_REC_SLABS) return SAM_ERR_ARG;
    int shift = 0;
    while ((1u << shift) < slab) shift++;
    w->slab_shift = shift;
    int64_t per_slot = ((64 + 96) * n + slab - 1) / slab + 2;
    int64_t slabs = o->pool_slabs ? o->pool_slabs : per_slot * o->batch;
    if (slabs < 2 || slabs > (1ll << 31) - 1 || slabs * (int64_t)slab > (1ll << 38)) return SAM_ERR_LIMIT;
    w->pool_slabs = (int32_t)slabs;
    w->text_stride = (int32_t)sam_align_up((size_t)n, 32);
    // the root has at most one transition per text position: twice that many slots
    uint32_t rc = pow2_ceil((uint64_t)2 * n);
    w->root_cap = rc < 64 ? 64 : (int32_t)rc;             // never fewer than two 32-entry probe windows
    w->max_host_stride = o->max_host_stride ? o->max_host_stride : 32;
    w->stage_words = (size_t)o->batch * ((size_t)w->max_host_stride + 1 + (size_t)o->max_draft_len + 7);

    size_t off = 0;
    w->off_hdr = off;   off = sam_align_up(off + 256, 256);
    w->off_ctrl = off;  off = sam_align_up(off + (size_t)o->batch * SAM_CTRL_WORDS * 4, 256);
    w->off_free = off;  off = sam_align_up(off + (size_t)slabs * 4, 256);
    w->off_owner = off; off = sam_align_up(off + (size_t)slabs * 4, 256);
    w->off_reset = off; off = sam_align_up(off + (size_t)o->batch * 4, 256);
    // two order buffers, the sort keys, two counts; the list of prompts
    w->off_order = off; off += ((size_t)o->batch * 3 + SAM_ORDER_WORDS) * 4;
    if (o->batch >= SAM_ORDER_MIN_BATCH) off += ((size_t)o->batch + 2) * 4;
    off = sam_align_up(off, 256);
    w->off_text = off;  off = sam_align_up(off + (size_t)o->batch * w->text_stride * 4, 256);
    w->off_pstate = off; off = sam_align_up(off + (size_t)o->batch * w->text_stride * 4, 256);
    w->off_root = off;  off = sam_align_up(off + (size_t)o->batch * w->root_cap * 8, 256);
    w->off_stage = off; off = sam_align_up(off + w->stage_words * 4, 256);
    w->off_pool = off;  off = sam_align_up(off + (size_t)slabs * slab, 256);
    w->total = off;
    return SAM_OK;
}

// ---- kernels ----------------------------------------------------------------

constexpr int RESET_THREADS = 128;

__device__ __forceinline__ void clear_slot(const SamBatchView& W, int b) {
    uint32_t* cb = W.ctrl + (size_t)b * SAM_CTRL_WORDS;
    for (int i = threadIdx.x; i < SAM_CTRL_WORDS; i += blockDim.x) cb[i] = 0;
    // (two empty root-table entries per store; the capacity is a multiple of 64)
    uint4* root = reinterpret_cast<uint4*>(W.root_tab + (size_t)b * W.root_cap);
    for (int i = threadIdx.x; i < W.root_cap / 2; i += blockDim.x) root[i] = make_uint4(SAM_NONE, 0, SAM_NONE, 0);
}

// Every slot empty, every slab free: a new batch, or a reset of all of it.  One launch: block b clears slot b, and all
// blocks together rewrite the pool's free stack and owners (nothing of the pool is in use afterwards).
__global__ void __launch_bounds__(RESET_THREADS) init_batch_kernel(SamBatchView W) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
    const size_t i = sam_grid_index(blockIdx.x, blockDim.x, threadIdx.x), stride = sam_grid_size(gridDim.x, blockDim.x);
    for (size_t s = i; s < (size_t)W.pool_slabs; s += stride) {
        W.free_stack[s] = W.pool_slabs - 1 - (int32_t)s;               // slab 0 is handed out first
        W.slab_owner[s] = -1;
    }
    if (threadIdx.x == 0) W.reset_mark[blockIdx.x] = 0;
    if (i == 0) { W.pool_hdr[0] = W.pool_slabs; W.pool_hdr[1] = W.pool_slabs; W.pool_hdr[4] = 0; }
    clear_slot(W, blockIdx.x);
}

// Some slots: clear them and mark them with this reset's number; the second kernel gives the slabs of slots that carry it
// back to the pool.  The slots come with the launch, so nothing is copied and nobody waits.
constexpr int RESET_LIST = 900;                                 // 4 KB of launch arguments hold them
struct ResetList { int32_t slot[RESET_LIST]; };

__global__ void __launch_bounds__(RESET_THREADS) reset_slots_kernel(SamBatchView W, const __grid_constant__ ResetList list, int32_t mark) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
    const int b = list.slot[blockIdx.x];
    clear_slot(W, b);
    if (threadIdx.x == 0) W.reset_mark[b] = mark;
}

__global__ void release_slabs_kernel(SamBatchView W, int32_t mark) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
    const size_t i = sam_grid_index(blockIdx.x, blockDim.x, threadIdx.x), stride = sam_grid_size(gridDim.x, blockDim.x);
    for (size_t s = i; s < (size_t)W.pool_slabs; s += stride) {
        const int owner = W.slab_owner[s];
        if (owner >= 0 && W.reset_mark[owner] == mark) {
            W.slab_owner[s] = -1;
            W.free_stack[atomicAdd(W.pool_hdr, 1)] = (int32_t)s;
        }
    }
}

template <class K, class... Args>
cudaError_t launch_after(K kernel, int blocks, int threads, cudaStream_t s, Args... args) {
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)blocks); cfg.blockDim = dim3((unsigned)threads); cfg.stream = s; cfg.attrs = attr; cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// one warp copies a slot's automaton into flat arrays; of records and edge blocks it reads what lies in the pool, whatever they say
__global__ void dump_kernel(SamBatchView W, int32_t slot, int32_t* hdr, int32_t* length, int32_t* link,
                            int32_t* min_endpos, int32_t* deg, int32_t max_states,
                            int32_t* e_src, int32_t* e_tok, int32_t* e_tgt, int32_t max_edges) {
    const int lane = threadIdx.x;
    const uint32_t* cb = W.ctrl + (size_t)slot * SAM_CTRL_WORDS;
    const int rps_shift = W.slab_shift - 5;
    const size_t slab_bytes = (size_t)1 << W.slab_shift, pool_bytes = (size_t)W.pool_slabs << W.slab_shift;
    const uint32_t most = (uint32_t)SAM_MAX_REC_SLABS << rps_shift;       // (a slab is at most 2^30 bytes)
    const uint32_t n_states = cb[CB_NSTATES] == 0 ? 1 : cb[CB_NSTATES] < most ? cb[CB_NSTATES] : most;
    int64_t n_edges = 0;
    auto put = [&](int64_t k, uint32_t from, uint32_t tok, uint32_t to) {
        if (k < max_edges) { e_src[k] = (int32_t)from; e_tok[k] = (int32_t)tok; e_tgt[k] = (int32_t)(to & SAM_IDMASK); }
    };
    // root: state 0
    if (lane == 0 && max_states > 0) { length[0] = 0; link[0] = -1; min_endpos[0] = 0; deg[0] = (int32_t)cb[CB_ROOTDEG]; }
    const uint2* root = W.root_tab + (size_t)slot * W.root_cap;
    for (int base = 0; base < W.root_cap; base += 32) {
        uint2 e = root[base + lane];
        unsigned has = __ballot_sync(0xFFFFFFFFu, e.x != SAM_NONE);
        if (e.x != SAM_NONE) put(n_edges + __popc(has & ((1u << lane) - 1)), 0, e.x, e.y);
        n_edges += __popc(has);
    }
    for (uint32_t s = 1; s < n_states; s++) {
        const uint32_t slab = cb[CB_SLABTAB + (s >> rps_shift)];
        uint4 a = make_uint4(0, 0, 0, 0), b = a;
        if (slab < (uint32_t)W.pool_slabs) {
            const uint4* rp = reinterpret_cast<const uint4*>(W.pool + ((size_t)slab << W.slab_shift) +
                                                             ((size_t)(s & ((1u << rps_shift) - 1)) << 5));
            a = rp[0]; b = rp[1];
        }
        if (lane == 0 && s < (uint32_t)max_states) {
            length[s] = (int32_t)a.x; link[s] = (int32_t)a.y; min_endpos[s] = (int32_t)a.z; deg[s] = (int32_t)a.w;
        }
        if (a.w <= 2) {
            if (lane == 0 && a.w >= 1) put(n_edges, s, b.x, b.y);
            if (lane == 0 && a.w == 2) put(n_edges + 1, s, b.z, b.w);
            n_edges += a.w;
        } else {
            const size_t at = (size_t)b.x * 128, bytes = (size_t)a.w * 8;
            if (bytes > slab_bytes || at + bytes > pool_bytes) continue;             // no edge block
            const uint2* blk = reinterpret_cast<const uint2*>(W.pool + at);
            for (uint32_t i = lane; i < a.w; i += 32) { const uint2 e = blk[i]; put(n_edges + i, s, e.x, e.y); }
            n_edges += a.w;
        }
    }
    if (lane == 0) { hdr[0] = (int32_t)cb[CB_NTOK]; hdr[1] = (int32_t)n_states; hdr[2] = (int32_t)(n_edges < INT32_MAX ? n_edges : INT32_MAX); }
}

}  // namespace

// ---- helpers for callers that bring their own memory for a short-lived batch ----------------

// Lay a batch with these options out over `base` (device memory of at least *total bytes).
int sam_plan_view(const sam_batch_opts_t* opts, int32_t vocab, void* base, SamBatchView* view,
                  size_t* total, size_t* stage_words) {
    WsLayout w;
    int rc = plan(opts, &w);
    if (rc) return rc;
    if (total) *total = w.total;
    if (stage_words) *stage_words = w.stage_words;
    if (base && view) {
        char* b = (char*)base;
        view->pool_hdr = (int32_t*)(b + w.off_hdr);
        view->ctrl = (uint32_t*)(b + w.off_ctrl);
        view->free_stack = (int32_t*)(b + w.off_free);
        view->slab_owner = (int32_t*)(b + w.off_owner);
        view->reset_mark = (int32_t*)(b + w.off_reset);
        view->order = (int32_t*)(b + w.off_order);
        view->text = (int32_t*)(b + w.off_text);
        view->pstate = (uint32_t*)(b + w.off_pstate);
        view->root_tab = (uint2*)(b + w.off_root);
        view->stage = (int32_t*)(b + w.off_stage);
        view->pool = (unsigned char*)(b + w.off_pool);
        view->batch = opts->batch; view->max_seq_len = opts->max_seq_len; view->text_stride = w.text_stride;
        view->root_cap = w.root_cap; view->slab_shift = w.slab_shift;
        view->l_bias = opts->l_bias; view->min_match = opts->min_match;
        view->vocab = vocab;
        view->pool_slabs = w.pool_slabs;
        view->stop_token = opts->stop_token_plus_one - 1;
    }
    return SAM_OK;
}

// Put every slot of the view into the empty state and fill the slab pool's free stack.
int sam_launch_init(const SamBatchView& V, cudaStream_t s) {
    cudaError_t e = launch_after(init_batch_kernel, V.batch, RESET_THREADS, s, V);
    if (e != cudaSuccess) { sam_set_cuda_error(e); return SAM_ERR_CUDA; }
    return SAM_OK;
}

extern "C" int sam_batch_workspace_bytes(const sam_batch_opts_t* opts, size_t* out) {
    if (!opts || !out) return SAM_ERR_ARG;
    WsLayout w;
    int rc = plan(opts, &w);
    if (rc) return rc;
    *out = w.total;
    return SAM_OK;
}

extern "C" int sam_batch_create(const sam_static_t* st, const sam_batch_opts_t* opts,
                                void* workspace_dev, size_t workspace_bytes, void* stream, sam_batch_t** out) {
    if (!out) return SAM_ERR_ARG;
    *out = nullptr;
    if (!opts || !workspace_dev) return SAM_ERR_ARG;
    if (!st && opts->vocab < 1) return SAM_ERR_ARG;
    WsLayout w;
    int rc = plan(opts, &w);
    if (rc) return rc;
    if (((uintptr_t)workspace_dev & 255) != 0 || workspace_bytes < w.total) return SAM_ERR_WORKSPACE;

    cudaPointerAttributes attr;
    cudaError_t e = cudaPointerGetAttributes(&attr, workspace_dev);
    if (e != cudaSuccess) { sam_set_cuda_error(e); cudaGetLastError(); return SAM_ERR_CUDA; }
    if (attr.type != cudaMemoryTypeDevice) return SAM_ERR_ARG;
    if (st && st->device != attr.device) return SAM_ERR_ARG;

    sam_batch* b = new (std::nothrow) sam_batch();
    if (!b) return SAM_ERR_NOMEM;
    memset(b, 0, sizeof(*b));
    b->device = attr.device;
    b->st = st;
    b->opts = *opts;
    b->workspace_bytes = w.total;
    b->max_host_stride = w.max_host_stride;
    b->stage_words = w.stage_words;
    char* base = (char*)workspace_dev;
    SamBatchView& V = b->view;
    V.pool_hdr = (int32_t*)(base + w.off_hdr);
    V.ctrl = (uint32_t*)(base + w.off_ctrl);
    V.free_stack = (int32_t*)(base + w.off_free);
    V.slab_owner = (int32_t*)(base + w.off_owner);
    V.reset_mark = (int32_t*)(base + w.off_reset);
    V.order = (int32_t*)(base + w.off_order);
    V.text = (int32_t*)(base + w.off_text);
    V.pstate = (uint32_t*)(base + w.off_pstate);
    V.root_tab = (uint2*)(base + w.off_root);
    V.stage = (int32_t*)(base + w.off_stage);
    V.pool = (unsigned char*)(base + w.off_pool);
    V.batch = opts->batch; V.max_seq_len = opts->max_seq_len; V.text_stride = w.text_stride;
    V.root_cap = w.root_cap; V.slab_shift = w.slab_shift;
    V.l_bias = opts->l_bias; V.min_match = opts->min_match;
    V.vocab = st ? st->info.vocab : opts->vocab;
    V.pool_slabs = w.pool_slabs;
    V.stop_token = opts->stop_token_plus_one - 1;

    SamDeviceGuard guard(b->device);
    if (!guard.ok) { delete b; return SAM_ERR_CUDA; }
    // the staging area, the completion flag, and (word, number) pairs for the outputs of a small step
    const size_t per_step = (size_t)opts->batch * ((size_t)opts->max_draft_len + 7);
    const size_t pairs = per_step < SAM_TAGGED_MAX_WORDS ? per_step : SAM_TAGGED_MAX_WORDS;
    const size_t pairs_at = sam_align_up(w.stage_words + 16, 16);
    e = cudaHostAlloc((void**)&b->host_stage, (pairs_at + 2 * pairs) * 4, cudaHostAllocMapped);
    if (e == cudaSuccess) e = cudaHostGetDevicePointer((void**)&b->host_stage_dev, b->host_stage, 0);
    if (e != cudaSuccess) {
        sam_set_cuda_error(e); cudaGetLastError();
        if (b->host_stage) cudaFreeHost(b->host_stage);
        delete b;
        return SAM_ERR_NOMEM;
    }
    b->host_stage[w.stage_words] = 0;
    b->host_tagged = b->host_stage + pairs_at; b->host_tagged_dev = b->host_stage_dev + pairs_at;
    memset(b->host_tagged, 0, 2 * pairs * 4);             // no step has the number 0
    cudaStream_t s = (cudaStream_t)stream;
    if (sam_launch_init(V, s) != SAM_OK) { cudaFreeHost(b->host_stage); delete b; return SAM_ERR_CUDA; }
    *out = b;
    return SAM_OK;
}

extern "C" void sam_batch_destroy(sam_batch_t* b) {
    if (!b) return;
    SamDeviceGuard guard(b->device);
    if (b->host_stage) cudaFreeHost(b->host_stage);
    delete b;
}

extern "C" int sam_batch_reset(sam_batch_t* b, const int32_t* slots_host, int32_t n, void* stream) {
    if (!b) return SAM_ERR_ARG;
    if (!slots_host && n >= 0) return n == 0 ? SAM_OK : SAM_ERR_ARG;
    SamDeviceGuard guard(b->device);
    if (!guard.ok) return SAM_ERR_CUDA;
    cudaStream_t s = (cudaStream_t)stream;
    const SamBatchView& V = b->view;
    if (!slots_host) return sam_launch_init(V, s);
    if (n > V.batch) return SAM_ERR_ARG;
    for (int32_t i = 0; i < n; i++) if (slots_host[i] < 0 || slots_host[i] >= V.batch) return SAM_ERR_ARG;
    if (n == 0) return SAM_OK;
    if (++b->reset_count <= 0) b->reset_count = 1;              // never 0, a slot's mark before its first reset
    for (int32_t at = 0; at < n; at += RESET_LIST) {
        ResetList list;
        const int32_t m = n - at < RESET_LIST ? n - at : RESET_LIST;
        memcpy(list.slot, slots_host + at, (size_t)m * 4);
        SAM_CUDA(launch_after(reset_slots_kernel, m, RESET_THREADS, s, V, list, b->reset_count));
    }
    const int blocks = (V.pool_slabs + 255) / 256;
    SAM_CUDA(launch_after(release_slabs_kernel, blocks < 592 ? blocks : 592, 256, s, V, b->reset_count));
    return SAM_OK;
}

static int check_step_args(const sam_batch* b, const void* toks, int32_t stride, const void* counts, int32_t L,
                           const void* dt, const void* dl, const void* ml, const void* src, const void* status) {
    if (!b || !toks || !counts || !dt || !dl || !ml || !src || !status) return SAM_ERR_ARG;
    if (stride < 1 || L < 1 || L > b->opts.max_draft_len) return SAM_ERR_ARG;
    return SAM_OK;
}

static SamStepIo step_io(const int32_t* new_tokens, int32_t stride, const int32_t* counts, int32_t L, int32_t* draft_tokens,
                         int32_t* draft_len, int32_t* match_len, int32_t* source, int32_t* state, int32_t* status) {
    SamStepIo io{};
    io.new_tokens = new_tokens; io.stride = stride; io.counts = counts; io.L = L;
    io.prompts = stride >= SAM_PREFILL_MIN;
    io.draft_tokens = draft_tokens; io.draft_len = draft_len; io.match_len = match_len; io.source = source; io.state = state; io.status = status;
    return io;
}

extern "C" int sam_step(sam_batch_t* b, const int32_t* new_tokens_dev, int32_t stride,
                        const int32_t* counts_dev, int32_t L,
                        int32_t* draft_tokens_dev, int32_t* draft_len_dev, int32_t* match_len_dev,
                        int32_t* source_dev, int32_t* state_dev, int32_t* status_dev, void* stream) {
    int rc = check_step_args(b, new_tokens_dev, stride, counts_dev, L, draft_tokens_dev, draft_len_dev,
                             match_len_dev, source_dev, status_dev);
    if (rc) return rc;
    return sam_launch_step(b, step_io(new_tokens_dev, stride, counts_dev, L, draft_tokens_dev, draft_len_dev, match_len_dev, source_dev,
                                      state_dev, status_dev), (cudaStream_t)stream);
}

extern "C" int sam_step_verified(sam_batch_t* b, const int32_t* target_tokens_dev, int32_t prev_L,
                                 const int32_t* prev_draft_tokens_dev, const int32_t* prev_draft_len_dev,
                                 const int32_t* max_new_dev, int32_t L,
                                 int32_t* draft_tokens_dev, int32_t* draft_len_dev, int32_t* match_len_dev,
                                 int32_t* source_dev, int32_t* state_dev, int32_t* status_dev,
                                 int32_t* counts_out_dev, int32_t* accepted_out_dev, void* stream) {
    int rc = check_step_args(b, target_tokens_dev, prev_L + 1, prev_draft_len_dev, L, draft_tokens_dev, draft_len_dev,
                             match_len_dev, source_dev, status_dev);
    if (rc) return rc;
    if (!prev_draft_tokens_dev || prev_L < 1 || prev_L > 128) return SAM_ERR_ARG;
    if (prev_draft_tokens_dev == draft_tokens_dev || prev_draft_len_dev == draft_len_dev) return SAM_ERR_ARG;
    SamStepIo io = step_io(target_tokens_dev, prev_L + 1, nullptr, L, draft_tokens_dev, draft_len_dev, match_len_dev, source_dev, state_dev, status_dev);
    io.prompts = false;
    io.v_draft = prev_draft_tokens_dev; io.v_draft_len = prev_draft_len_dev; io.v_max_new = max_new_dev;
    io.v_counts_out = counts_out_dev; io.v_accepted_out = accepted_out_dev;
    return sam_launch_step(b, io, (cudaStream_t)stream);
}

extern "C" int sam_run_steps(sam_batch_t* b, const int32_t* new_tokens_dev, int32_t stride,
                             const int32_t* counts_dev, int32_t n_steps, int32_t L, int32_t out_per_step,
                             int32_t* draft_tokens_dev, int32_t* draft_len_dev, int32_t* match_len_dev,
                             int32_t* source_dev, int32_t* state_dev, int32_t* status_dev, void* stream) {
    int rc = check_step_args(b, new_tokens_dev, stride, counts_dev, L, draft_tokens_dev, draft_len_dev,
                             match_len_dev, source_dev, status_dev);
    if (rc) return rc;
    if (n_steps < 0) return SAM_ERR_ARG;
    if (sam_runs_in_one_launch(stride, n_steps))
        return sam_launch_run(b, new_tokens_dev, stride, counts_dev, n_steps, L, out_per_step != 0, draft_tokens_dev, draft_len_dev,
                              match_len_dev, source_dev, state_dev, status_dev, (cudaStream_t)stream);
    const size_t B = (size_t)b->view.batch;
    for (int32_t s = 0; s < n_steps; s++) {
        const size_t o = out_per_step ? (size_t)s : 0;
        rc = sam_launch_step(b, step_io(new_tokens_dev + (size_t)s * B * stride, stride, counts_dev + (size_t)s * B, L,
                                        draft_tokens_dev + o * B * L, draft_len_dev + o * B, match_len_dev + o * B * 2,
                                        source_dev + o * B, state_dev ? state_dev + o * B * 2 : nullptr, status_dev + o * B),
                             (cudaStream_t)stream);
        if (rc) return rc;
    }
    return SAM_OK;
}

extern "C" int sam_step_host(sam_batch_t* b, const int32_t* new_tokens_host, int32_t stride,
                             const int32_t* counts_host, int32_t L,
                             int32_t* draft_tokens_host, int32_t* draft_len_host, int32_t* match_len_host,
                             int32_t* source_host, int32_t* state_host, int32_t* status_host, void* stream) {
    int rc = check_step_args(b, new_tokens_host, stride, counts_host, L, draft_tokens_host, draft_len_host,
                             match_len_host, source_host, status_host);
    if (rc) return rc;
    if (stride > b->max_host_stride) return SAM_ERR_ARG;
    SamDeviceGuard guard(b->device);
    if (!guard.ok) return SAM_ERR_CUDA;
    cudaStream_t s = (cudaStream_t)stream;
    const size_t B = (size_t)b->view.batch;
    // staging layout (int32 words): inputs [tokens B*stride | counts B], then outputs
    // [draft B*L | draft_len B | match_len 2B | source B | state 2B | status B], or B rows of L + 7 (word, number) pairs
    int32_t* dev = b->view.stage;
    int32_t* hst = b->host_stage;
    const size_t in_words = B * stride + B, out_words = B * L + 7 * B;
    const int32_t seq = ++b->host_seq == 0 ? ++b->host_seq : b->host_seq;
    bool prompts = false;
    for (size_t i = 0; i < B; i++) prompts |= counts_host[i] >= SAM_PREFILL_MIN;
    const bool with_launch = !prompts && sam_step_is_inline(b, stride);
    // The waits below poll: the bytes are there sooner than a stream synchronisation returns.  They are bounded; past the
    // bound (other work queued ahead on the stream, or a failed launch) the stream is synchronised, after which
    // everything has to be there.
    const auto t0 = std::chrono::steady_clock::now();
    uint32_t spin = 0;
    bool synced = false;
    auto not_yet = [&]() -> int {
        if ((++spin & 1023u) != 1023u || std::chrono::steady_clock::now() - t0 < std::chrono::microseconds(SAM_POLL_LIMIT_US)) return SAM_OK;
        if (synced) return SAM_ERR_CUDA;
        SAM_CUDA(cudaStreamSynchronize(s));
        synced = true;
        return SAM_OK;
    };

    if (out_words <= SAM_TAGGED_MAX_WORDS && !prompts) {
        // Small steps: the rows and counts come with the launch, or are read by the kernel from the mapped staging area.  Each
        // output word comes back with the step's number beside it, in one 8-byte store, so no block waits for another or for its
        // stores to host memory: a word whose number is the step's is there.  (A step with prompts takes two launches, and is
        // done when the second is.)
        SamStepIo io = step_io(b->host_stage_dev, stride, b->host_stage_dev + B * stride, L, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr);
        io.from_host = true; io.prompts = false; io.done_seq = seq; io.tagged = b->host_tagged_dev;
        if (with_launch) { io.inline_rows = new_tokens_host; io.inline_counts = counts_host; }
        else {
            memcpy(hst, new_tokens_host, B * stride * 4);
            memcpy(hst + B * stride, counts_host, B * 4);
        }
        rc = sam_launch_step(b, io, s);
        if (rc) return rc;
        const volatile uint64_t* w = reinterpret_cast<const volatile uint64_t*>(b->host_tagged);
        const size_t R = (size_t)L + 7;
        for (size_t i = 0; i < B; i++, w += R) {
            int32_t* draft = draft_tokens_host + i * L;
            int32_t rest[7];
            for (size_t k = 0; k < R; k++) {
                uint64_t v;
                while ((v = w[k]) >> 32 != (uint64_t)(uint32_t)seq) if ((rc = not_yet()) != SAM_OK) return rc;
                if (k < (size_t)L) draft[k] = (int32_t)v; else rest[k - L] = (int32_t)v;
            }
            draft_len_host[i] = rest[0]; match_len_host[2 * i] = rest[1]; match_len_host[2 * i + 1] = rest[2]; source_host[i] = rest[3];
            if (state_host) { state_host[2 * i] = rest[4]; state_host[2 * i + 1] = rest[5]; }
            status_host[i] = rest[6];
        }
        return SAM_OK;
    }

    // Larger steps: the kernel writes to host memory itself, and the last block to finish writes this step's number into the
    // flag word behind the staging area.  Rows and counts come with the launch where they fit, are brought over ahead of it
    // where they are many, and are read by the kernel in between.
    int32_t* flag_dev = b->host_stage_dev + b->stage_words;
    const volatile int32_t* flag = b->host_stage + b->stage_words;
    auto run = [&](const int32_t* rows, const int32_t* cnt, int32_t* d, int32_t* dl, int32_t* ml, int32_t* so, int32_t* st, int32_t* sta,
                   const int32_t* rows_host, const int32_t* cnt_host) -> int {
        SamStepIo io = step_io(rows, stride, cnt, L, d, dl, ml, so, st, sta);
        io.from_host = true; io.prompts = prompts; io.done_flag = flag_dev; io.done_seq = seq;
        if (with_launch) { io.inline_rows = rows_host; io.inline_counts = cnt_host; }
        else if (in_words >= SAM_FETCH_MIN_WORDS) {
            int r = sam_launch_fetch(b, rows, cnt, dev, stride, s);
            if (r) return r;
            io.new_tokens = dev; io.counts = dev + B * stride;
        }
        int r = sam_launch_step(b, io, s);
        if (r) return r;
        while (*flag != seq) if ((r = not_yet()) != SAM_OK) return r;
        std::atomic_thread_fence(std::memory_order_acquire);
        return SAM_OK;
    };
    if ((in_words + out_words) * 4 >= SAM_DIRECT_MIN_BYTES) {
        // Copying the arrays through the staging area on the host costs more than the step.
        // If every array the caller passed is page-locked memory the device can address (cudaHostAlloc /
        // cudaHostRegister: what a pinned torch tensor is), the kernel reads and writes them in place.
        const void* hp[8] = {new_tokens_host, counts_host, draft_tokens_host, draft_len_host, match_len_host,
                             source_host, status_host, state_host};
        void* dp[8] = {nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr};
        bool direct = true;
        for (int i = 0; i < 8 && direct; i++) {
            if (!hp[i]) continue;                              // state_host may be null
            if (cudaHostGetDevicePointer(&dp[i], const_cast<void*>(hp[i]), 0) != cudaSuccess) { cudaGetLastError(); direct = false; }
        }
        if (direct)
            return run((const int32_t*)dp[0], (const int32_t*)dp[1], (int32_t*)dp[2], (int32_t*)dp[3], (int32_t*)dp[4], (int32_t*)dp[5],
                       (int32_t*)dp[7], (int32_t*)dp[6], new_tokens_host, counts_host);
    }
    memcpy(hst, new_tokens_host, B * stride * 4);
    memcpy(hst + B * stride, counts_host, B * 4);
    int32_t* ho = hst + in_words;
    if ((in_words + out_words) * 4 <= SAM_ZERO_COPY_MAX_BYTES) {
        int32_t* zd = b->host_stage_dev;
        int32_t* zo = zd + in_words;
        rc = run(zd, zd + B * stride, zo, zo + B * L, zo + B * L + B, zo + B * L + 3 * B, zo + B * L + 4 * B, zo + B * L + 6 * B, hst, hst + B * stride);
        if (rc) return rc;
    } else {
        SAM_CUDA(cudaMemcpyAsync(dev, hst, in_words * 4, cudaMemcpyHostToDevice, s));
        int32_t* o = dev + in_words;
        SamStepIo io = step_io(dev, stride, dev + B * stride, L, o, o + B * L, o + B * L + B, o + B * L + 3 * B, o + B * L + 4 * B, o + B * L + 6 * B);
        io.prompts = prompts;
        rc = sam_launch_step(b, io, s);
        if (rc) return rc;
        SAM_CUDA(cudaMemcpyAsync(ho, o, out_words * 4, cudaMemcpyDeviceToHost, s));
        SAM_CUDA(cudaStreamSynchronize(s));
    }
    memcpy(draft_tokens_host, ho, B * L * 4);
    memcpy(draft_len_host, ho + B * L, B * 4);
    memcpy(match_len_host, ho + B * L + B, 2 * B * 4);
    memcpy(source_host, ho + B * L + 3 * B, B * 4);
    if (state_host) memcpy(state_host, ho + B * L + 4 * B, 2 * B * 4);
    memcpy(status_host, ho + B * L + 6 * B, B * 4);
    return SAM_OK;
}

extern "C" int sam_batch_launches_per_step(const sam_batch_t* b) {
    if (!b) return SAM_ERR_ARG;
    return sam_step_launch_count(b);
}

extern "C" int sam_batch_pool_info(sam_batch_t* b, int64_t* total_slabs, int64_t* free_slabs, void* stream) {
    if (!b || !total_slabs || !free_slabs) return SAM_ERR_ARG;
    SamDeviceGuard guard(b->device);
    if (!guard.ok) return SAM_ERR_CUDA;
    int32_t hdr[2] = {0, 0};
    SAM_CUDA(cudaMemcpyAsync(hdr, b->view.pool_hdr, 8, cudaMemcpyDeviceToHost, (cudaStream_t)stream));
    SAM_CUDA(cudaStreamSynchronize((cudaStream_t)stream));
    *free_slabs = hdr[0]; *total_slabs = b->view.pool_slabs;
    return SAM_OK;
}

extern "C" int sam_batch_dump(sam_batch_t* b, int32_t slot, int32_t* n_tokens, int32_t* n_states,
                              int32_t* n_edges, int32_t* length, int32_t* link, int32_t* min_endpos,
                              int32_t* deg, int32_t max_states,
                              int32_t* edge_src, int32_t* edge_tok, int32_t* edge_tgt, int32_t max_edges,
                              void* stream) {
    if (!b || slot < 0 || slot >= b->view.batch || max_states < 0 || max_edges < 0) return SAM_ERR_ARG;
    if (max_states > 0 && (!length || !link || !min_endpos || !deg)) return SAM_ERR_ARG;
    if (max_edges > 0 && (!edge_src || !edge_tok || !edge_tgt)) return SAM_ERR_ARG;
    SamDeviceGuard guard(b->device);
    if (!guard.ok) return SAM_ERR_CUDA;
    cudaStream_t s = (cudaStream_t)stream;
    const size_t words = 4 + 4 * (size_t)max_states + 3 * (size_t)max_edges;
    int32_t* dev = nullptr;
    cudaError_t e = cudaMalloc(&dev, words * 4);
    if (e != cudaSuccess) { sam_set_cuda_error(e); cudaGetLastError(); return SAM_ERR_NOMEM; }
    int32_t* d_len = dev + 4; int32_t* d_link = d_len + max_states; int32_t* d_end = d_link + max_states;
    int32_t* d_deg = d_end + max_states; int32_t* d_es = d_deg + max_states; int32_t* d_et = d_es + max_edges;
    int32_t* d_eg = d_et + max_edges;
    dump_kernel<<<1, 32, 0, s>>>(b->view, slot, dev, d_len, d_link, d_end, d_deg, max_states, d_es, d_et, d_eg, max_edges);
    std::vector<int32_t> host;
    try { host.resize(words); } catch (const std::bad_alloc&) { cudaFree(dev); return SAM_ERR_NOMEM; }
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(host.data(), dev, words * 4, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFree(dev);
    if (e != cudaSuccess) { sam_set_cuda_error(e); return SAM_ERR_CUDA; }
    if (n_tokens) *n_tokens = host[0];
    if (n_states) *n_states = host[1];
    if (n_edges) *n_edges = host[2];
    const int32_t ns = host[1] < max_states ? host[1] : max_states;
    const int32_t ne = host[2] < max_edges ? host[2] : max_edges;
    if (ns > 0) {
        memcpy(length, host.data() + 4, (size_t)ns * 4);
        memcpy(link, host.data() + 4 + max_states, (size_t)ns * 4);
        memcpy(min_endpos, host.data() + 4 + 2 * (size_t)max_states, (size_t)ns * 4);
        memcpy(deg, host.data() + 4 + 3 * (size_t)max_states, (size_t)ns * 4);
    }
    if (ne > 0) {
        const int32_t* eb = host.data() + 4 + 4 * (size_t)max_states;
        memcpy(edge_src, eb, (size_t)ne * 4);
        memcpy(edge_tok, eb + max_edges, (size_t)ne * 4);
        memcpy(edge_tgt, eb + 2 * (size_t)max_edges, (size_t)ne * 4);
    }
    return SAM_OK;
}
