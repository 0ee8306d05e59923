// Internal definitions shared by the library's translation units.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include <stddef.h>
#include "layout.h"
#include "../../include/samdraft.h"

struct sam_static {
    int device;
    void* dev_base;               // one allocation holding every section
    size_t dev_bytes;
    size_t off_rec, off_root, off_hash, off_corpus, off_freq, off_topk, off_pstate, off_path;   // section offsets in dev_base
    size_t len_rec, len_root, len_hash, len_corpus, len_freq, len_topk, len_pstate, len_path;   // section sizes in bytes
    SamStaticView view;
    sam_static_info_t info;
};

struct sam_batch {
    int device;
    const sam_static* st;
    sam_batch_opts_t opts;
    SamBatchView view;
    size_t workspace_bytes;
    int32_t max_host_stride;
    size_t stage_words;           // int32 words of device staging
    int32_t* host_stage;          // pinned, device-mapped host staging area
    int32_t* host_stage_dev;      // the same memory as the device addresses it
    int32_t* host_tagged;         // part of it: (word, step number) pairs, and as the device addresses them
    int32_t* host_tagged_dev;
    int32_t host_seq;             // sequence number of the last host-array step (completion flag value)
    int32_t reset_count;          // number of the last reset of some slots
    mutable int32_t order_phase;  // which of the two slot-order buffers the next large-batch step uses
};

void sam_set_cuda_error(cudaError_t e);

#define SAM_CUDA(call)                                          \
    do {                                                        \
        cudaError_t _e = (call);                                \
        if (_e != cudaSuccess) { sam_set_cuda_error(_e); return SAM_ERR_CUDA; } \
    } while (0)

// RAII device switch (nothing is set where the device is the current one already)
struct SamDeviceGuard {
    int prev = -1;
    bool ok = true, switched = false;
    explicit SamDeviceGuard(int dev) {
        if (cudaGetDevice(&prev) != cudaSuccess) { ok = false; return; }
        if (prev != dev) { if (cudaSetDevice(dev) == cudaSuccess) switched = true; else ok = false; }
    }
    ~SamDeviceGuard() { if (switched) cudaSetDevice(prev); }
};

static inline size_t sam_align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// From how many tokens an empty slot's row is a prompt, whose automaton is built at once (step.cu).
constexpr int32_t SAM_PREFILL_MIN = 48;

// From how many slots a step's slots are ordered by their token counts: more than a B200 holds blocks of the step kernel (148 x 10).
constexpr int32_t SAM_ORDER_MIN_BATCH = 1536;

// What one step reads and writes (launchers in step.cu).
struct SamStepIo {
    const int32_t* new_tokens; int32_t stride; const int32_t* counts; int32_t L;
    bool prompts;                 // some counts may be SAM_PREFILL_MIN or more
    int32_t *draft_tokens, *draft_len, *match_len, *source, *state, *status;
    // sam_step_verified
    const int32_t *v_draft, *v_draft_len, *v_max_new;
    int32_t *v_counts_out, *v_accepted_out;
    // sam_step_host: rows and counts to carry with the launch, if any; completion: either the last block writes done_seq to
    // *done_flag, or every output word goes to `tagged` with done_seq beside it
    bool from_host;
    const int32_t *inline_rows, *inline_counts;
    int32_t* done_flag; int32_t done_seq;
    void* tagged;
};
int sam_launch_step(const sam_batch* b, const SamStepIo& io, cudaStream_t stream);
bool sam_step_is_inline(const sam_batch* b, int32_t stride);
// host-mapped rows and counts to device memory, one behind the other
int sam_launch_fetch(const sam_batch* b, const int32_t* rows, const int32_t* counts, int32_t* to, int32_t stride, cudaStream_t stream);

// n_steps steps in one launch (step.cu), and whether they can be
int sam_launch_run(const sam_batch* b, const int32_t* new_tokens, int32_t stride, const int32_t* counts, int32_t n_steps,
                   int32_t L, int32_t keep, int32_t* draft_tokens, int32_t* draft_len, int32_t* match_len,
                   int32_t* source, int32_t* state, int32_t* status, cudaStream_t stream);
bool sam_runs_in_one_launch(int32_t stride, int32_t n_steps);

// 1, or 2 when the batch is large enough for the slot-ordering kernel (step.cu)
int sam_step_launch_count(const sam_batch* b);

// helpers implemented in batch.cu
int sam_plan_view(const sam_batch_opts_t* opts, int32_t vocab, void* base, SamBatchView* view,
                  size_t* total, size_t* stage_words);
int sam_launch_init(const SamBatchView& V, cudaStream_t s);
