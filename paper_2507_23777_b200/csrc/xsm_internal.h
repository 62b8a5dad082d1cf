// Internal declarations shared by the host API (xsm_api.cu) and the kernels.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace xsm {

constexpr int kMaxDraft = 16;                        // size of the histogram rows (n_draft itself is <= 15)
constexpr int kMaxTokens = 128;                      // largest M = batch * (K + 1)
constexpr int kMaxBatch = 128;
constexpr int kMaxDevices = 64;                      // device ordinals the per-device host tables cover
// Every device-side wait is bounded: polls of a word in global memory and mbarrier try_wait calls.
constexpr unsigned kSpinLimit = 1u << 21, kMbarSpinLimit = 1u << 22;
constexpr int kShareLd = 160;                        // shares of a row's sum of squares: [row][kShareLd]

// What a request may change without changing the launch chain (which is recorded once): kept in device memory.
struct RunParams {
    int verify_mode, k_accept, sample_mode, k_sample;
    float delta, temperature;
    uint32_t key0, key1;
    int max_new, prompt_len;
    int call;                      // number of the xsm_generate that runs: what the host is told when it needs no more steps
    // scripted drafts (load generator of the benchmark): null, or [B][script_n] tokens by absolute position; the commit
    // then drafts script tokens, of which the first floor((t+1) a) - floor(t a) are left intact at step t (a = script_acc / 1024)
    const int *script;
    int script_n, script_acc;
};

// Where the keys and values of a token row go: element offset of its row in head 0 of its page (< 0: nowhere), row in the page.
struct __align__(16) RowInfo {
    long long place;
    int rp, pad_;
};

// Everything a kernel needs; passed by value.
struct Dev {
    // shape
    int L, d, H, dh, f, V, C, dc, K, K1, B, M, P;
    int ldv;                       // V rounded up to four: rows of logits are copied in 16-byte pieces
    int max_blocks, n_pages, cpages, max_seq_len, tok_ld;
    int p_shift;                   // log2 of the page size P if that is a power of two, else -1
    int head_kind;
    float eps, scale;
    int bos, eos;
    unsigned spin_limit, mbar_limit;   // bounds of the device-side waits (kSpinLimit, kMbarSpinLimit unless a test shortens them)
    const void *E;                 // embedding table
    const void *gain_first;        // RMSNorm gain that the first stage of a step applies to the embeddings
    // per-sequence state
    int *len, *window, *finished, *n_gen, *n_blocks, *block_table;
    uint32_t *step_idx;
    int *free_stack, *n_free, *n_active, *status;
    unsigned long long *hist, *steps;
    int *tok_log, *step_tokens, *step_n_new;
    const int *prompt;
    RunParams *rp;
    int *host_done;                // host memory: the last xsm_generate that needs no more steps (every sequence has ended, or the status word is raised)
    int *stage_word;               // single stages (inspection): stages of the current step that have run
    // activations: bf16 models as hi and lo planes of Mp rows (layout: xsm_proj.cuh), queries fp16 [2][Mp][d]; fp32 models
    // [row][column]
    int Mp;                        // rows of a plane for a step of the batch
    void *xa_;                     // the residual stream times the gain of the RMSNorm that reads it next
    void *qp_, *aa_, *actp_, *yp_; // queries, attention rows, gated activations, decoding heads' hidden states (a set per head)
    void *hq_, *ha_;               // cross-attention heads: queries, attention rows (a set per head)
    float *ss;                     // [row][kShareLd] shares of the sums of squares of the rows of h
    float *logits0, *hlogits;      // [M][ldv], [K][M][ldv]
    float *h;                      // residual stream [row][d]
    RowInfo *row_info;             // [row]; with row_cs written when the row is embedded, so that nobody else looks up positions and pages
    float2 *row_cs;                // [row][dh/2] cos, sin of the row's position
    float2 *rope_cs;               // [max_seq_len + K + 2][dh/2] cos, sin of position * theta^(-2i/dh)
    // caches
    void *kv_pool;                 // [L][2][n_pages][H] tiles of P x dh
    void *ckv_pool;                // [L][2][B*cpages][H] tiles of P x dh
    void *hckv_pool;               // [K][2][B*cpages][H] tiles: keys and values of the condition under every head's own projections
    unsigned long long *trace;     // null, or [1 + 2 * stages][kTraceCtas] nanosecond timestamps of the step
};

// Prefill and inspection kernels (xsm_kernels.cu).  All return the CUDA error of the launch.
// fp32 models: keys and values of the condition under n_sets projections (offsets into the flat weights W)
cudaError_t launch_cross_kv(const Dev &D, const void *W, const size_t *wkc_off, const size_t *wvc_off,
                            const void *cond, void *pool, int n_sets, cudaStream_t st);
cudaError_t launch_gather_kv(const Dev &D, int dtype, int layer, int seq, int pos0, int n, float *out_k,
                             float *out_v, cudaStream_t st);
cudaError_t launch_export(const Dev &D, int max_new, int *d_tokens, int *d_lengths, cudaStream_t st);

}  // namespace xsm
