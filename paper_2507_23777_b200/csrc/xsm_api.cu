// Host side of the C ABI declared in include/xsm.h: argument checks, workspace layout, requests.  No device memory is allocated here; everything lives in the caller's workspace.
#include "../../include/xsm.h"
#include "xsm_host.h"

#include <limits.h>
#include <math.h>
#include <stdio.h>
#include <string.h>

#include <string>
#include <vector>

using namespace xsm;

namespace {

constexpr int kKvStagePositions = 256;

thread_local std::string g_create_error;

struct Layout {
    size_t total = 0;
    size_t wkc_off, wvc_off, hk_off, hv_off;
    size_t len, window, finished, n_gen, n_blocks, step_idx, block_table, free_stack, scalars, hist, steps, tok_log, step_tokens,
        step_n_new, prompt, script;
    size_t h, rope_cs, row_info, row_cs, logits0, hlogits;
    size_t rp, xa, qp, aa, actp, yp, hq, ha, ss;
    size_t stage_cond, stage_kv, stage_tok, trace, ckv_pool, hckv_pool, kv_pool;
    int n_pages = 0, max_blocks = 0, cpages = 0, tok_ld = 0, n_stages = 0;
    size_t page_bytes = 0;
};

size_t esize(const xsm_model_config &c) { return c.dtype == 1 ? 2 : 4; }

// elements from one row of logits to the next (the tail copies rows in 16-byte pieces)
size_t logits_ld(const xsm_model_config &c) { return ((size_t)c.vocab + 3) / 4 * 4; }

size_t take(size_t &cur, size_t bytes) {
    size_t o = cur;
    cur = (cur + bytes + 255) / 256 * 256;
    return o;
}

// workspace_bytes == 0: size the pool for max_batch full sequences
bool make_layout(const xsm_model_config &c, size_t workspace_bytes, Layout &L) {
    const size_t B = c.max_batch, K1 = c.n_draft + 1, M = B * K1, d = c.d_model, f = c.d_ff;
    const size_t P = c.page_size, H = c.n_heads, dh = c.d_head, ldv = logits_ld(c);
    L.max_blocks = (int)((c.max_seq_len + K1 + P - 1) / P);
    L.cpages = (int)((c.n_cond + P - 1) / P);
    L.tok_ld = c.max_seq_len + (int)K1;
    const bool ca = c.head_kind == 1 && c.n_draft > 0;
    L.n_stages = c.n_layers * 8 + 2 + (c.n_draft > 0 ? 1 : 0) + (ca ? 2 : 0);
    size_t cur = 0;
    L.wkc_off = take(cur, sizeof(size_t) * c.n_layers);
    L.wvc_off = take(cur, sizeof(size_t) * c.n_layers);
    L.hk_off = take(cur, sizeof(size_t) * (c.n_draft + 1));
    L.hv_off = take(cur, sizeof(size_t) * (c.n_draft + 1));
    L.len = take(cur, 4 * B);
    L.window = take(cur, 4 * M);
    L.finished = take(cur, 4 * B);
    L.n_gen = take(cur, 4 * B);
    L.n_blocks = take(cur, 4 * B);
    L.step_idx = take(cur, 4 * B);
    L.block_table = take(cur, 4 * B * L.max_blocks);
    L.scalars = take(cur, 256);   // n_active, status, n_free, stage_word
    L.hist = take(cur, 8 * B * (kMaxDraft + 1));
    L.steps = take(cur, 8 * B);
    L.tok_log = take(cur, 4 * B * L.tok_ld);
    L.step_tokens = take(cur, 4 * M);
    L.step_n_new = take(cur, 4 * B);
    L.prompt = take(cur, 4 * B * (c.max_seq_len + 1));
    L.script = take(cur, 4 * B * L.tok_ld);
    L.rp = take(cur, sizeof(RunParams));
    // activations of a step or of a chunk of a prompt: four bytes an element (bf16 models: hi and lo parts)
    const size_t rows = prompt_rows(c), row = 4 * rows, step_row = 4 * (size_t)kMaxTokens, nh = ca ? (size_t)c.n_draft : 0;
    L.h = take(cur, row * d);
    L.rope_cs = take(cur, 8 * (size_t)(c.max_seq_len + K1 + 1) * (dh / 2));
    L.row_info = take(cur, sizeof(RowInfo) * rows);
    L.row_cs = take(cur, 8 * rows * (dh / 2));
    L.xa = take(cur, row * d);
    L.qp = take(cur, row * d);
    L.aa = take(cur, row * d);
    L.actp = take(cur, row * f);
    L.yp = take(cur, step_row * d * c.n_draft);
    L.hq = take(cur, step_row * d * nh);
    L.ha = take(cur, step_row * d * nh);
    L.ss = take(cur, row * kShareLd);
    // The padding of the logits' rows (25 KB at most) adds nothing to the workspace, so that a size that held a batch of other
    // vocabularies before there was padding still does: the timeline and the gathered keys, neither of which outlasts the call that
    // returns it, share a place (47 and 256 KB at least), and what that leaves over stays unused.
    const size_t heads = c.n_draft > 0 ? c.n_draft : 1, cond = esize(c) * B * c.n_cond * c.d_cond;
    const size_t kv = 4 * 2 * (size_t)kKvStagePositions * d, trace = 8 * (size_t)(1 + 2 * L.n_stages) * kTraceCtas;
    size_t unpadded = cur;
    for (const size_t bytes : {4 * M * c.vocab, 4 * M * c.vocab * heads, cond, kv, 4 * B * (c.max_seq_len + 1), trace}) take(unpadded, bytes);
    L.logits0 = take(cur, 4 * M * ldv);
    L.hlogits = take(cur, 4 * M * ldv * heads);
    L.stage_cond = take(cur, cond);
    L.stage_tok = take(cur, 4 * B * (c.max_seq_len + 1));
    L.stage_kv = L.trace = take(cur, kv > trace ? kv : trace);
    cur = unpadded > cur ? unpadded : cur;
    L.ckv_pool = take(cur, esize(c) * (size_t)c.n_layers * 2 * B * L.cpages * H * P * dh);
    L.hckv_pool = take(cur, esize(c) * nh * 2 * B * L.cpages * H * P * dh);
    L.page_bytes = esize(c) * (size_t)c.n_layers * 2 * H * P * dh;
    // the rest is the shared page pool, preceded by its free stack (4 bytes per page)
    if (workspace_bytes == 0) {
        L.n_pages = (int)(B * L.max_blocks);
    } else {
        if (workspace_bytes <= cur) return false;
        size_t n = (workspace_bytes - cur) / (L.page_bytes + 4);   // upper bound; the stack is 256-byte padded
        if (n > (size_t)INT_MAX / 2) n = INT_MAX / 2;
        while (n > 0) {
            size_t c2 = cur;
            take(c2, 4 * n);
            if (c2 + L.page_bytes * n <= workspace_bytes) break;
            --n;
        }
        if (n < (size_t)L.max_blocks) return false;
        L.n_pages = (int)n;
    }
    L.free_stack = take(cur, 4 * (size_t)L.n_pages);
    L.kv_pool = cur;
    L.total = cur + L.page_bytes * L.n_pages;
    return true;
}

const char *check_config(const xsm_model_config &c) {
    if (c.n_layers < 1 || c.d_model < 32 || c.n_heads < 1 || c.d_head < 2 || c.d_ff < 32 || c.vocab < 2 ||
        c.n_cond < 1 || c.d_cond < 32 || c.max_batch < 1 || c.max_seq_len < 1)
        return "a model dimension is out of range";
    if (c.n_heads * c.d_head != c.d_model) return "n_heads * d_head must equal d_model";
    if (c.d_model % 128 || c.d_ff % 128) return "d_model and d_ff must be multiples of 128";
    if (c.d_cond % 32) return "d_cond must be a multiple of 32";
    if ((long long)(c.d_model > c.d_ff ? c.d_model : c.d_ff) * (c.dtype == 1 ? 2 : 4) > 16384)
        return "d_model and d_ff are limited to 16 KB per weight row (8192 bf16 or 4096 fp32 elements)";
    if ((long long)c.d_model * (c.dtype == 1 ? 2 : 4) > 4096)
        return "d_model is limited to 4 KB per weight row (2048 bf16 or 1024 fp32 elements)";
    if (c.d_head != 32 && c.d_head != 64 && c.d_head != 128) return "d_head must be 32, 64 or 128";
    if (c.n_draft < 0 || c.n_draft >= XSM_MAX_DRAFT) return "n_draft must be in [0, 15]";
    if (c.head_hidden != c.d_model) return "head_hidden must equal d_model (the head block is residual)";
    if (c.head_kind != 0 && c.head_kind != 1) return "head_kind must be 0 (MLP heads) or 1 (cross-attention heads)";
    if (c.dtype != 0 && c.dtype != 1) return "dtype must be 0 (fp32) or 1 (bf16)";
    if (c.page_size < 32 || c.page_size % 32) return "page_size must be a positive multiple of 32";
    if ((long long)c.page_size * c.d_head * (c.dtype == 1 ? 2 : 4) > 16384 * (c.dtype == 1 ? 1 : 4))
        return "page_size * d_head is too large for one cache tile";
    if (c.max_batch > kMaxBatch) return "max_batch exceeds 128";
    if ((long long)c.max_batch * (c.n_draft + 1) > kMaxTokens) return "max_batch * (n_draft + 1) exceeds 128";
    if (c.vocab > (1 << 20)) return "vocab too large";
    if (!(c.rope_theta > 1.0f) || !(c.rms_eps > 0.0f)) return "rope_theta must be > 1 and rms_eps > 0";
    if (c.bos_id < 0 || c.bos_id >= c.vocab || c.eos_id >= c.vocab) return "bos_id / eos_id out of range";
    return nullptr;
}

WeightOffsets weight_offsets(const xsm_model_config &c) {
    WeightOffsets w;
    const size_t d = c.d_model, f = c.d_ff, V = c.vocab, dc = c.d_cond, hd = c.head_hidden;
    size_t o = 0;
    w.E = o; o += V * d;
    for (int l = 0; l < c.n_layers; ++l) {
        w.g1.push_back(o); o += d;
        w.wq.push_back(o); o += 3 * d * d;      // Wq, Wk, Wv are consecutive
        w.wo.push_back(o); o += d * d;
        w.g2.push_back(o); o += d;
        w.wqc.push_back(o); o += d * d;
        w.wkc.push_back(o); o += d * dc;
        w.wvc.push_back(o); o += d * dc;
        w.woc.push_back(o); o += d * d;
        w.g3.push_back(o); o += d;
        w.wgate.push_back(o); o += f * d;
        w.wup.push_back(o); o += f * d;
        w.wdown.push_back(o); o += d * f;
    }
    w.gf = o; o += d;
    w.W0 = o; o += V * d;
    for (int i = 0; i < c.n_draft; ++i) {
        if (c.head_kind == 1) {          // cross-attention head (Eq. 3): Wq, Wk, Wv, Wo of its own, then W(i)
            w.hq.push_back(o); o += d * d;
            w.hk.push_back(o); o += d * dc;
            w.hv.push_back(o); o += d * dc;
            w.ho.push_back(o); o += d * d;
            w.Wout.push_back(o); o += V * d;
        } else {
            w.W1.push_back(o); o += hd * d;
            w.Wout.push_back(o); o += V * hd;
        }
    }
    w.total = o;
    return w;
}

// what the launch chain goes by
void set_shape(Dev &D, const xsm_model_config &c, const Layout &L) {
    D.L = c.n_layers; D.d = c.d_model; D.H = c.n_heads; D.dh = c.d_head; D.f = c.d_ff;
    D.V = c.vocab; D.ldv = (int)logits_ld(c); D.C = c.n_cond; D.dc = c.d_cond; D.K = c.n_draft; D.K1 = c.n_draft + 1;
    D.P = c.page_size; D.max_blocks = L.max_blocks; D.n_pages = L.n_pages; D.cpages = L.cpages;
    D.head_kind = c.head_kind;
    D.scale = (float)(1.0 / sqrt((double)c.d_head));
}
void set_batch(Dev &D, int batch) { D.B = batch; D.M = batch * D.K1; D.Mp = (D.M + 7) / 8 * 8; }

}  // namespace

struct xsm_ctx {
    xsm_model_config cfg;
    Layout lay;
    WeightOffsets wo;
    const char *weights;
    char *ws;
    cudaStream_t stream;
    Dev dev;
    int sm_count, phase_launch, prefilled, n_stages;
    unsigned long long launches;
    std::string err;
    Chain chain;              // the kernels of a decoding step
    bool limited;             // the token limit of an xsm_generate may be in device memory
    int generate_call;        // number of the latest xsm_generate
    int *pinned;              // [16] n_active and status; at 8: the last xsm_generate that needs no more steps
    cudaEvent_t ev0, ev1, step_ev[2];
};

namespace {

xsm_status fail(xsm_ctx *ctx, xsm_status st, const std::string &msg) {
    if (ctx) ctx->err = msg; else g_create_error = msg;
    return st;
}
xsm_status cuda_fail(xsm_ctx *ctx, cudaError_t e, const char *what) {
    (void)cudaGetLastError();      // reported here: the next call starts clean
    return fail(ctx, XSM_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
}
#define XSM_CUDA(ctx, call)                                             \
    do {                                                                \
        cudaError_t e_ = (call);                                        \
        if (e_ != cudaSuccess) return cuda_fail(ctx, e_, #call);        \
    } while (0)

template <typename T> T *at(xsm_ctx *ctx, size_t off) { return reinterpret_cast<T *>(ctx->ws + off); }
const void *wptr(const xsm_ctx *ctx, size_t elem_off) { return ctx->weights + elem_off * esize(ctx->cfg); }

xsm_status check_device_status(xsm_ctx *ctx) {
    XSM_CUDA(ctx, cudaMemcpyAsync(ctx->pinned, ctx->dev.n_active, 8, cudaMemcpyDeviceToHost, ctx->stream));
    XSM_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    const int st = ctx->pinned[1];
    if (st == XSM_ERR_TIMEOUT) return fail(ctx, XSM_ERR_TIMEOUT, "a bounded device-side wait ran out of patience");
    if (st == XSM_ERR_CAPACITY) return fail(ctx, XSM_ERR_CAPACITY, "the page pool ran dry during decoding");
    if (st != 0) return fail(ctx, XSM_ERR_CUDA, "device status word is set");
    return XSM_OK;
}

// one decoding step on the stream
xsm_status run_step(xsm_ctx *ctx, bool may_record = true) {
    // a recording is replayed unless single launches were asked for, a timeline is taken (the recording has none), or the
    // call must not make the driver allocate anything
    const bool graph = !ctx->phase_launch && may_record && ctx->dev.trace == nullptr;
    XSM_CUDA(ctx, ctx->chain.step(ctx->dev, ctx->stream, graph, !ctx->phase_launch, &ctx->launches));
    return XSM_OK;
}

// does the stream record into a graph of the caller's, so that what is launched does not run now, but at every replay?
xsm_status is_captured(xsm_ctx *ctx, bool *yes) {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    XSM_CUDA(ctx, cudaStreamIsCapturing(ctx->stream, &cs));
    *yes = cs != cudaStreamCaptureStatusNone;
    return XSM_OK;
}
// A step on its own has no token limit: one that xsm_generate has stored is taken back, unless xsm_prefill has done so.  A
// captured step takes it back at every replay, since nothing is known of what will have run before.
xsm_status lift_limit(xsm_ctx *ctx) {
    bool captured = false;
    const xsm_status st = is_captured(ctx, &captured);
    if (st != XSM_OK || (!captured && !ctx->limited)) return st;
    XSM_CUDA(ctx, launch_set_limit(ctx->dev, INT_MAX, 0, ctx->stream));
    ctx->launches += 1;
    if (!captured) ctx->limited = false;
    return XSM_OK;
}
// the tokens committed by the latest step -> the caller
xsm_status copy_step(xsm_ctx *ctx, int32_t *d_new_tokens, int32_t *d_n_new) {
    const Dev &D = ctx->dev;
    if (d_new_tokens)
        XSM_CUDA(ctx, cudaMemcpyAsync(d_new_tokens, D.step_tokens, sizeof(int32_t) * D.M, cudaMemcpyDeviceToDevice, ctx->stream));
    if (d_n_new)
        XSM_CUDA(ctx, cudaMemcpyAsync(d_n_new, D.step_n_new, sizeof(int32_t) * D.B, cudaMemcpyDeviceToDevice, ctx->stream));
    return XSM_OK;
}

}  // namespace

extern "C" {

size_t xsm_weights_bytes(const xsm_model_config *cfg) {
    if (!cfg || check_config(*cfg)) return 0;
    return weight_offsets(*cfg).total * esize(*cfg);
}

size_t xsm_workspace_bytes(const xsm_model_config *cfg) {
    if (!cfg || check_config(*cfg)) return 0;
    Layout L;
    make_layout(*cfg, 0, L);
    return L.total;
}

xsm_status xsm_create(const xsm_model_config *cfg, const void *d_weights, void *d_workspace, size_t workspace_bytes,
                      void *cuda_stream, xsm_ctx **out) {
    if (!cfg || !d_weights || !d_workspace || !out) return fail(nullptr, XSM_ERR_INVALID_ARG, "null argument");
    if (const char *m = check_config(*cfg)) return fail(nullptr, XSM_ERR_INVALID_ARG, m);
    if (((uintptr_t)d_weights & 255) || ((uintptr_t)d_workspace & 255))
        return fail(nullptr, XSM_ERR_INVALID_ARG, "weights and workspace must be 256-byte aligned");
    Layout L;
    if (!make_layout(*cfg, workspace_bytes, L))
        return fail(nullptr, XSM_ERR_CAPACITY, "workspace cannot hold the buffers plus one sequence of cache pages");
    xsm_ctx *ctx = new xsm_ctx();
    ctx->cfg = *cfg;
    ctx->lay = L;
    ctx->wo = weight_offsets(*cfg);
    ctx->weights = (const char *)d_weights;
    ctx->ws = (char *)d_workspace;
    ctx->stream = (cudaStream_t)cuda_stream;
    ctx->phase_launch = 0; ctx->prefilled = 0; ctx->launches = 0; ctx->generate_call = 0; ctx->n_stages = 0;
    ctx->limited = true;
    ctx->pinned = nullptr; ctx->ev0 = ctx->ev1 = ctx->step_ev[0] = ctx->step_ev[1] = nullptr;
    auto bail = [&](cudaError_t e, const char *what) {
        g_create_error = std::string(what) + ": " + cudaGetErrorString(e);
        if (ctx->pinned) cudaFreeHost(ctx->pinned);
        if (ctx->ev0) cudaEventDestroy(ctx->ev0);
        if (ctx->ev1) cudaEventDestroy(ctx->ev1);
        for (cudaEvent_t ev : ctx->step_ev)
            if (ev) cudaEventDestroy(ev);
        delete ctx;
        return XSM_ERR_CUDA;
    };
    cudaError_t e;
    {
        int dev = 0;
        if ((e = cudaGetDevice(&dev)) != cudaSuccess) return bail(e, "cudaGetDevice");
        if ((e = cudaDeviceGetAttribute(&ctx->sm_count, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return bail(e, "device query");
    }
    if ((e = cudaHostAlloc((void **)&ctx->pinned, 64, cudaHostAllocDefault)) != cudaSuccess) return bail(e, "cudaHostAlloc");
    if (!ctx->chain.init(*cfg, ctx->wo, ctx->weights, ctx->sm_count)) return bail(cudaErrorNotSupported, "tensor maps of the weights");
    if ((e = cudaEventCreate(&ctx->ev0)) != cudaSuccess) return bail(e, "cudaEventCreate");
    if ((e = cudaEventCreate(&ctx->ev1)) != cudaSuccess) return bail(e, "cudaEventCreate");
    for (cudaEvent_t &ev : ctx->step_ev)
        if ((e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming)) != cudaSuccess) return bail(e, "cudaEventCreate");
    memset(ctx->pinned, 0, 64);

    // The state starts at zero as well: a step behind a prefill that was captured and has not run yet finds positions, pages and
    // tokens that exist, and ends in XSM_ERR_CAPACITY (the pool is empty).
    if ((e = cudaMemsetAsync(ctx->ws + L.len, 0, L.xa - L.len, ctx->stream)) != cudaSuccess) return bail(e, "memset");

    // constant tables
    // cos and sin of position * theta^(-2i/dh) for every position a window row can take
    const int half = cfg->d_head / 2, n_pos = cfg->max_seq_len + cfg->n_draft + 2;
    std::vector<float> rope((size_t)n_pos * half * 2);
    for (int i = 0; i < half; ++i) {
        const double inv_freq = pow((double)cfg->rope_theta, -2.0 * i / cfg->d_head);
        for (int p = 0; p < n_pos; ++p) {
            rope[((size_t)p * half + i) * 2] = (float)cos((double)p * inv_freq);
            rope[((size_t)p * half + i) * 2 + 1] = (float)sin((double)p * inv_freq);
        }
    }
    if ((e = cudaMemcpyAsync(ctx->ws + L.rope_cs, rope.data(), sizeof(float) * rope.size(),
                             cudaMemcpyHostToDevice, ctx->stream)) != cudaSuccess) return bail(e, "upload");
    if ((e = cudaMemcpyAsync(ctx->ws + L.wkc_off, ctx->wo.wkc.data(), sizeof(size_t) * cfg->n_layers,
                             cudaMemcpyHostToDevice, ctx->stream)) != cudaSuccess) return bail(e, "upload");
    if ((e = cudaMemcpyAsync(ctx->ws + L.wvc_off, ctx->wo.wvc.data(), sizeof(size_t) * cfg->n_layers,
                             cudaMemcpyHostToDevice, ctx->stream)) != cudaSuccess) return bail(e, "upload");
    if (cfg->head_kind == 1 && cfg->n_draft > 0) {
        if ((e = cudaMemcpyAsync(ctx->ws + L.hk_off, ctx->wo.hk.data(), sizeof(size_t) * cfg->n_draft, cudaMemcpyHostToDevice,
                                 ctx->stream)) != cudaSuccess) return bail(e, "upload");
        if ((e = cudaMemcpyAsync(ctx->ws + L.hv_off, ctx->wo.hv.data(), sizeof(size_t) * cfg->n_draft, cudaMemcpyHostToDevice,
                                 ctx->stream)) != cudaSuccess) return bail(e, "upload");
    }
    // the caches start at zero: slots that were never written are multiplied by zero weights and must be finite
    if ((e = cudaMemsetAsync(ctx->ws + L.ckv_pool, 0, L.total - L.ckv_pool, ctx->stream)) != cudaSuccess) return bail(e, "memset");
    if ((e = cudaStreamSynchronize(ctx->stream)) != cudaSuccess) return bail(e, "sync");

    Dev &D = ctx->dev;
    memset(&D, 0, sizeof(D));
    set_shape(D, *cfg, L);
    D.p_shift = -1;
    for (int sh = 0; sh < 30; ++sh)
        if ((1 << sh) == cfg->page_size) D.p_shift = sh;
    D.max_seq_len = cfg->max_seq_len; D.tok_ld = L.tok_ld;
    D.eps = cfg->rms_eps; D.bos = cfg->bos_id; D.eos = cfg->eos_id;
    D.spin_limit = kSpinLimit; D.mbar_limit = kMbarSpinLimit;
    D.E = wptr(ctx, ctx->wo.E); D.gain_first = wptr(ctx, ctx->wo.g1[0]);
    D.len = at<int>(ctx, L.len); D.window = at<int>(ctx, L.window);
    D.finished = at<int>(ctx, L.finished); D.n_gen = at<int>(ctx, L.n_gen);
    D.n_blocks = at<int>(ctx, L.n_blocks); D.block_table = at<int>(ctx, L.block_table);
    D.step_idx = at<uint32_t>(ctx, L.step_idx);
    D.free_stack = at<int>(ctx, L.free_stack);
    int *sc = at<int>(ctx, L.scalars);
    D.n_active = sc; D.status = sc + 1; D.n_free = sc + 2; D.stage_word = sc + 3;
    D.hist = at<unsigned long long>(ctx, L.hist); D.steps = at<unsigned long long>(ctx, L.steps);
    D.tok_log = at<int>(ctx, L.tok_log); D.step_tokens = at<int>(ctx, L.step_tokens);
    D.step_n_new = at<int>(ctx, L.step_n_new); D.prompt = at<int>(ctx, L.prompt);
    D.rp = at<RunParams>(ctx, L.rp);
    D.host_done = ctx->pinned + 8;
    D.h = at<float>(ctx, L.h); D.rope_cs = at<float2>(ctx, L.rope_cs);
    D.row_info = at<RowInfo>(ctx, L.row_info); D.row_cs = at<float2>(ctx, L.row_cs);
    D.xa_ = ctx->ws + L.xa; D.qp_ = ctx->ws + L.qp; D.aa_ = ctx->ws + L.aa; D.actp_ = ctx->ws + L.actp;
    D.yp_ = ctx->ws + L.yp; D.hq_ = ctx->ws + L.hq; D.ha_ = ctx->ws + L.ha; D.ss = at<float>(ctx, L.ss);
    D.logits0 = at<float>(ctx, L.logits0); D.hlogits = at<float>(ctx, L.hlogits);
    D.kv_pool = ctx->ws + L.kv_pool; D.ckv_pool = ctx->ws + L.ckv_pool; D.hckv_pool = ctx->ws + L.hckv_pool;
    *out = ctx;
    return XSM_OK;
}

xsm_status xsm_prefill(xsm_ctx *ctx, int batch, const void *d_cond, const int32_t *d_prompt, int prompt_len,
                       const xsm_decode_config *dc) {
    if (!ctx) return XSM_ERR_INVALID_ARG;
    if (!d_cond || !d_prompt || !dc) return fail(ctx, XSM_ERR_INVALID_ARG, "null argument");
    const xsm_model_config &c = ctx->cfg;
    if (batch < 1 || batch > c.max_batch) return fail(ctx, XSM_ERR_INVALID_ARG, "batch must be in [1, max_batch]");
    if (prompt_len < 1 || prompt_len - 1 > c.max_seq_len) return fail(ctx, XSM_ERR_INVALID_ARG, "prompt_len out of range");
    if (dc->verify_mode < 0 || dc->verify_mode > 2 || dc->sample_mode < 0 || dc->sample_mode > 2)
        return fail(ctx, XSM_ERR_INVALID_ARG, "unknown verify_mode or sample_mode");
    if (dc->verify_mode == 1 && dc->k_accept < 1) return fail(ctx, XSM_ERR_INVALID_ARG, "k_accept must be >= 1");
    if (dc->sample_mode == 1 && (dc->k_sample < 1 || dc->k_sample > 64 || !(dc->temperature > 0.f)))
        return fail(ctx, XSM_ERR_INVALID_ARG, "k_sample must be in [1, 64] and temperature > 0");
    if (dc->sample_mode == 2) {
        if (dc->k_sample < 1 || dc->k_sample > 8 || !(dc->temperature > 0.f))
            return fail(ctx, XSM_ERR_INVALID_ARG, "probability-tree sampling: k_sample must be in [1, 8] and temperature > 0");
        double leaves = 1.0;
        for (int i = 0; i < c.n_draft; ++i) leaves *= dc->k_sample;
        if (leaves > 4096.0) return fail(ctx, XSM_ERR_INVALID_ARG, "probability-tree sampling: k_sample ^ n_draft must not exceed 4096 paths");
    }
    if ((long long)batch * ctx->lay.max_blocks > ctx->lay.n_pages)
        return fail(ctx, XSM_ERR_CAPACITY, "the page pool cannot hold `batch` sequences of max_seq_len positions");
    bool captured = false;
    const xsm_status capture = is_captured(ctx, &captured);
    if (capture != XSM_OK) return capture;
    Dev &D = ctx->dev;
    if (c.dtype == 0 && batch * D.K1 > kF32Rows) return fail(ctx, XSM_ERR_CAPACITY, "fp32 models support at most 24 token rows per step");
    set_batch(D, batch);
    if (!ctx->chain.select(D)) return fail(ctx, XSM_ERR_CUDA, "the tensor maps of the step could not be made");
    ctx->n_stages = ctx->chain.n_ops();
    RunParams r;
    memset(&r, 0, sizeof(r));
    r.verify_mode = dc->verify_mode; r.k_accept = dc->k_accept; r.delta = dc->delta;
    r.sample_mode = dc->sample_mode; r.k_sample = dc->k_sample; r.temperature = dc->temperature;
    r.key0 = (uint32_t)dc->seed; r.key1 = (uint32_t)(dc->seed >> 32);
    r.max_new = INT_MAX; r.prompt_len = prompt_len;
    if ((const void *)d_prompt != (const void *)D.prompt)
        XSM_CUDA(ctx, cudaMemcpyAsync((void *)D.prompt, d_prompt, sizeof(int32_t) * batch * prompt_len, cudaMemcpyDeviceToDevice, ctx->stream));
    XSM_CUDA(ctx, launch_begin(D, r, ctx->stream));
    ctx->launches += 2;
    if (!captured) ctx->limited = false;
    if (c.dtype == 1) {
        XSM_CUDA(ctx, ctx->chain.condition(D, d_cond, ctx->stream, &ctx->launches));
    } else {
        XSM_CUDA(ctx, launch_cross_kv(D, ctx->weights, at<size_t>(ctx, ctx->lay.wkc_off), at<size_t>(ctx, ctx->lay.wvc_off), d_cond,
                                      D.ckv_pool, D.L, ctx->stream));
        ctx->launches += 1;
        if (c.head_kind == 1 && D.K > 0) {
            XSM_CUDA(ctx, launch_cross_kv(D, ctx->weights, at<size_t>(ctx, ctx->lay.hk_off), at<size_t>(ctx, ctx->lay.hv_off), d_cond,
                                          D.hckv_pool, D.K, ctx->stream));
            ctx->launches += 1;
        }
    }
    if (prompt_len > 1) XSM_CUDA(ctx, ctx->chain.ingest(D, prompt_len - 1, ctx->stream, &ctx->launches));
    XSM_CUDA(ctx, launch_embed_rows(D, c.dtype, D.K1, -1, 0, ChainLaunch{ctx->stream, false, &ctx->launches}));
    ctx->prefilled = 1;
    return XSM_OK;
}

xsm_status xsm_spec_step(xsm_ctx *ctx, int32_t *d_new_tokens, int32_t *d_n_new) {
    if (!ctx) return XSM_ERR_INVALID_ARG;
    if (!ctx->prefilled) return fail(ctx, XSM_ERR_STATE, "xsm_spec_step before xsm_prefill");
    xsm_status st = lift_limit(ctx);
    if (st == XSM_OK) st = run_step(ctx);
    return st == XSM_OK ? copy_step(ctx, d_new_tokens, d_n_new) : st;
}

// The partial results of the key splits travel within clusters and need no memory; the call keeps the limit that it had when
// they lay in an array of the library.
constexpr size_t kStaticScratchBytes = (size_t)1 << 20;

xsm_status xsm_spec_step_static(xsm_ctx *ctx, int32_t *d_new_tokens, int32_t *d_n_new) {
    if (!ctx) return XSM_ERR_INVALID_ARG;
    if (!ctx->prefilled) return fail(ctx, XSM_ERR_STATE, "xsm_spec_step_static before xsm_prefill");
    const Dev &D = ctx->dev;
    // the partial results of the key splits of self- and cross-attention: [batch * n_heads * splits][K + 1][d_head + 2] floats
    // each, with as many splits as leave an SM for each (one stage's at a time are in use); cross-attention heads count K more
    const int splits = ctx->sm_count / (D.B * D.H);
    const size_t one = (size_t)D.B * D.H * (splits < 1 ? 1 : splits > 64 ? 64 : splits) * D.K1 * (D.dh + 2) * sizeof(float);
    const size_t half = (one + 255) / 256 * 256;
    const size_t n_sets = 2 + (D.head_kind == 1 ? (size_t)D.K : 0);
    if (n_sets * half > kStaticScratchBytes)
        return fail(ctx, XSM_ERR_CAPACITY, "xsm_spec_step_static: the attention partials of this batch would need " +
                                               std::to_string(n_sets * half) + " bytes of scratch, more than " +
                                               std::to_string(kStaticScratchBytes));
    xsm_status st = lift_limit(ctx);
    if (st == XSM_OK) st = run_step(ctx, false);
    return st == XSM_OK ? copy_step(ctx, d_new_tokens, d_n_new) : st;
}

xsm_status xsm_generate(xsm_ctx *ctx, int max_new_tokens, int32_t *d_tokens, int32_t *d_lengths, xsm_stats *host_stats) {
    if (!ctx) return XSM_ERR_INVALID_ARG;
    if (!ctx->prefilled) return fail(ctx, XSM_ERR_STATE, "xsm_generate before xsm_prefill");
    if (max_new_tokens < 1 || max_new_tokens > ctx->cfg.max_seq_len)
        return fail(ctx, XSM_ERR_INVALID_ARG, "max_new_tokens must be in [1, max_seq_len]");
    Dev &D = ctx->dev;
    // Stored anew by every call, under a number of its own: a prefill that the caller has captured begins the same request
    // whenever it is replayed, without this code's knowledge.
    const int call = ++ctx->generate_call;
    ctx->limited = true;
    XSM_CUDA(ctx, launch_set_limit(D, max_new_tokens, call, ctx->stream));
    ctx->launches += 1;
    XSM_CUDA(ctx, cudaEventRecord(ctx->ev0, ctx->stream));
    // One step ahead of the device: the next is on its way while one runs, and the one too many at the end finds every
    // sequence ended and does nothing.  Every step commits at least one token per live sequence.  A step that finds the status
    // word raised ends the loop too: the rest would be void, and each might wait out its limits again.
    volatile int *const done = ctx->pinned + 8;
    for (long long i = 0; i < (long long)max_new_tokens + 2 && *done != call; ++i) {
        xsm_status st = run_step(ctx);
        if (st != XSM_OK) return st;
        XSM_CUDA(ctx, cudaEventRecord(ctx->step_ev[i & 1], ctx->stream));
        if (i > 0) XSM_CUDA(ctx, cudaEventSynchronize(ctx->step_ev[(i - 1) & 1]));
    }
    XSM_CUDA(ctx, cudaEventRecord(ctx->ev1, ctx->stream));
    if (d_tokens || d_lengths) {
        XSM_CUDA(ctx, launch_export(D, max_new_tokens, d_tokens, d_lengths, ctx->stream));
        ctx->launches += 1;
    }
    const xsm_status end = check_device_status(ctx);      // waits for the stream
    if (end != XSM_OK) return end;
    float ms = 0.f;
    XSM_CUDA(ctx, cudaEventElapsedTime(&ms, ctx->ev0, ctx->ev1));
    if (host_stats) {
        std::vector<unsigned long long> hist((size_t)D.B * (kMaxDraft + 1)), steps(D.B);
        std::vector<int> ngen(D.B);
        XSM_CUDA(ctx, cudaMemcpy(hist.data(), D.hist, 8 * hist.size(), cudaMemcpyDeviceToHost));
        XSM_CUDA(ctx, cudaMemcpy(steps.data(), D.steps, 8 * steps.size(), cudaMemcpyDeviceToHost));
        XSM_CUDA(ctx, cudaMemcpy(ngen.data(), D.n_gen, 4 * ngen.size(), cudaMemcpyDeviceToHost));
        memset(host_stats, 0, sizeof(*host_stats));
        for (int b = 0; b < D.B; ++b) {
            host_stats->steps += steps[b];
            host_stats->tokens += (uint64_t)ngen[b];
            for (int a = 0; a <= kMaxDraft; ++a) host_stats->accept_hist[a] += hist[(size_t)b * (kMaxDraft + 1) + a];
        }
        host_stats->wall_ms = ms;
        host_stats->scr = host_stats->steps ? (double)host_stats->tokens / (double)host_stats->steps : 0.0;
    }
    return XSM_OK;
}

xsm_status xsm_generate_host(xsm_ctx *ctx, int batch, const void *h_cond, const int32_t *h_prompt, int prompt_len,
                             const xsm_decode_config *dc, int max_new_tokens, int32_t *h_tokens, int32_t *h_lengths,
                             xsm_stats *host_stats) {
    if (!ctx) return XSM_ERR_INVALID_ARG;
    if (!h_cond || !h_prompt || !dc || !h_tokens || !h_lengths) return fail(ctx, XSM_ERR_INVALID_ARG, "null argument");
    const xsm_model_config &c = ctx->cfg;
    if (batch < 1 || batch > c.max_batch) return fail(ctx, XSM_ERR_INVALID_ARG, "batch must be in [1, max_batch]");
    if (prompt_len < 1 || prompt_len - 1 > c.max_seq_len) return fail(ctx, XSM_ERR_INVALID_ARG, "prompt_len out of range");
    if (max_new_tokens < 1 || max_new_tokens > c.max_seq_len)
        return fail(ctx, XSM_ERR_INVALID_ARG, "max_new_tokens must be in [1, max_seq_len]");
    void *d_cond = ctx->ws + ctx->lay.stage_cond;
    int32_t *d_prompt = at<int32_t>(ctx, ctx->lay.prompt);
    int32_t *d_tok = at<int32_t>(ctx, ctx->lay.stage_tok);
    XSM_CUDA(ctx, cudaMemcpyAsync(d_cond, h_cond, esize(c) * (size_t)batch * c.n_cond * c.d_cond, cudaMemcpyHostToDevice, ctx->stream));
    XSM_CUDA(ctx, cudaMemcpyAsync(d_prompt, h_prompt, sizeof(int32_t) * (size_t)batch * prompt_len, cudaMemcpyHostToDevice, ctx->stream));
    xsm_status st = xsm_prefill(ctx, batch, d_cond, d_prompt, prompt_len, dc);
    if (st != XSM_OK) return st;
    // lengths are staged behind the tokens
    int32_t *d_len = at<int32_t>(ctx, ctx->lay.step_n_new);
    st = xsm_generate(ctx, max_new_tokens, d_tok, d_len, host_stats);
    if (st != XSM_OK) return st;
    XSM_CUDA(ctx, cudaMemcpyAsync(h_tokens, d_tok, sizeof(int32_t) * (size_t)batch * max_new_tokens, cudaMemcpyDeviceToHost, ctx->stream));
    XSM_CUDA(ctx, cudaMemcpyAsync(h_lengths, d_len, sizeof(int32_t) * batch, cudaMemcpyDeviceToHost, ctx->stream));
    XSM_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    return XSM_OK;
}

xsm_status xsm_destroy(xsm_ctx *ctx) {
    if (!ctx) return XSM_ERR_INVALID_ARG;
    cudaStreamSynchronize(ctx->stream);
    if (ctx->pinned) cudaFreeHost(ctx->pinned);
    if (ctx->ev0) cudaEventDestroy(ctx->ev0);
    if (ctx->ev1) cudaEventDestroy(ctx->ev1);
    for (cudaEvent_t ev : ctx->step_ev)
        if (ev) cudaEventDestroy(ev);
    delete ctx;
    return XSM_OK;
}

const char *xsm_last_error(const xsm_ctx *ctx) { return ctx ? ctx->err.c_str() : g_create_error.c_str(); }

uint64_t xsm_kernel_launches(const xsm_ctx *ctx) { return ctx ? ctx->launches : 0; }

xsm_status xsm_debug_get_logits(xsm_ctx *ctx, float *h_logits0, float *h_head_logits) {
    if (!ctx) return XSM_ERR_INVALID_ARG;
    if (!ctx->prefilled) return fail(ctx, XSM_ERR_STATE, "no step has run");
    const Dev &D = ctx->dev;
    xsm_status st = check_device_status(ctx);
    if (st != XSM_OK) return st;
    if (h_logits0)
        XSM_CUDA(ctx, cudaMemcpy2D(h_logits0, sizeof(float) * D.V, D.logits0, sizeof(float) * D.ldv, sizeof(float) * D.V, D.M, cudaMemcpyDeviceToHost));
    if (h_head_logits && D.K > 0)
        XSM_CUDA(ctx, cudaMemcpy2D(h_head_logits, sizeof(float) * D.V, D.hlogits, sizeof(float) * D.ldv, sizeof(float) * D.V, (size_t)D.K * D.M, cudaMemcpyDeviceToHost));
    return XSM_OK;
}

xsm_status xsm_debug_get_kv(xsm_ctx *ctx, int layer, int seq, int pos0, int n, float *h_k, float *h_v) {
    if (!ctx) return XSM_ERR_INVALID_ARG;
    if (!ctx->prefilled) return fail(ctx, XSM_ERR_STATE, "no cache yet");
    const Dev &D = ctx->dev;
    if (layer < 0 || layer >= D.L || seq < 0 || seq >= D.B || pos0 < 0 || n < 0 || !h_k || !h_v)
        return fail(ctx, XSM_ERR_INVALID_ARG, "bad layer, sequence or range");
    xsm_status st = check_device_status(ctx);
    if (st != XSM_OK) return st;
    int held = 0;
    XSM_CUDA(ctx, cudaMemcpy(&held, D.n_blocks + seq, 4, cudaMemcpyDeviceToHost));
    if ((long long)pos0 + n > (long long)held * D.P) return fail(ctx, XSM_ERR_INVALID_ARG, "range beyond the pages held");
    float *sk = at<float>(ctx, ctx->lay.stage_kv), *sv = sk + (size_t)kKvStagePositions * D.d;
    for (int p = 0; p < n; p += kKvStagePositions) {
        const int m = n - p < kKvStagePositions ? n - p : kKvStagePositions;
        XSM_CUDA(ctx, launch_gather_kv(D, ctx->cfg.dtype, layer, seq, pos0 + p, m, sk, sv, ctx->stream));
        ctx->launches += 1;
        XSM_CUDA(ctx, cudaMemcpyAsync(h_k + (size_t)p * D.d, sk, sizeof(float) * (size_t)m * D.d, cudaMemcpyDeviceToHost, ctx->stream));
        XSM_CUDA(ctx, cudaMemcpyAsync(h_v + (size_t)p * D.d, sv, sizeof(float) * (size_t)m * D.d, cudaMemcpyDeviceToHost, ctx->stream));
        XSM_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    }
    return XSM_OK;
}

xsm_status xsm_debug_set_drafts(xsm_ctx *ctx, const int32_t *h_drafts) {
    if (!ctx || !h_drafts) return XSM_ERR_INVALID_ARG;
    if (!ctx->prefilled) return fail(ctx, XSM_ERR_STATE, "xsm_debug_set_drafts before xsm_prefill");
    const Dev &D = ctx->dev;
    if (D.K == 0) return XSM_OK;
    for (int i = 0; i < D.B * D.K; ++i)
        if (h_drafts[i] < 0 || h_drafts[i] >= D.V) return fail(ctx, XSM_ERR_INVALID_ARG, "draft token out of range");
    const xsm_status st = check_device_status(ctx);
    if (st != XSM_OK) return st;
    XSM_CUDA(ctx, cudaMemcpy2D(D.window + 1, sizeof(int32_t) * D.K1, h_drafts, sizeof(int32_t) * D.K,
                               sizeof(int32_t) * D.K, D.B, cudaMemcpyHostToDevice));
    XSM_CUDA(ctx, launch_embed_rows(D, ctx->cfg.dtype, D.K1, -1, 0, ChainLaunch{ctx->stream, false, &ctx->launches}));
    return XSM_OK;
}

xsm_status xsm_debug_get_state(xsm_ctx *ctx, int32_t *h_len, int32_t *h_window, int32_t *h_finished, int32_t *h_pages,
                               int32_t *h_free_pages) {
    if (!ctx) return XSM_ERR_INVALID_ARG;
    if (!ctx->prefilled) return fail(ctx, XSM_ERR_STATE, "no state before xsm_prefill");
    const Dev &D = ctx->dev;
    xsm_status st = check_device_status(ctx);
    if (st != XSM_OK) return st;
    if (h_len) XSM_CUDA(ctx, cudaMemcpy(h_len, D.len, 4 * D.B, cudaMemcpyDeviceToHost));
    if (h_window) XSM_CUDA(ctx, cudaMemcpy(h_window, D.window, 4 * D.M, cudaMemcpyDeviceToHost));
    if (h_finished) XSM_CUDA(ctx, cudaMemcpy(h_finished, D.finished, 4 * D.B, cudaMemcpyDeviceToHost));
    if (h_pages) XSM_CUDA(ctx, cudaMemcpy(h_pages, D.n_blocks, 4 * D.B, cudaMemcpyDeviceToHost));
    if (h_free_pages) XSM_CUDA(ctx, cudaMemcpy(h_free_pages, D.n_free, 4, cudaMemcpyDeviceToHost));
    return XSM_OK;
}

xsm_status xsm_debug_trace_step(xsm_ctx *ctx, uint64_t *h_times, size_t capacity, int *n_rows, int *n_ctas) {
    if (!ctx || !h_times || !n_rows || !n_ctas) return XSM_ERR_INVALID_ARG;
    if (!ctx->prefilled) return fail(ctx, XSM_ERR_STATE, "xsm_debug_trace_step before xsm_prefill");
    if (ctx->phase_launch) return fail(ctx, XSM_ERR_STATE, "the timeline is taken from overlapping launches");
    const int rows = 1 + 2 * ctx->n_stages;
    const size_t words = (size_t)rows * kTraceCtas;
    if (capacity < words) return fail(ctx, XSM_ERR_CAPACITY, "h_times is too small");
    unsigned long long *d_trace = at<unsigned long long>(ctx, ctx->lay.trace);
    XSM_CUDA(ctx, cudaMemsetAsync(d_trace, 0, 8 * words, ctx->stream));
    xsm_status st = lift_limit(ctx);
    if (st != XSM_OK) return st;
    ctx->dev.trace = d_trace;
    st = run_step(ctx);
    ctx->dev.trace = nullptr;
    if (st != XSM_OK) return st;
    st = check_device_status(ctx);
    if (st != XSM_OK) return st;
    XSM_CUDA(ctx, cudaMemcpy(h_times, d_trace, 8 * words, cudaMemcpyDeviceToHost));
    *n_rows = rows;
    *n_ctas = kTraceCtas;
    return XSM_OK;
}

xsm_status xsm_debug_set_script(xsm_ctx *ctx, const int32_t *h_tokens, int n, float mean_accept) {
    if (!ctx) return XSM_ERR_INVALID_ARG;
    if (!ctx->prefilled) return fail(ctx, XSM_ERR_STATE, "xsm_debug_set_script before xsm_prefill");
    Dev &D = ctx->dev;
    if (h_tokens == nullptr || n <= 0) {
        XSM_CUDA(ctx, launch_set_script(D, nullptr, 0, 0, ctx->stream));
        ctx->launches += 1;
        return XSM_OK;
    }
    if (n > ctx->lay.tok_ld) return fail(ctx, XSM_ERR_INVALID_ARG, "script longer than max_seq_len + n_draft + 1");
    if (!(mean_accept >= 0.f) || mean_accept > (float)D.K) return fail(ctx, XSM_ERR_INVALID_ARG, "mean_accept must be in [0, n_draft]");
    for (long long i = 0; i < (long long)D.B * n; ++i)
        if (h_tokens[i] < 0 || h_tokens[i] >= D.V) return fail(ctx, XSM_ERR_INVALID_ARG, "script token out of range");
    int *d_script = at<int>(ctx, ctx->lay.script);
    const xsm_status st = check_device_status(ctx);
    if (st != XSM_OK) return st;
    XSM_CUDA(ctx, cudaMemcpy(d_script, h_tokens, sizeof(int32_t) * (size_t)D.B * n, cudaMemcpyHostToDevice));
    XSM_CUDA(ctx, launch_set_script(D, d_script, n, (int)lrintf(mean_accept * 1024.f), ctx->stream));
    ctx->launches += 1;
    return XSM_OK;
}

xsm_status xsm_debug_set_wait_limits(xsm_ctx *ctx, uint32_t polls, uint32_t barrier_tries) {
    if (!ctx) return XSM_ERR_INVALID_ARG;
    ctx->dev.spin_limit = polls ? polls : kSpinLimit;
    ctx->dev.mbar_limit = barrier_tries ? barrier_tries : kMbarSpinLimit;
    if (ctx->prefilled) {      // the limits are part of the recordings
        ctx->chain.forget();
        if (!ctx->chain.select(ctx->dev)) return fail(ctx, XSM_ERR_CUDA, "the tensor maps of the step could not be made");
    }
    return XSM_OK;
}

xsm_status xsm_debug_launch_stage(xsm_ctx *ctx, int stage) {
    if (!ctx) return XSM_ERR_INVALID_ARG;
    if (!ctx->prefilled) return fail(ctx, XSM_ERR_STATE, "xsm_debug_launch_stage before xsm_prefill");
    if (stage < 0 || stage >= ctx->n_stages) return fail(ctx, XSM_ERR_INVALID_ARG, "no such stage");
    XSM_CUDA(ctx, launch_stage_gate(ctx->dev, stage, ctx->stream));
    XSM_CUDA(ctx, ctx->chain.run_op(ctx->dev, stage, ctx->stream, &ctx->launches));
    XSM_CUDA(ctx, launch_stage_mark(ctx->dev, (stage + 1) % ctx->n_stages, ctx->stream));
    ctx->launches += 2;
    return XSM_OK;
}

int xsm_debug_plan(const xsm_model_config *cfg, int batch, int prompt_positions, int sms, const int32_t *clusters, int32_t *h_stages, int capacity) {
    if (!cfg || !h_stages || check_config(*cfg) || cfg->n_layers > capacity || batch < 1 || batch > cfg->max_batch || prompt_positions < 0 || prompt_positions > cfg->max_seq_len) return 0;
    if (prompt_positions > 0 && (long long)batch * prompt_positions > prompt_rows(*cfg)) return 0;
    if (cfg->dtype == 0 && prompt_positions == 0 && batch * (cfg->n_draft + 1) > kF32Rows) return 0;
    int own[9] = {};
    if (!clusters) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
            (void)cudaGetLastError();
            return 0;
        }
        for (int s = 2; s <= 8; ++s) own[s] = resident_clusters(s);
    }
    if (sms < 1) return 0;
    Layout L;
    make_layout(*cfg, 0, L);
    Dev D;
    memset(&D, 0, sizeof(D));
    set_shape(D, *cfg, L);
    set_batch(D, batch);
    Chain chain;
    std::vector<ChainOp> ops;
    if (!chain.plan(*cfg, weight_offsets(*cfg), sms, clusters ? clusters : own, D, prompt_positions ? prompt_positions : D.K1, prompt_positions > 0, ops)) return 0;
    if ((int)ops.size() > capacity) return 0;
    for (size_t i = 0; i < ops.size(); ++i) {
        const ProjArgs &A = ops[i].proj;
        const int32_t words[8] = {(int32_t)ops[i].kind, A.epi0, A.threads, A.S, A.tok, A.tps, A.tmem_cols, ops[i].smem + kProjDeclared + 1024};
        for (int k = 0; k < 8; ++k) h_stages[8 * i + k] = k == 0 || ops[i].kind == ChainOp::PROJ ? words[k] : 0;
    }
    return (int)ops.size();
}

xsm_status xsm_debug_set_phase_launch(xsm_ctx *ctx, int on) {
    if (!ctx) return XSM_ERR_INVALID_ARG;
    ctx->phase_launch = on ? 1 : 0;
    return XSM_OK;
}

}  // extern "C"
