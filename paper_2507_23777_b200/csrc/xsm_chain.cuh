// The launch chain: one decoding step (or one chunk of a prompt) as a sequence of kernels on one stream, each launched
// with programmatic stream serialization so that it starts, and fetches what does not depend on the step, while its
// predecessor still runs.
#pragma once
#include "xsm_common.cuh"

#include <stddef.h>

namespace xsm {

// what a projection does with its dot products
enum ProjEpilogue : int {
    PE_QKV = 0,       // self-attention: rotated, scaled queries as fp16 planes; rotated keys and values into the cache
    PE_ADD = 1,       // residual stream: h += y, and h * (next RMSNorm gain) as bf16 planes, with its sums of squares
    PE_QUERY = 2,     // cross-attention queries, scaled, as fp16 planes
    PE_GATEUP = 3,    // SiLU(gate) * up as bf16 planes
    PE_LOGITS = 4,    // fp32
    PE_HEADY = 5,     // g + SiLU(y) as bf16 planes (MLP decoding head)
    PE_HEADADD = 6    // g + y as bf16 planes (cross-attention decoding head)
};

constexpr float kLog2e = 1.4426950408889634f;
constexpr int kTokenTile = 128;       // token rows that share a plane
constexpr int kProjRing = 16;         // most operand blocks of one kind that a CTA keeps in shared memory
constexpr int kClusterThreads = 384;  // most threads of a projection's CTA in a cluster
constexpr int kTileThreads = 512;     // of one without
constexpr int kCtaSmem = 227 * 1024;  // shared memory that a CTA may have
constexpr int kSmSmem = 228 * 1024, kSmTmemCols = 512;      // of an SM: shared memory (1 KB of every CTA's is the system's), columns of tensor memory
constexpr int kProjDeclared = (4 * kProjRing + 1) * 8 + kTokenTile * 4;      // shared memory that every tcgen05 projection declares, at least
// dynamic shared memory of a projection, at most (what a kernel declares comes on top: for q, k, v the token rows' places too)
__host__ __device__ constexpr int proj_smem_max(int epi0) { return epi0 == PE_QKV ? 224 * 1024 - 128 : 224 * 1024; }

// A group of weight matrices of one shape in a projection stage: one matrix, or one per decoding head.
struct ProjGroup {
    int units, jobs, ld;              // output units of one matrix; matrices; row length of the output
    int job_tiles, tiles;             // row tiles of one matrix, of the group
    bf16 *out;                        // planes of ld columns (a set per decoding head; layout: xsm_proj.cuh)
    float *logits;                    // PE_LOGITS: [jobs][M][ld]
    const bf16 *w;                    // first matrix (few token rows: read without tensor maps)
    size_t w_stride;                  // elements from one matrix of the group to the next
};

struct ProjArgs {
    int epi0, epi1;                   // of the two groups; epi1 < 0: one group
    int stage;                        // index of the kernel in its chain
    int layer, kdim, rows, Mp;        // rows: token rows; Mp: rows of a plane (a multiple of 8, at most kTokenTile)
    int tt, tok, qp;                  // tiles of tok token rows (parts of one plane set, or one for each); rows of the planes of queries
    int t, pos0, pos_end;             // token row m is position start + m % t of sequence m / t; start: pos0, or the sequence's length if pos0 < 0
    int threads;                      // of a CTA
    int S, tps, group;                // CTAs per cluster (cuts of the columns), token rows each of them finishes, dealt out in groups of so many
    uint32_t inv_s, inv_q;            // 65536 / S + 1, 65536 / (tps / group) + 1: small numbers are divided by multiplying
    int na, nb, tmem_cols;            // operand blocks in shared memory (weights, activations), accumulator columns
    int many, chain;                  // a CTA may have several accumulators; operand blocks that each adds up
    int norm, ss_parts;               // the input is an RMSNorm input; shares of its sums of squares (0: not needed)
    int z_jobs, x_jobs;               // group 0 has one matrix per decoding head; the activations too
    const bf16 *x;                    // planes of kdim columns (x_jobs: a set per decoding head)
    int upc, ctas;                    // few token rows: units (pairs of rows) per CTA, CTAs (per decoding head with x_jobs)
    int slots, chunk, slot_rows;      // weight tiles in shared memory; columns, rows of one
    int late_go;                      // let the next kernel start only after this one's wait
    float scale;                      // queries
    const void *gain;                 // PE_ADD: gain of the RMSNorm that reads h next; PE_HEADY / PE_HEADADD: of the final RMSNorm
    __half *q;                        // PE_QKV, PE_QUERY: planes [2][qp][d] (a set per decoding head)
    ProjGroup g[2];
};

// Attention of a stage: t query rows of every sequence against the cached keys of the sequence (self) or of the condition.
struct AttnArgs {
    int stage;
    int cross, sets, layer;           // sets: decoding heads that attend in this stage (cross-attention heads), else 1
    int t, rows, Mp, qp, pos0, pos_end;      // as in ProjArgs
    int qt;                           // tiles of kTokenTile rows of a sequence
    int warps, warm;                  // that attend (few rows: 8 or 16); run the code once before the wait
    int S, split, slots, ring;        // most CTAs per (sequence, head) (a cluster), keys for each; page pairs in shared memory, its bytes
    int recv;                         // where the other CTAs' partial results arrive in shared memory
    const void *pool;                 // cache tiles
    const __half *q;                  // planes [2][qp][d] (a set per decoding head)
    bf16 *out;                        // planes of d columns (a set per decoding head; layout: xsm_proj.cuh)
    const bf16 *wq, *x;               // wq not null: the queries are projected here, wq x (x: planes of d columns)
    int ss_parts;                     // shares of the sums of squares of x
    float scale;                      // of the queries
};

// How the kernels of a chain are launched.
struct ChainLaunch {
    cudaStream_t stream;
    bool overlap;                     // programmatic stream serialization
    unsigned long long *count;        // launches

    template <typename... Args>
    cudaError_t launch(dim3 grid, dim3 block, int smem, int cluster, const void *fn, const Args &...args) const {
        cudaLaunchConfig_t c = {};
        c.gridDim = grid;
        c.blockDim = block;
        c.dynamicSmemBytes = (size_t)smem;
        c.stream = stream;
        cudaLaunchAttribute at[2];
        int n = 0;
        if (overlap) {
            at[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
            at[n++].val.programmaticStreamSerializationAllowed = 1;
        }
        if (cluster > 1) {
            at[n].id = cudaLaunchAttributeClusterDimension;
            at[n].val.clusterDim.x = (unsigned)cluster;
            at[n].val.clusterDim.y = 1;
            at[n++].val.clusterDim.z = 1;
        }
        c.attrs = at;
        c.numAttrs = (unsigned)n;
        void *p[] = {const_cast<void *>(static_cast<const void *>(&args))...};
        ++*count;
        return cudaLaunchKernelExC(&c, fn, p);
    }
};

// opens a kernel for `smem` bytes of dynamic shared memory (and for clusters of more than eight CTAs) on the current device
cudaError_t open_kernel(const void *fn, int smem, bool large_cluster);

// Instance of the projection over few token rows that serves `rows` token rows and rows of kdim weights: warps that multiply, tiles of
// eight token rows, blocks of 32 columns that each holds in registers, columns of one pass, hi and lo parts in one product
struct FewShape { int warps, nt, blocks, pass; bool pack; };
inline FewShape few_shape(int rows, int kdim) {
    FewShape f;
    f.pack = rows <= 4;
    f.nt = rows <= 8 ? 1 : 2;
    f.warps = kdim > 2048 ? 15 : 8;
    f.blocks = kdim > 2048 ? 9 : kdim > 1024 ? 8 : 4;
    f.pass = f.warps * f.blocks * 32;
    return f;
}
cudaError_t launch_proj_few(const Dev &D, const ProjArgs &A, int smem, const ChainLaunch &L);
int resident_clusters(int size);      // clusters of the projection below that the device runs at a time, an SM for each CTA
cudaError_t launch_proj_umma(const Dev &D, const ProjArgs &A, const void *maps, int smem, const ChainLaunch &L);
cudaError_t launch_attn(const Dev &D, const AttnArgs &A, const ChainLaunch &L);
int attn_query_smem(const Dev &D, int t);
int attn_park(const Dev &D, int t, int warps);
int attn_recv(const Dev &D, int S, int t);
// fp32 models: at most this many token rows
constexpr int kF32Rows = 24;
cudaError_t launch_proj_f32(const Dev &D, const ProjArgs &A, int smem, const ChainLaunch &L);
cudaError_t launch_attn_f32(const Dev &D, const AttnArgs &A, const ChainLaunch &L);
int cond_tile(int n_cond);
cudaError_t launch_cond_kv(const Dev &D, const void *maps, void *pool, int n_sets, cudaStream_t st);
cudaError_t launch_tail(const Dev &D, int dtype, int stage, const ChainLaunch &L);
// embeds the window of every sequence (pos0 < 0) or t prompt tokens of each from position pos0 on
cudaError_t launch_embed_rows(const Dev &D, int dtype, int t, int pos0, int pos_end, const ChainLaunch &L);
// state of a new request: pool, sequences with prompt_len - 1 positions in the cache, first window
cudaError_t launch_begin(const Dev &D, const RunParams &R, cudaStream_t st);
// single stages (inspection): waits until the stages before `stage` have run one by one; notes that `done` of them have
cudaError_t launch_stage_gate(const Dev &D, int stage, cudaStream_t st);
cudaError_t launch_stage_mark(const Dev &D, int done, cudaStream_t st);
// request parameters that change between prefills: the token limit and the xsm_generate it is for, scripted drafts
cudaError_t launch_set_limit(const Dev &D, int max_new, int call, cudaStream_t st);
cudaError_t launch_set_script(const Dev &D, const int *script, int n, int acc, cudaStream_t st);

}  // namespace xsm
