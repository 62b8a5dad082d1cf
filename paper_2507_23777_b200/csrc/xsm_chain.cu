// Host side of the launch chain: tensor maps, how each stage is cut over the chip, recording and replay of a step.
#include "xsm_host.h"

#include <cuda.h>
#include <string.h>

#include <algorithm>
#include <mutex>
#include <unordered_map>

namespace xsm {

static_assert(sizeof(TensorMap) == sizeof(CUtensorMap), "tensor map size");

constexpr int kMaxPlans = 8;                      // batch sizes whose recordings are kept
constexpr int kAccumulators = 256;                // columns of tensor memory of a CTA, at most

cudaError_t open_kernel(const void *fn, int smem, bool large_cluster) {
    static std::mutex mu;
    struct Opened { int smem = 0; bool large = false; };
    static std::unordered_map<const void *, Opened> opened[kMaxDevices];      // what each kernel has been opened for, by device
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(mu);
    Opened &o = opened[dev][fn];
    if (large_cluster && !o.large) {
        if ((e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1)) != cudaSuccess) return e;
        o.large = true;
    }
    if (smem > o.smem) {
        if ((e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)) != cudaSuccess) return e;
        o.smem = smem;
    }
    return cudaSuccess;
}

StepPlan::~StepPlan() {
    if (exec) cudaGraphExecDestroy(exec);
    if (graph) cudaGraphDestroy(graph);
}

Chain::~Chain() {
    forget();
    if (record_) cudaStreamDestroy(record_);
}

void Chain::forget() {
    plan_ = nullptr;
    plans_.clear();
}

// ------------------------------------------------------------------------------------- tensor maps

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                                  const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static bool encode(void *fn, TensorMap *out, const void *base, int cols, int rows, int sets, size_t set_bytes, int box_rows) {
    cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)sets};
    cuuint64_t strides[2] = {(cuuint64_t)cols * 2, (cuuint64_t)set_bytes};
    cuuint32_t box[3] = {64, (cuuint32_t)box_rows, 1}, estr[3] = {1, 1, 1};
    return ((EncodeTiledFn)fn)(reinterpret_cast<CUtensorMap *>(out), CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(base), dims, strides,
                               box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// `count` matrices [rows][kdim] of bf16, stride_elems apart (the layers' copies, or the decoding heads'): boxes of 64 columns
bool Chain::weight_map(TensorMap *out, size_t elem_off, int rows, int kdim, int count, size_t stride_elems, int box_rows) {
    const size_t stride = count > 1 ? stride_elems * 2 : (size_t)rows * kdim * 2;
    return encode(encode_, out, weights_ + elem_off * 2, kdim, rows, count, stride, box_rows);
}
bool Chain::init(const xsm_model_config &c, const WeightOffsets &w, const char *weights, int sm_count) {
    c_ = c;
    w_ = w;
    weights_ = weights;
    sms_ = sm_count;
    if (c.dtype == 0) return true;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &encode_, cudaEnableDefault, &q) != cudaSuccess || q != cudaDriverEntryPointSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    for (int s = 2; s <= 8; ++s) clusters_[s] = resident_clusters(s);
    const int d = c.d_model, f = c.d_ff, V = c.vocab, L = c.n_layers, K = c.n_draft;
    const size_t ls = L > 1 ? w.wq[1] - w.wq[0] : 0;
    bool ok = weight_map(&qkv_, w.wq[0], 3 * d, d, L, ls, 128) && weight_map(&o_, w.wo[0], d, d, L, ls, 128) &&
              weight_map(&qc_, w.wqc[0], d, d, L, ls, 128) && weight_map(&oc_, w.woc[0], d, d, L, ls, 128) &&
              weight_map(&gate_, w.wgate[0], f, d, L, ls, 64) && weight_map(&up_, w.wup[0], f, d, L, ls, 64) &&
              weight_map(&down_, w.wdown[0], d, f, L, ls, 128) && weight_map(&kc_, w.wkc[0], d, c.d_cond, L, ls, 128) &&
              weight_map(&vc_, w.wvc[0], d, c.d_cond, L, ls, 128) && weight_map(&lm_, w.W0, V, d, 1, 0, 128);
    if (K > 0) {
        const size_t hs = K > 1 ? w.Wout[1] - w.Wout[0] : 0;
        ok = ok && weight_map(&head_out_, w.Wout[0], V, d, K, hs, 128);
        if (c.head_kind == 1)
            ok = ok && weight_map(&head_in_, w.hq[0], d, d, K, hs, 128) && weight_map(&head_o_, w.ho[0], d, d, K, hs, 128) &&
                 weight_map(&head_kc_, w.hk[0], d, c.d_cond, K, hs, 128) && weight_map(&head_vc_, w.hv[0], d, c.d_cond, K, hs, 128);
        else
            ok = ok && weight_map(&head_in_, w.W1[0], d, d, K, hs, 128);
    }
    return ok;
}

// ------------------------------------------------------------------------------------- cuts of a stage

// Cluster size, rings and shared memory of a projection over `rows` token rows.  The row tiles of a stage (8 to 128) leave
// SMs idle at one CTA each, so the columns are cut as far as all clusters still run at once.
void Chain::plan_proj(ChainOp &op, int rows, int Mp, int kdim) {
    ProjArgs &A = op.proj;
    if (c_.dtype == 0) {      // a warp for every unit as long as there are SMs; the activations of a chunk of columns in 96 KB
        const int units = A.epi0 == PE_QKV ? A.g[0].units / 2 : A.g[0].units + (A.epi1 >= 0 ? A.g[1].units * A.g[1].jobs : 0);
        A.kdim = kdim;
        A.rows = rows;
        A.Mp = rows;
        A.ctas = std::min((units + 7) / 8, std::max(1, A.x_jobs ? sms_ / A.g[0].jobs : sms_));
        A.chunk = std::min(kdim, 96 * 1024 / (4 * rows) / 128 * 128);
        op.kind = ChainOp::F32;
        op.smem = std::max(A.chunk * rows * 4, 8 * kF32Rows * 4);
        return;
    }
    if (plan_few(op, rows, Mp, kdim)) return;
    A.kdim = kdim;
    A.rows = rows;
    A.Mp = Mp;
    const int tiles = A.g[0].tiles + (A.epi1 >= 0 ? A.g[1].tiles : 0), nblk = kdim / 64;
    // How a tile of weight rows is cut: its columns over a cluster of S CTAs, as many as fit into the GPCs at a time, an SM to each
    // CTA (of six CTAs 22 clusters, of eight 15; where two CTAs fit an SM more would run, which has not been tried).  More than 48 token rows in one plane: these into T parts too,
    // each with the weights for itself, which leaves less to exchange and to finish in a CTA.  There the stage's time after the
    // wait in cycles, as measured, chooses among S and T: a product 47, or N / 2 where the token rows (hi and lo) bound it;
    // activations, and weights that do not fit the ring, 59 bytes a cycle; 45 for every token row that is sent, 250 for every
    // one that is finished.  Eight layers of width 1024, whole rows and parts: 112 rows 565 and 459 us a step, 90 rows 470 and 424, 80
    // rows 433 and 411, 60 rows 401 and 369, 50 rows 373 and 361; with one accumulator 40 rows 354 and 356, 30 rows 304 and 331, so
    // up to 48 rows T is 1 and the largest S that fits is taken, without weighing.
    //
    // How many blocks an accumulator adds up: every instruction cuts off what lies below the accumulator's last bit, so the error of a
    // sum grows with their number (projections alone, against 64 bits, in units of 1e-6 of the result: sums of 128 instructions at
    // width 2048 7.9, of at most 16 6.9, as warps that share the columns have with mma.sync).  Up to 16 token rows four blocks, 16
    // instructions; token rows in parts: as many as a CTA would have with the largest S of whole token rows.  From 17 to 48 rows
    // one for all blocks (8.0 at width 2048, 7.2 at 1024): several cost 1 to 4 % of a step.
    int S = 1, T = 1, whole = 1;      // whole: that largest S
    const bool parts = A.tt == 1 && rows > 48;
    for (int s = 2; s <= std::min(8, nblk); ++s)
        if (tiles * A.tt <= clusters_[s]) whole = s;
    const int chain = parts ? (nblk + whole - 1) / whole : rows <= 16 ? 4 : nblk;
    double best = 1e30;
    for (int t = 1; t <= (parts ? Mp / 8 : 1); ++t) {
        const int nt = parts ? (Mp / 8 + t - 1) / t * 8 : std::min(Mp, kTokenTile);
        if ((Mp + nt - 1) / nt != t) continue;
        for (int s = 1; s <= std::min(8, nblk); ++s) {
            const int n = (nblk + s - 1) / s;
            if (s > 1 ? tiles * A.tt * t > clusters_[s] : t > 1 && tiles * t > sms_) continue;
            if (parts && (n + chain - 1) / chain * 2 * nt > kAccumulators) continue;
            const double late = std::max(0.0, n * 16384.0 - 160 * 1024), sent = s > 1 ? 600 + 45.0 * nt : 0;
            const double cost = n * 4 * std::max(47.0, nt * 1.0) + (n * 256.0 * nt + late) / 59 + sent + 250.0 * ((nt + 4 * s - 1) / (4 * s) * 4);
            if (!parts || cost < best) { best = cost; S = s; T = t; }
        }
    }
    A.S = S;
    const int planes = A.tt;
    A.tok = planes > 1 ? Mp : (Mp / 8 + T - 1) / T * 8;
    A.tt = planes * T;
    // Token rows are dealt out to the CTAs that finish them one by one where there are few (in fours, two of eight CTAs finished
    // five rows, four by each thread: 763 -> 683 us a step at width 1024, 20 rows 771 -> 748); 28 rows at width 2048, five to a
    // CTA, are finished faster in fours, read as 16 bytes (2085 against 2129).
    const int tile_rows = std::min(rows, A.tok), G = S > 1 && rows <= 24 ? 1 : 4;
    A.group = G;
    A.tps = ((tile_rows + G - 1) / G + S - 1) / S * G;
    // Four warps more than finish token rows, or as many as the accumulator's columns keep busy, at most twelve.  Eight are enough where a
    // CTA finishes one row (two in gate/up, whose rows take 64 threads each): the first four fetch and multiply, the others finish.
    // Against twelve there too: 5 rows of width 768 33.83 -> 33.57 ms a request, of width 1024 57.45 -> 56.48, one row 54.90 -> 53.76.  Of
    // twelve warps the first four do both, and those that are left over prepare the rows' scales and wait for nothing.
    A.threads = S == 1 ? kTileThreads : G == 1 ? 128 * std::min(kClusterThreads / 128, std::max(1 + (A.epi0 == PE_GATEUP ? (A.tps + 1) / 2 : A.tps), A.tok / 8)) : kClusterThreads;
    A.inv_s = 65536 / S + 1;
    A.inv_q = 65536 / (A.tps / G) + 1;
    const int n = (nblk + S - 1) / S, b_bytes = 2 * A.tok * 128, a_bytes = 128 * 128, sums = S * A.tps * 512;
    // more tiles than SMs: two CTAs to an SM
    // (the activations' share of the ring: from the L2, but all of them after the wait)
    const int most = proj_smem_max(A.epi0), room = (tiles * A.tt * S > sms_ ? most / 2 : most) - 1024 - (S > 1 ? sums : 0);
    A.nb = std::min(n, std::max(2, std::min(kProjRing, (rows > 32 ? room * 9 / 20 : room / 3) / b_bytes)));
    A.na = std::min(n, std::min(kProjRing, (room - A.nb * b_bytes) / a_bytes));
    A.nb = std::min(n, std::min(kProjRing, (room - A.na * a_bytes) / b_bytes));
    const int sums_fit = kAccumulators / (2 * A.tok);
    A.chain = std::max(chain, (n + sums_fit - 1) / sums_fit);
    // (the residual projections of a step share a kernel: with one for out and one for down, each evicts the other's code, and five
    // rows of width 768 take 299 us a step instead of 292; with several accumulators in all kernels 295)
    A.many = n > A.chain || (A.epi0 == PE_ADD && (parts || rows <= 16));
    A.tmem_cols = 32;
    while (A.tmem_cols < (n + A.chain - 1) / A.chain * 2 * A.tok) A.tmem_cols *= 2;
    const int rings = A.na * a_bytes + A.nb * b_bytes;
    op.smem = 1024 + (S > 1 ? rings + sums : std::max(rings, sums));
    // A CTA that asks for tensor memory waits until there is enough, and its cluster, which holds some, waits for it: two clusters of
    // different streams must never wait for each other so.  CTAs of a cluster take at least the share of an SM's shared memory that
    // their columns are of its tensor memory: what fits the one fits the other, whichever meet there and however few registers they
    // have.  (Kernels without clusters wait for nobody who may be waiting so.  From 33 rows on, in narrow models and short cuts of the
    // columns, there is something to add: 50 KB become 57, 103 become 114.)
    if (S > 1) op.smem = std::max(op.smem, A.tmem_cols * (kSmSmem / kSmTmemCols) - 1024 - kProjDeclared);
}

// The projections over few token rows: how the units are dealt out, passes over the columns, shared memory.  False: the
// shape does not fit, or the tensor cores of the 5th generation do better: a CTA reads all activations here and a slice of them there,
// which tells as soon as they are more than a few KB.  Whole steps of eight layers (four times as many gated as model columns, K
// heads, vocabulary 2048), us, this path and that one:
//   token rows         1, K 0     3, K 2     4, K 3     4, K 0     5, K 4     8, K 7     9, K 2    16, K 3
//   width 128         132 154    138 165    140 167    138 159    147 169    154 180    166 182    173 199
//   width 256         141 161    152 171    153 175    152 164    165 174    173 179    190 184    202 195
//   width 384         156 170    166 180    168 182    164 177    186 187    198 189    220 184    239 199
//   width 512         162 172    175 185    177 188    173 181    197 192    217 196    239 195    255 206
//   width 640         176 182    191 193    194 195    185 190    208 198    228 207    252 204    266 217
//   width 768         183 193    198 203    201 207    195 192    219 194    241 201    261 197    277 205
// With eight times as many gated columns four rows lose in the down projection from 3072 columns on (width 384 191 against 179);
// with a vocabulary of 8001 five rows of width 256 are even and eight lose (178 against 178, 195 against 184).
bool Chain::plan_few(ChainOp &op, int rows, int Mp, int kdim) {
    ProjArgs &A = op.proj;
    const int width = rows <= 3 ? 768 : rows == 4 ? 640 : 128, columns = rows <= 3 ? 8192 : rows == 4 ? 2560 : 1024;      // most of each
    if (rows > 16 || c_.d_model > width || kdim > columns) return false;
    const bool pairs = A.epi0 == PE_QKV || A.epi0 == PE_GATEUP;
    const int units = A.epi0 == PE_QKV ? A.g[0].units / 2 : A.g[0].units + (A.epi1 >= 0 ? A.g[1].units * A.g[1].jobs : 0);
    const int share = A.x_jobs ? std::max(1, sms_ / A.g[0].jobs) : sms_;      // CTAs for `units`
    A.upc = (units + share - 1) / share;
    A.ctas = (units + A.upc - 1) / A.upc;
    const FewShape f = few_shape(rows, kdim);
    const int n_rows = A.upc * (pairs ? 2 : 1), tiles = (n_rows + 15) / 16;
    const int red = tiles * f.warps * 16 * (f.nt * 8 + 1) * 4;
    A.slot_rows = tiles == 1 ? (n_rows + 7) / 8 * 8 : 16;
    // passes no wider than the registers hold, and narrow enough for two of them in flight
    int slots = 0;
    for (int passes = (kdim + f.pass - 1) / f.pass; passes <= 16; ++passes) {
        A.chunk = ((kdim + passes - 1) / passes + 63) / 64 * 64;
        const int pitch = A.chunk * 2 + 64, stages = tiles * ((kdim + A.chunk - 1) / A.chunk);
        slots = std::min(std::min(stages, kProjRing), (proj_smem_max(A.epi0) - red) / (A.slot_rows * pitch));
        if (slots >= std::min(stages, 2)) break;
        slots = 0;
    }
    // (a residual projection folds a token row over 32 lanes at most: enough on 24 SMs and more)
    if (slots == 0 || (A.upc > 32 && A.epi0 == PE_ADD) || A.ctas > kShareLd) return false;
    A.kdim = kdim;
    A.rows = rows;
    A.Mp = Mp;
    A.S = 1;
    A.slots = slots;
    op.kind = ChainOp::FEW;
    op.smem = slots * A.slot_rows * (A.chunk * 2 + 64) + red;
    return true;
}

AttnArgs Chain::plan_attn(const Dev &D, bool cross, int sets, int t, int Mp) {
    AttnArgs A;
    memset(&A, 0, sizeof(A));
    A.cross = cross;
    A.sets = sets;
    A.t = t;
    A.Mp = Mp;
    A.qt = (t + kTokenTile - 1) / kTokenTile;
    const int items = D.B * D.H * sets * A.qt, upp = D.P / 32, pair = 2 * D.P * D.dh * 2;
    // A (sequence, head) is cut over a cluster of S CTAs, about one per SM in all and no more than run at a time.  A CTA more pays
    // for every 384 keys (192 in heads of 128; 12 or 6 units of 32 keys, 1 us each, over eight warps) and less than that costs
    // more in the exchange: medium width at 500 keys 797 -> 758 us a step, at 1500 851 -> 818, heads of 128 at 513 keys 9.2 -> 7.0
    // us a stage.  Tiles of 16 rows: a unit serves all of them, 128 keys.  Sixteen warps where a CTA can have more than 512
    // keys and an SM to itself.
    A.S = 1;
    const int per_sm = t <= 8 && D.dh <= 64 ? 2 : 1;      // CTAs that an SM can hold
    for (int s = 2; s <= 8; ++s)
        if (items <= per_sm * clusters_[s] && items * s <= sms_ + sms_ / 8) A.S = s;
    A.split = t <= 8 ? (D.dh <= 64 ? 384 : 192) : 128;
    const int keys = cross ? D.C : D.max_blocks * D.P;
    A.S = std::min(A.S, (keys + A.split - 1) / A.split);
    const bool alone = items * A.S <= sms_ && (A.S == 1 || items <= clusters_[A.S]);      // an SM for every CTA
    A.warps = t <= 8 && D.dh <= 64 && alone && keys > 512 * A.S ? 16 : 8;
    A.warm = A.S == 1 && items <= sms_;
    const int round = upp == 1 || upp == 2 || upp == 4 ? 8 / upp : 1;
    const int pages = ((cross ? D.cpages : D.max_blocks) + A.S - 1) / A.S;
    const int budget = alone ? 128 * 1024 : 100 * 1024;
    int slots = std::min(16, budget / pair) / round * round;
    slots = std::max(round, std::min(slots, (pages + round - 1) / round * round));
    A.slots = slots;
    A.ring = std::max(slots * pair, attn_park(D, t, A.warps));
    return A;
}

// Does a cross-attention stage project its own queries?  The head's weights have to fit beside the pages (all of them, else at
// least two at a time), and every CTA needs an SM to itself.
bool Chain::own_queries(const Dev &D, AttnArgs &A) const {
    const int weights = attn_query_smem(D, A.t), pair = 2 * D.P * D.dh * 2;
    if (c_.dtype != 1 || weights == 0 || A.S * D.H * D.B > sms_ || (A.S > 1 && D.H * D.B > clusters_[A.S])) return false;
    const int room = proj_smem_max(PE_QUERY) - weights - attn_recv(D, A.S, A.t), pages = (D.cpages + A.S - 1) / A.S;
    const int all = A.S > 1 ? pages * pair : (pages - 1) * pair + ((D.C - (pages - 1) * D.P + 31) / 32 * 32) * D.dh * 4;
    A.ring = std::max(all <= room ? all : room / pair * pair, attn_park(D, A.t, 16));
    A.slots = std::min(16, A.ring / pair);
    return A.ring <= room && (all <= room || A.slots >= 2);
}

bool Chain::build(const Dev &D, int t, bool prompt, std::vector<ChainOp> &ops) {
    const xsm_model_config &c = c_;
    const int d = c.d_model, f = c.d_ff, V = c.vocab, K = c.n_draft, L = c.n_layers, rows = D.B * t;
    const int Mp = rows > kTokenTile ? kTokenTile : (rows + 7) / 8 * 8, tt = (rows + kTokenTile - 1) / kTokenTile, qp = tt * Mp;
    const bool ca = c.head_kind == 1;
    const float qscale = D.scale * kLog2e;      // softmax in base 2
    const size_t es = c.dtype == 1 ? 2 : 4;
    auto gain = [&](size_t off) { return (const void *)(weights_ + off * es); };
    const size_t head_stride = K > 1 ? w_.Wout[1] - w_.Wout[0] : 0;
    int shares = 1;                       // of the sums of squares of h: one from the embedding, then four per row tile of the writer
    auto proj = [&](int epi0, int epi1, int layer, const TensorMap &w0, const TensorMap *w1, size_t w_off, size_t w1_off, const void *x) -> ChainOp & {
        ops.emplace_back();
        ChainOp &op = ops.back();
        op.kind = ChainOp::PROJ;
        memset(&op.proj, 0, sizeof(op.proj));
        op.maps.w0 = w0;
        op.maps.w1 = w1 ? *w1 : w0;
        ProjArgs &A = op.proj;
        A.x = (const bf16 *)x;
        A.g[0].w = (const bf16 *)(weights_ + w_off * es);
        A.g[1].w = (const bf16 *)(weights_ + w1_off * es);
        A.g[0].w_stride = A.g[1].w_stride = head_stride;
        A.epi0 = epi0; A.epi1 = epi1; A.layer = layer; A.t = t; A.pos0 = -1; A.scale = qscale; A.tt = tt; A.qp = qp;
        return op;
    };
    auto group = [&](ProjGroup &g, int units, int tile_rows, int jobs, int ld, void *out, float *logits) {
        g.units = units; g.jobs = jobs; g.job_tiles = (units + tile_rows - 1) / tile_rows; g.tiles = g.job_tiles * jobs;
        g.ld = ld; g.out = (bf16 *)out; g.logits = logits;
    };
    auto attn = [&](bool cross, int sets, int layer, const void *pool, const void *q, void *out) {
        ops.emplace_back();
        ChainOp &op = ops.back();
        op.kind = ChainOp::ATTN;
        op.attn = plan_attn(D, cross, sets, t, Mp);
        op.attn.layer = layer; op.attn.rows = rows; op.attn.pos0 = -1; op.attn.qp = qp;
        op.attn.pool = pool; op.attn.q = (const __half *)q; op.attn.out = (bf16 *)out;
    };
    auto residual = [&](int layer, const TensorMap &w, size_t w_off, const void *x, int kdim, size_t next_gain) {
        ChainOp &op = proj(PE_ADD, -1, layer, w, nullptr, w_off, 0, x);
        group(op.proj.g[0], d, 128, 1, d, D.xa_, nullptr);
        op.proj.gain = gain(next_gain);
        plan_proj(op, rows, Mp, kdim);
        shares = op.kind == ChainOp::PROJ ? d / 128 * 4 : op.proj.ctas;
    };
    auto normed = [&](ChainOp &op) {
        op.proj.norm = 1;
        op.proj.ss_parts = shares;
        plan_proj(op, rows, Mp, d);
    };
    if (prompt) { ops.emplace_back(); ops.back().kind = ChainOp::EMBED; }
    for (int l = 0; l < L; ++l) {
        {
            ChainOp &op = proj(PE_QKV, -1, l, qkv_, nullptr, w_.wq[l], 0, D.xa_);
            group(op.proj.g[0], 3 * d, 128, 1, 0, nullptr, nullptr);
            op.proj.q = (__half *)D.qp_;
            op.proj.late_go = l == 0;
            normed(op);
        }
        if (prompt && l == L - 1) break;      // the last keys and values are in the cache
        attn(false, 1, l, D.kv_pool, D.qp_, D.aa_);
        residual(l, o_, w_.wo[l], D.aa_, d, w_.g2[l]);
        const size_t at = ops.size();
        attn(true, 1, l, D.ckv_pool, D.qp_, D.aa_);
        if (!prompt && own_queries(D, ops[at].attn)) {
            AttnArgs &A = ops[at].attn;
            A.wq = (const bf16 *)weights_ + w_.wqc[l];
            A.x = (const bf16 *)D.xa_;
            A.ss_parts = shares;
            A.scale = qscale;
        } else {
            ops.pop_back();
            ChainOp &op = proj(PE_QUERY, -1, l, qc_, nullptr, w_.wqc[l], 0, D.xa_);
            group(op.proj.g[0], d, 128, 1, 0, nullptr, nullptr);
            op.proj.q = (__half *)D.qp_;
            normed(op);
            attn(true, 1, l, D.ckv_pool, D.qp_, D.aa_);
        }
        residual(l, oc_, w_.woc[l], D.aa_, d, w_.g3[l]);
        {
            ChainOp &op = proj(PE_GATEUP, -1, l, gate_, &up_, w_.wgate[l], w_.wup[l], D.xa_);
            group(op.proj.g[0], f, 64, 1, f, D.actp_, nullptr);
            normed(op);
        }
        residual(l, down_, w_.wdown[l], D.actp_, f, l + 1 < L ? w_.g1[l + 1] : w_.gf);
    }
    if (prompt) return true;
    {
        ChainOp &op = proj(PE_LOGITS, K == 0 ? -1 : ca ? PE_QUERY : PE_HEADY, 0, lm_, K > 0 ? &head_in_ : nullptr, w_.W0,
                            K == 0 ? 0 : ca ? w_.hq[0] : w_.W1[0], D.xa_);
        group(op.proj.g[0], V, 128, 1, D.ldv, nullptr, D.logits0);
        if (K > 0) group(op.proj.g[1], d, 128, K, d, D.yp_, nullptr);
        op.proj.gain = gain(w_.gf);
        op.proj.q = (__half *)D.hq_;
        normed(op);
    }
    if (K > 0 && ca) {
        attn(true, K, 0, D.hckv_pool, D.hq_, D.ha_);
        ChainOp &op = proj(PE_HEADADD, -1, 0, head_o_, nullptr, w_.ho[0], 0, D.ha_);
        group(op.proj.g[0], d, 128, K, d, D.yp_, nullptr);
        op.proj.gain = gain(w_.gf);
        op.proj.z_jobs = op.proj.x_jobs = 1;
        op.proj.ss_parts = shares;
        plan_proj(op, rows, Mp, d);
    }
    if (K > 0) {
        ChainOp &op = proj(PE_LOGITS, -1, 0, head_out_, nullptr, w_.Wout[0], 0, D.yp_);
        group(op.proj.g[0], V, 128, K, D.ldv, nullptr, D.hlogits);
        op.proj.z_jobs = op.proj.x_jobs = 1;
        plan_proj(op, rows, Mp, d);
    }
    ops.emplace_back();
    ops.back().kind = ChainOp::TAIL;
    return true;
}

// ---------------------------------------------------------------------------------------- running

// Token rows of a chunk of a prompt.  bf16: 2048, where the narrowest projections (d_model 1024) have a tile for nearly
// every SM; no more than the prompts of a batch can have.
int prompt_rows(const xsm_model_config &c) {
    if (c.dtype == 0) return kF32Rows;
    const long long all = ((long long)c.max_batch * c.max_seq_len + kTokenTile - 1) / kTokenTile * kTokenTile;
    return (int)std::max<long long>(kTokenTile, std::min<long long>(2048, all));
}

cudaError_t Chain::run(const Dev &D, const ChainOp &op, int t, const ChainLaunch &L) {
    switch (op.kind) {
        case ChainOp::PROJ: return launch_proj_umma(D, op.proj, &op.maps, op.smem, L);
        case ChainOp::FEW: return launch_proj_few(D, op.proj, op.smem, L);
        case ChainOp::F32: return launch_proj_f32(D, op.proj, op.smem, L);
        case ChainOp::ATTN: return c_.dtype == 1 ? launch_attn(D, op.attn, L) : launch_attn_f32(D, op.attn, L);
        case ChainOp::TAIL: return launch_tail(D, c_.dtype, op.proj.stage, L);
        case ChainOp::EMBED: return launch_embed_rows(D, c_.dtype, t, op.attn.pos0, op.attn.pos_end, L);
    }
    return cudaErrorInvalidValue;
}

bool Chain::plan(const xsm_model_config &c, const WeightOffsets &w, int sms, const int *clusters, const Dev &D, int t, bool prompt, std::vector<ChainOp> &ops) {
    c_ = c;
    w_ = w;
    sms_ = sms;
    for (int s = 2; s <= 8; ++s) clusters_[s] = clusters[s];
    return build(D, t, prompt, ops);
}

bool Chain::select(const Dev &D) {
    auto it = plans_.find(D.B);
    if (it == plans_.end()) {
        if ((int)plans_.size() >= kMaxPlans) plans_.clear();
        std::unique_ptr<StepPlan> p(new StepPlan());
        if (!build(D, D.K1, false, p->ops)) return false;
        for (size_t i = 0; i < p->ops.size(); ++i) p->ops[i].proj.stage = p->ops[i].attn.stage = (int)i;
        it = plans_.emplace(D.B, std::move(p)).first;
    }
    plan_ = it->second.get();
    return true;
}

cudaError_t Chain::run_op(const Dev &D, int i, cudaStream_t st, unsigned long long *count) {
    return run(D, plan_->ops[i], D.K1, ChainLaunch{st, false, count});
}

cudaError_t Chain::step(const Dev &D, cudaStream_t st, bool graph, bool overlap, unsigned long long *count) {
    cudaError_t e;
    if (graph) {
        // a stream that is being captured by the caller takes the kernels themselves
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        if ((e = cudaStreamIsCapturing(st, &cs)) != cudaSuccess) return e;
        if (cs != cudaStreamCaptureStatusNone) graph = false;
    }
    if (!graph) {
        const ChainLaunch L{st, overlap, count};
        for (const ChainOp &op : plan_->ops)
            if ((e = run(D, op, D.K1, L)) != cudaSuccess) return e;
        return cudaSuccess;
    }
    StepPlan &p = *plan_;
    if (!p.exec) {
        if (!record_ && (e = cudaStreamCreateWithFlags(&record_, cudaStreamNonBlocking)) != cudaSuccess) return e;
        if ((e = cudaStreamBeginCapture(record_, cudaStreamCaptureModeThreadLocal)) != cudaSuccess) return e;
        unsigned long long n = 0;
        const ChainLaunch L{record_, true, &n};
        for (const ChainOp &op : p.ops)
            if ((e = run(D, op, D.K1, L)) != cudaSuccess) break;
        const cudaError_t end = cudaStreamEndCapture(record_, &p.graph);
        if (e != cudaSuccess) return e;
        if (end != cudaSuccess) return end;
        if ((e = cudaGraphInstantiate(&p.exec, p.graph, 0)) != cudaSuccess) return e;
        p.kernels = n;
    }
    *count += p.kernels;
    return cudaGraphLaunch(p.exec, st);
}

cudaError_t Chain::condition(const Dev &D, const void *d_cond, cudaStream_t st, unsigned long long *count) {
    struct { TensorMap wk, wv, cond; } m;
    if (!encode(encode_, &m.cond, d_cond, D.dc, D.C, D.B, (size_t)D.C * D.dc * 2, cond_tile(D.C))) return cudaErrorInvalidValue;
    m.wk = kc_;
    m.wv = vc_;
    cudaError_t e = launch_cond_kv(D, &m, D.ckv_pool, D.L, st);
    *count += 1;
    if (e != cudaSuccess || c_.head_kind != 1 || D.K == 0) return e;
    m.wk = head_kc_;
    m.wv = head_vc_;
    *count += 1;
    return launch_cond_kv(D, &m, D.hckv_pool, D.K, st);
}

cudaError_t Chain::ingest(const Dev &D, int n, cudaStream_t st, unsigned long long *count) {
    // chunks of as many positions of every sequence as fit the token rows that the kernels take, of equal length
    const int most = std::max(1, prompt_rows(c_) / D.B), chunks = (n + most - 1) / most, t = (n + chunks - 1) / chunks;
    std::vector<ChainOp> ops;
    if (!build(D, t, true, ops)) return cudaErrorInvalidValue;
    const ChainLaunch L{st, true, count};
    cudaError_t e;
    for (int pos = 0; pos < n; pos += t) {
        for (ChainOp &op : ops) {
            op.attn.pos0 = op.proj.pos0 = pos;
            op.attn.pos_end = op.proj.pos_end = n;
            if ((e = run(D, op, t, L)) != cudaSuccess) return e;
        }
    }
    return cudaSuccess;
}

}  // namespace xsm
