// Host side of the launch chain (xsm_chain.cu), used by the C ABI (xsm_api.cu).
#pragma once
#include "../../include/xsm.h"
#include "xsm_chain.cuh"

#include <map>
#include <memory>
#include <vector>

namespace xsm {

// element offsets of the weight matrices in the caller's buffer
struct WeightOffsets {
    size_t E, gf, W0;
    std::vector<size_t> g1, wq, wo, g2, wqc, wkc, wvc, woc, g3, wgate, wup, wdown, W1, Wout, hq, hk, hv, ho;
    size_t total;
};

struct alignas(64) TensorMap { unsigned char bytes[128]; };
struct WeightMaps { TensorMap w0, w1; };

// one kernel of a chain
struct ChainOp {
    enum Kind { PROJ, FEW, F32, ATTN, TAIL, EMBED } kind;
    WeightMaps maps;
    ProjArgs proj;
    AttnArgs attn;
    int smem;
};

// the kernels of one decoding step of a batch, and their recording
struct StepPlan {
    std::vector<ChainOp> ops;
    unsigned long long kernels = 0;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    ~StepPlan();
};

int prompt_rows(const xsm_model_config &c);      // most token rows of a chunk of a prompt (buffers are sized for them)

class Chain {
  public:
    ~Chain();
    // weight tensor maps; false: the driver has no encoder for them
    bool init(const xsm_model_config &c, const WeightOffsets &w, const char *weights, int sm_count);
    // the kernels of a decoding step for the batch in D (D.B, D.M, D.Mp set); they are kept for later requests
    bool select(const Dev &D);
    // the kernels alone, of a step or of a chunk of t positions of a prompt, on a chip of that many SMs and clusters: no device is needed
    bool plan(const xsm_model_config &c, const WeightOffsets &w, int sms, const int *clusters, const Dev &D, int t, bool prompt, std::vector<ChainOp> &ops);
    void forget();                       // drops what is kept (a launch parameter has changed)
    int n_ops() const { return plan_ ? (int)plan_->ops.size() : 0; }
    // one decoding step; graph: replay the recording (made at the first call)
    cudaError_t step(const Dev &D, cudaStream_t st, bool graph, bool overlap, unsigned long long *count);
    cudaError_t run_op(const Dev &D, int i, cudaStream_t st, unsigned long long *count);
    // keys and values of the condition: of the layers, and of cross-attention decoding heads
    cudaError_t condition(const Dev &D, const void *d_cond, cudaStream_t st, unsigned long long *count);
    // runs prompt tokens 0..n-1 of every sequence through the layers: their keys and values enter the cache
    cudaError_t ingest(const Dev &D, int n, cudaStream_t st, unsigned long long *count);

  private:
    bool weight_map(TensorMap *out, size_t elem_off, int rows, int kdim, int count, size_t stride_elems, int box_rows);
    bool build(const Dev &D, int t, bool prompt, std::vector<ChainOp> &ops);
    void plan_proj(ChainOp &op, int rows, int Mp, int kdim);
    bool plan_few(ChainOp &op, int rows, int Mp, int kdim);
    AttnArgs plan_attn(const Dev &D, bool cross, int sets, int t, int Mp);
    bool own_queries(const Dev &D, AttnArgs &A) const;
    cudaError_t run(const Dev &D, const ChainOp &op, int t, const ChainLaunch &L);

    xsm_model_config c_;
    WeightOffsets w_;
    const char *weights_ = nullptr;
    int sms_ = 0, clusters_[9] = {};      // clusters of s CTAs (with an SM each) that run at a time
    void *encode_ = nullptr;
    TensorMap qkv_, o_, qc_, oc_, gate_, up_, down_, lm_, head_in_, head_o_, head_out_, kc_, vc_, head_kc_, head_vc_;
    std::map<int, std::unique_ptr<StepPlan>> plans_;
    StepPlan *plan_ = nullptr;
    cudaStream_t record_ = nullptr;
};

}  // namespace xsm
