"""The decoding work that is timed: whole calls of the C ABI as a mesh generation service makes them.

A pass is one request: `xsm_prefill` on the condition latents and the prompt, then either `xsm_generate` for a number of
tokens, or `xsm_spec_step` again and again where the caller streams tokens as they come, or both in one call from host
buffers (`xsm_generate_host`).  The shapes are those of `inputs.CONFIGS` with other batches, head counts, lengths of
prompt and output, condition and vocabulary sizes, and every verification and sampling rule.

The weights stand in for a trained model in the one respect that matters to the decoding loop: the next token follows
from the last one with a clear margin, as a trained mesh model's mostly does, and a decoding head is right about a
stated share of the tokens (`accept`).  Matrices inside the blocks are N(0, sigma) as everywhere in this repository.
With independent random output projections instead, every choice would be a near tie between thousands of tokens and
no draft would ever pass, which no user of speculative decoding has.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2507_23777_b200 import binding, inputs

TINY, SMALL, MEDIUM, BATCHED, LARGE = range(5)      # inputs.CONFIGS


def _case(name, model, api="generate", batch=1, draft=4, tokens=128, prompt=1, accept=0.53, **more):
    """accept: share of the tokens that each decoding head predicts rightly; 0.53 for each of four heads gives the
    2.02 tokens a step that the paper reports."""
    c = dict(model=model, api=api, batch=batch, draft=draft, tokens=tokens, prompt=prompt, accept=accept)
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest request: a short sequence from the fp32 parity model, latency of tiny stages
        _case("tiny fp32, 48 tokens", TINY, draft=3, tokens=48),
        # a caller that streams: one xsm_spec_step per iteration, tokens on the device after each
        _case("small, streamed steps", SMALL, api="step", tokens=24),
        # one mesh from the small model, greedy
        _case("small, batch 1", SMALL, tokens=256),
        # two meshes for a caller that holds host buffers, threshold acceptance, odd sizes all round
        _case("small, host buffers, odd sizes", SMALL, api="host", batch=2, draft=3, tokens=99, prompt=37, n_cond=301,
              vocab=5013, verify_mode=2, delta=0.4),
        # the headline: one mesh from the medium model, top-5 acceptance and sampling
        _case("medium, batch 1", MEDIUM, tokens=192),
        # the same model without decoding heads: plain decoding, the baseline that speculation is measured against
        _case("medium, no heads", MEDIUM, draft=0, tokens=96),
        # cross-attention heads (Eq. 3) with the probability tree of the Appendix
        _case("medium, cross-attention heads, tree", MEDIUM, tokens=96, head_kind=1, sample_mode=2, k_sample=4),
        # completion of a long partial mesh: the prompt is read, then decoding goes on at a long context
        _case("medium, prompt of 4000", MEDIUM, tokens=96, prompt=4000),
        # a few meshes at once
        _case("medium, batch 4", MEDIUM, batch=4, tokens=96, prompt=2),
        # the batched configuration: sixteen meshes with their own conditions and ragged accept lengths, from a partial mesh
        _case("medium, batch 16", BATCHED, batch=16, tokens=64, prompt=100),
        # the large model for one mesh and as configured for four
        _case("large, batch 1", LARGE, draft=6, tokens=64),
        _case("large, batch 4", LARGE, batch=4, draft=6, tokens=48, prompt=48),
    ]


def draw(rng):
    """Another request of the same ranges; prompts and outputs are shorter the larger the model and the batch."""
    def log(lo, hi):
        return int(round(lo * (hi / lo) ** rng.random()))

    model = rng.choice([TINY, SMALL, SMALL, MEDIUM, MEDIUM, MEDIUM, LARGE])
    draft = rng.choice([0, 1, 2, 3, 4, 4, 4, 5, 6])
    batch = log(1, {TINY: 5, SMALL: 18, MEDIUM: 18, LARGE: 6}[model])
    if model == TINY:
        batch = max(1, min(batch, 24 // (draft + 1)))
    longest = {TINY: 500, SMALL: 4000, MEDIUM: 3000, LARGE: 500}[model]
    prompt = log(2, max(3, longest // batch)) if batch > 1 or rng.random() < 0.5 else 1
    tokens = log(16, {TINY: 256, SMALL: 256, MEDIUM: 128, LARGE: 48}[model])
    c = _case(None, model, rng.choice(["generate", "generate", "generate", "step", "host"]), batch, draft, tokens, prompt,
              accept=round(0.25 + 0.6 * rng.random(), 2))
    c["n_cond"] = log(40, 600)
    c["vocab"] = log(500, 9000) | 1
    rule = rng.choice(["config", "greedy", "top-k", "threshold", "tree"])
    if rule == "greedy":
        c.update(verify_mode=0, sample_mode=0)
    elif rule == "top-k":
        c.update(verify_mode=1, k_accept=rng.randrange(2, 9), sample_mode=1, k_sample=rng.randrange(2, 33), temperature=0.5)
    elif rule == "threshold":
        c.update(verify_mode=2, delta=round(0.1 + 0.5 * rng.random(), 2))
    elif rule == "tree" and draft <= 5:
        c.update(sample_mode=2, k_sample=4)
    if draft and rng.random() < 0.2:
        c["head_kind"] = 1
    return c


# ---------------------------------------------------------------- the model of a case

_OWN = {"name", "model", "api", "batch", "draft", "tokens", "prompt", "accept"}


def _config(case):
    cfg = inputs.config(case["model"], n_draft=case["draft"], batch=case["batch"])
    cfg.update({k: v for k, v in case.items() if k not in _OWN})
    cfg["max_seq_len"] = case["prompt"] + case["tokens"] + 64
    cfg["eos_id"] = -1
    return cfg


def _successors(V, g):
    """Token -> next token: a random order of the vocabulary, walked round."""
    order = torch.randperm(V, generator=g, device="cuda")
    nxt = torch.empty_like(order)
    nxt[order] = order.roll(-1)
    return nxt


def _weights(cfg, accept, g):
    """Flat weight buffer on the GPU in the order of include/xsm.h, and the map from a token to its successor.  Embeddings
    are large against what the blocks add, and the output projections hold, in the row of a token's successor, a multiple
    of that token's embedding: its logit comes out at about thirty times the deviation of the others."""
    dt = torch.bfloat16 if cfg["dtype"] == 1 else torch.float32
    off = inputs.weight_offsets(cfg)
    buf = torch.empty(off["__total__"][0], dtype=dt, device="cuda")
    buf.normal_(0.0, cfg["sigma"], generator=g)
    V, d, sigma = cfg["vocab"], cfg["d_model"], cfg["sigma"]

    def view(name):
        o, shape = off[name]
        return buf[o:o + int(np.prod(shape))].view(shape)

    for name in off:
        if name.rpartition(".")[2] in ("g1", "g2", "g3", "gf"):
            view(name).fill_(1.0)
    E = torch.randn(V, d, generator=g, device="cuda")
    view("E").copy_(E * 4.0)
    nxt = _successors(V, g)
    gain = 10.0 * sigma / d ** 0.5
    ahead, out = nxt, ["W0"] + [f"h{i}.Wout" for i in range(1, cfg["n_draft"] + 1)]
    for i, name in enumerate(out):
        W = view(name)
        to = ahead
        if i:      # a head is wrong about the rest: it names some other token
            wrong = torch.rand(V, generator=g, device="cuda") >= accept
            to = torch.where(wrong, ahead.roll(1), ahead)
        rows = torch.zeros(V, d, device="cuda").index_add_(0, to, E)
        W.copy_((W.float() + gain * rows) * cfg["out_scale"])
        ahead = nxt[ahead]
    return buf, nxt


class _Request:
    """A service's state: the bound model, the inputs of one request and room for its outputs."""

    def __init__(self, case, seed):
        cfg = self.cfg = _config(case)
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)
        B, P, T, K1 = case["batch"], case["prompt"], case["tokens"], case["draft"] + 1
        self.case, self.batch, self.prompt_len, self.tokens = case, B, P, T
        self.weights, nxt = _weights(cfg, case["accept"], g)
        cond = torch.randn(B, cfg["n_cond"], cfg["d_cond"], generator=g, device="cuda").to(self.weights.dtype)
        prompt = torch.zeros(B, P, dtype=torch.int32)
        walk, nxt = torch.randint(1, cfg["vocab"], (B,), generator=g, device="cuda").cpu(), nxt.cpu()
        for p in range(1, P):
            prompt[:, p] = walk
            walk = nxt[walk]
        self.lib = binding.load()
        mc, self.dc = binding.model_config(cfg, B), binding.decode_config(dict(cfg, seed=cfg["seed"] + seed))
        n = binding.xsm_workspace_bytes(mc)
        self.workspace = torch.empty(n, dtype=torch.uint8, device="cuda")
        self.handle = ctypes.c_void_p()
        self.check(self.lib.xsm_create(ctypes.byref(mc), self.weights.data_ptr(), self.workspace.data_ptr(), n,
                                       torch.cuda.current_stream().cuda_stream, ctypes.byref(self.handle)))
        self.stats = binding.Stats()
        if case["api"] == "host":
            self.cond, self.prompt = cond.cpu().pin_memory(), prompt.pin_memory()
            self.out, self.lengths = torch.empty(B, T, dtype=torch.int32).pin_memory(), torch.empty(B, dtype=torch.int32).pin_memory()
        else:
            self.cond, self.prompt = cond, prompt.cuda()
            self.lengths = torch.empty(B, dtype=torch.int32, device="cuda")
            self.out = torch.empty(B, T, dtype=torch.int32, device="cuda")
            if case["api"] == "step":      # one row of committed tokens and their number for every step
                self.out = torch.empty(_steps(case), B, K1, dtype=torch.int32, device="cuda")
                self.lengths = torch.empty(_steps(case), B, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()

    def check(self, status):
        if status != binding.XSM_OK:
            raise binding.XsmError(status, self.lib.xsm_last_error(self.handle or None).decode())

    def __del__(self):
        if getattr(self, "handle", None):
            self.lib.xsm_destroy(self.handle)


def prepare(case, seed):
    return _Request(case, seed)


def run(s):
    if s.case["api"] == "host":
        s.check(s.lib.xsm_generate_host(s.handle, s.batch, s.cond.data_ptr(), s.prompt.data_ptr(), s.prompt_len, ctypes.byref(s.dc),
                                        s.tokens, s.out.data_ptr(), s.lengths.data_ptr(), ctypes.byref(s.stats)))
    else:
        s.check(s.lib.xsm_prefill(s.handle, s.batch, s.cond.data_ptr(), s.prompt.data_ptr(), s.prompt_len, ctypes.byref(s.dc)))
        if s.case["api"] == "step":
            for i in range(s.out.shape[0]):
                s.check(s.lib.xsm_spec_step(s.handle, s.out[i].data_ptr(), s.lengths[i].data_ptr()))
            return {"tokens": s.out, "lengths": s.lengths}
        s.check(s.lib.xsm_generate(s.handle, s.tokens, s.out.data_ptr(), s.lengths.data_ptr(), ctypes.byref(s.stats)))
    return {"tokens": s.out, "lengths": s.lengths, "steps": int(s.stats.steps), "accepted": [int(n) for n in s.stats.accept_hist]}


def _steps(case):
    """Decoding steps of a pass, from the heads' share of right drafts: a step commits 1 + p + p^2 + ... tokens."""
    a, K = case["accept"], case["draft"]
    return math.ceil(case["tokens"] / sum(a ** i for i in range(K + 1)))


def work(case):
    """Weights once for the prompt and once for every step, the cache once for every step, in the model's data type; the
    multiplications of every prompt token and of every row of a step's window."""
    c, B, K, T, P = _config(case), case["batch"], case["draft"], case["tokens"], case["prompt"]
    L, d, f, V, C, dc, e = c["n_layers"], c["d_model"], c["d_ff"], c["vocab"], c["n_cond"], c["d_cond"], 2 if c["dtype"] == 1 else 4
    steps, rows = _steps(case), B * (K + 1)
    layers = L * (6 * d * d + 3 * d * f)
    ca = c.get("head_kind", 0) == 1
    tail = V * d + K * ((2 if ca else 1) * d * d + V * d)
    sets = L + (K if ca else 0)
    weights = layers + tail
    cond_kv = 2 * sets * C * d * B
    context = P + T / 2
    bytes_ = e * (2 * sets * d * dc + B * C * dc + cond_kv)                       # keys and values of the condition
    bytes_ += e * steps * (weights + cond_kv + 2 * L * d * B * context)
    flops = 2 * B * C * 2 * sets * d * dc + 2 * steps * rows * weights + 4 * d * L * steps * rows * (context + C)
    if P > 1:
        bytes_ += e * (layers + 2 * L * d * B * P)
        flops += 2 * B * (P - 1) * layers + 4 * d * L * B * (P - 1) * (P / 2 + C)
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    return "exact"
