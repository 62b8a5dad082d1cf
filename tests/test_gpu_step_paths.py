"""GPU parity on both sides of the lines at which a decoding step changes path: mma.sync or tcgen05 projections, several accumulators
or one, token rows dealt out one by one or in fours and cut into parts, warps of a projection, the tail's rows of logits and its choice of the best tokens, and the token
rows that fp32 kernels fold together."""
import numpy as np
import pytest

from paper_2507_23777_b200 import inputs

pytestmark = pytest.mark.gpu

BF16_TOL = dict(atol=2e-2, rtol=1e-2)      # the bound of every bf16 parity test: 2e-2 + 1e-2 |logit|
F32_TOL = dict(atol=2e-4, rtol=2e-4)


def _model(d=256, H=4, dh=64, f=512, K=4, V=777, C=40, **kw):
    return dict(d_model=d, n_heads=H, d_head=dh, d_ff=f, d_cond=d, head_hidden=d, n_draft=K, n_layers=1, vocab=V, n_cond=C,
                sigma=0.02 * (1024 / d) ** 0.5, **kw)


def _pick(k):
    return dict(verify_mode=1, k_accept=3, sample_mode=1, k_sample=k, temperature=0.8)


# model, sequences
SHAPES = {
    "three token rows, width 768": (_model(768, 12, f=3072, K=2), 1),
    "three token rows, width 896": (_model(896, 14, f=1024, K=2), 1),
    "four token rows, width 768": (_model(768, 12, f=3072, K=3), 1),
    "five token rows, width 1792: rings that fill the shared memory of a CTA": (_model(1792, 28, f=4096, K=4), 1),
    "four token rows, width 640": (_model(640, 10, f=2560, K=3), 1),
    "four token rows, width 512, tcgen05 for the down projection": (_model(512, 8, f=4096, K=3), 1),
    "five token rows, width 128": (_model(128, 2, K=4), 1),
    "eight token rows, width 128, tcgen05 for the down projection": (_model(128, 4, 32, 2048, K=7), 1),
    "nine token rows, width 128": (_model(128, 4, 32, 1024, K=2), 3),
    "sixteen token rows, width 128": (_model(128, 2, K=3), 4),
    "seventeen token rows, width 128": (_model(128, 2, K=0), 17),
    "five token rows, width 128, cross-attention heads": (_model(128, 2, K=4, head_kind=1), 1),
    "fifteen token rows, width 128, cross-attention heads": (_model(128, 2, K=4, head_kind=1), 3),
    "two token rows, width 2048": (_model(2048, 16, 128, 2048, K=1), 1),
    "five token rows over eight CTAs": (_model(1024, 16, f=4096, K=4), 1),
    "sixteen token rows, width 2048, four accumulators": (_model(2048, 16, 128, 2048, K=3, V=1500), 4),
    "seventeen token rows, width 2048, one accumulator": (_model(2048, 16, 128, 2048, K=0, V=1500), 17),
    "eight token rows, two to a CTA": (_model(1792, 28, f=2048, K=7), 1),
    "sixteen token rows over eight CTAs, two to a CTA": (_model(1024, 16, f=4096, K=3), 4),
    "sixteen token rows, the accumulator in two parts, warps apart": (_model(512, 8, f=512, K=3), 4),
    "sixteen token rows, width 2048, eight accumulators without a cluster": (_model(2048, 16, 128, 4864, K=3, V=1500), 4),
    "two token rows, width 1024": (_model(1024, 16, f=4096, K=1), 1),
    "twenty-four token rows": (_model(512, 8, K=5), 4),
    "twenty-five token rows": (_model(512, 8, K=4), 5),
    "forty-eight token rows": (_model(512, 8, K=5), 8),
    "forty-nine token rows": (_model(512, 8, K=6), 7),
    "eighty token rows, width 1024": (_model(1024, 16, f=2048, K=4), 16),
    "all rows of logits, one CTA to an SM": (_model(V=8001, **_pick(5)), 1),
    "rows of logits one after the other": (_model(V=12003, **_pick(5)), 2),
    "rows of logits in place": (_model(V=52001, K=1, **_pick(5)), 1),
    "no drafts, a row of logits of 180 KB": (_model(V=46002, K=0, **_pick(3)), 1),
    "two candidates": (_model(V=1001, **_pick(2)), 2),
    "three candidates of thirty tokens": (_model(V=30, **_pick(3)), 2),
    "sixteen candidates": (_model(V=1003, **_pick(16)), 2),
    "seventeen candidates": (_model(V=1003, **_pick(17)), 2),
    "fp32, three token rows": (_model(K=2, dtype=0), 1),
    "fp32, eight token rows": (_model(K=3, dtype=0), 2),
    "fp32, nine token rows": (_model(K=2, dtype=0), 3),
}


MMA, UMMA, ANY = {1}, {0}, None
QKV, RESIDUAL, CROSS_Q, GATE_UP, LOGITS = 0, 1, 2, 3, 4
# What a shape is there for: kinds of its projections; (what one does, threads, token rows of a tile, token rows that a CTA finishes,
# columns of tensor memory), on every chip of 148 SMs however its GPCs are cut
SELECTS = {
    "three token rows, width 768": (MMA,),
    "three token rows, width 896": (UMMA,),
    "four token rows, width 768": (UMMA,),
    "four token rows, width 640": (MMA,),
    "four token rows, width 512, tcgen05 for the down projection": (MMA | UMMA, (RESIDUAL, 256, 8, 1, 32)),
    "eight token rows, width 128, tcgen05 for the down projection": (MMA | UMMA, (RESIDUAL, 256, 8, 1, 32)),
    "nine token rows, width 128": (MMA,),
    "sixteen token rows, width 128": (MMA,),
    "seventeen token rows, width 128": (UMMA,),
    "two token rows, width 2048": (UMMA, (QKV, 256, 8, 1, 64), (RESIDUAL, 256, 8, 1, 32), (CROSS_Q, 256, 8, 1, 32), (GATE_UP, 256, 8, 1, 32),
                                   (LOGITS, 256, 8, 1, 32)),
    "five token rows over eight CTAs": (UMMA, (RESIDUAL, 256, 8, 1, 32), (GATE_UP, 384, 8, 3, 32)),
    "sixteen token rows, width 2048, four accumulators": (UMMA, (QKV, 384, 16, ANY, 128)),
    "seventeen token rows, width 2048, one accumulator": (UMMA, (QKV, 384, 24, ANY, 64)),
    "eight token rows, two to a CTA": (UMMA, (GATE_UP, 256, 8, 2, 32)),
    "sixteen token rows over eight CTAs, two to a CTA": (UMMA, (RESIDUAL, 384, 16, 2, 32)),
    "sixteen token rows, the accumulator in two parts, warps apart": (UMMA, (GATE_UP, 256, 16, 2, 32)),
    "sixteen token rows, width 2048, eight accumulators without a cluster": (UMMA, (GATE_UP, 512, 16, 16, 256)),
    "twenty-four token rows": (UMMA, (QKV, 384, 24, 3, 64)),
    "twenty-five token rows": (UMMA, (QKV, 384, 32, 4, 64)),
    "forty-eight token rows": (UMMA, (QKV, 384, 48, 8, 128)),
    "forty-nine token rows": (UMMA, (RESIDUAL, 384, 8, 4, 32), (GATE_UP, 384, 16, 4, 64)),
    "eighty token rows, width 1024": (UMMA, (RESIDUAL, 384, 24, 8, 128), (GATE_UP, 384, 40, 20, 256)),
}


def check_what_is_selected(shape, **chip):
    """The plan of the step (of the current device, or of the chip that is told) has what the shape is there for."""
    from paper_2507_23777_b200 import binding
    over, batch = SHAPES[shape]
    cfg = inputs.config(2, **over)
    cfg["max_seq_len"] = 48
    rows = [[int(v) for v in r] for r in binding.xsm_debug_plan(binding.model_config(cfg, batch), batch, **chip)]
    kinds, *wanted = SELECTS[shape]
    assert {r[0] for r in rows if r[0] < 3} == kinds
    found = [(r[1], r[2], r[4], r[5], r[6]) for r in rows if r[0] == 0]
    for w in wanted:
        assert any(all(a in (ANY, b) for a, b in zip(w, f)) for f in found), (w, found)


@pytest.mark.parametrize("shape", list(SHAPES))
def test_step_against_the_oracle(shape):
    import torch
    assert torch.cuda.is_available(), "this test needs a B200"
    from paper_2507_23777_b200 import build
    build.build()
    import parity
    if shape in SELECTS:
        check_what_is_selected(shape)
    over, batch = SHAPES[shape]
    cfg = inputs.config(2, **over)
    cfg["max_seq_len"] = 48
    tol = F32_TOL if cfg["dtype"] == 0 else BF16_TOL
    ls = parity.LockStep(cfg, batch=batch)
    ls.begin([0, 3, 7])
    for _ in range(2):
        ls.step(**tol)
    ls.compare_cache(**tol)
    ls.close()


@pytest.mark.parametrize("vocab", [400, 5001])
def test_equal_logits_rank_by_token(vocab):
    """Output projections of zeros make every logit equal: the best tokens are then the first ones, whether they fit the list of
    those that may be among the best (400) or not (5001)."""
    import torch
    assert torch.cuda.is_available(), "this test needs a B200"
    from paper_2507_23777_b200 import binding, build
    build.build()
    cfg = inputs.config(2, **_model(V=vocab, **_pick(5)))
    cfg["max_seq_len"] = 64
    w = inputs.make_weights(cfg)
    off = inputs.weight_offsets(cfg)
    for name in ["W0"] + [f"h{i}.Wout" for i in range(1, cfg["n_draft"] + 1)]:
        o, shape = off[name]
        w[o:o + int(np.prod(shape))] = 0
    ctx = binding.Context(cfg, w)
    ctx.prefill(inputs.make_cond(cfg, 1), [0], binding.decode_config(cfg))
    toks, lens, _ = ctx.generate(40)
    assert lens[0] == 40 and toks[0].min() >= 0
    assert toks[0].max() < 5 and len(set(toks[0].tolist())) > 1      # five candidates with equal weights
    ctx.xsm_destroy()
