"""The tail where its rows of logits do not all fit shared memory, under every rule of verification and sampling, and its choice of the
best tokens where logits are infinite or not numbers."""
import numpy as np
import pytest

from paper_2507_23777_b200 import inputs

pytestmark = pytest.mark.gpu

BF16_TOL = dict(atol=2e-2, rtol=1e-2)      # the bounds of every parity test
F32_TOL = dict(atol=2e-4, rtol=2e-4)


def _model(V, K, d=256, **kw):
    return dict(d_model=d, n_heads=d // 64, d_head=64, d_ff=512, d_cond=d, head_hidden=d, n_draft=K, n_layers=1, vocab=V, n_cond=40,
                sigma=0.02 * (1024 / d) ** 0.5, max_seq_len=64, **kw)


# vocabulary, drafts: (K + 2) rows of 4 V bytes are more than 200 KB, or one is
ROWS = {"one after the other": (12003, 4), "one after the other, ten CTAs to a sequence": (12003, 9), "in place": (52001, 2)}
RULES = {
    "threshold": dict(verify_mode=2, delta=0.03, sample_mode=1, k_sample=5, temperature=0.5),
    "greedy": dict(verify_mode=0, sample_mode=0),
    "top-3, seventeen candidates": dict(verify_mode=1, k_accept=3, sample_mode=1, k_sample=17, temperature=0.5),
    "tree": dict(verify_mode=1, k_accept=3, sample_mode=2, k_sample=2, temperature=0.5),
}


@pytest.mark.parametrize("dtype", [1, 0])
@pytest.mark.parametrize("rule", list(RULES))
@pytest.mark.parametrize("rows", list(ROWS))
def test_rules_with_rows_that_do_not_fit(rows, rule, dtype):
    import torch
    assert torch.cuda.is_available(), "this test needs a B200"
    from paper_2507_23777_b200 import build
    build.build()
    import parity
    from test_gpu_parity import planted_chain
    V, K = ROWS[rows]
    cfg = inputs.config(2, **_model(V, K, dtype=dtype, **RULES[rule]))
    tol = F32_TOL if dtype == 0 else BF16_TOL
    ls = parity.LockStep(cfg, batch=2)
    ls.begin([0, 5])
    accepted = []
    for it in range(3):      # drafts of which some pass, in the first sequence none, one, ..
        drafts = ls.ctx.xsm_debug_get_state()["window"][:, 1:].copy()
        for b in range(2):
            drafts[b] = planted_chain(ls, b, min(K, it + b), rank=0)
        accepted += ls.step(drafts=drafts, margin=1e-3 if dtype == 0 else 1e-2, **tol)[1]
    assert max(accepted) >= 1 and min(accepted) < K, accepted
    ls.compare_cache(**tol)
    ls.close()


def _ranked(z):
    """Tokens by logit, larger first, then by token: bit patterns as the kernels order them (-0 as 0, NaN by its sign and bits)."""
    u = (z + np.float32(0)).view(np.uint32)
    key = np.where(u >> 31, ~u, u | np.uint32(1 << 31)).astype(np.uint64)
    return np.lexsort((np.arange(z.size), np.uint64(1 << 32) - key))


@pytest.mark.parametrize("dtype", [1, 0])
@pytest.mark.parametrize("vocab", [400, 5001])
@pytest.mark.parametrize("k", [3, 16, 17])
@pytest.mark.parametrize("what", ["one infinite", "some infinite", "most infinite", "not a number", "two finite"])
def test_logits_that_are_not_finite(what, k, vocab, dtype):
    """With an infinite or undefined best logit every weight is undefined, no share of their sum is ever passed, and the last of the k
    best is drawn; minus infinity (a masked token) has no weight."""
    import torch
    assert torch.cuda.is_available(), "this test needs a B200"
    from paper_2507_23777_b200 import binding, build
    build.build()
    cfg = inputs.config(2, **_model(vocab, 0, dtype=dtype, verify_mode=1, k_accept=1, sample_mode=1, k_sample=k, temperature=0.5))
    off = inputs.weight_offsets(cfg)
    w = np.zeros(off["__total__"][0], dtype=np.float32)
    rng = np.random.default_rng(5)

    def view(name):
        o, shape = off[name]
        return w[o:o + int(np.prod(shape))].reshape(shape)

    view("E")[:] = rng.uniform(0.5, 1.5, view("E").shape)
    for name in ("l0.g1", "l0.g2", "l0.g3", "gf"):
        view(name)[:] = 1.0
    W0 = view("W0")
    W0[:] = rng.normal(0.0, 0.01, W0.shape)
    some = rng.permutation(vocab)
    if what == "one infinite":
        W0[some[0]] = 3e38
    elif what == "some infinite":
        W0[some[:k - 1]] = 3e38
        W0[some[k:k + 20]] = -3e38
    elif what == "most infinite":
        W0[some[:vocab * 3 // 4]] = 3e38
    elif what == "not a number":
        W0[some[:2], 7] = np.nan
        W0[some[2:9]] = 3e38
    else:
        W0[some[2:]] = -3e38
        W0[some[:2]] = 0.01
    if dtype == 1:
        bits = inputs.f32_to_bf16_bits(np.nan_to_num(w))
        bits[np.isnan(w)] = 0x7FC0
        w = bits
    ctx = binding.Context(cfg, w, max_batch=1)
    ctx.prefill(inputs.make_cond(cfg, 1), [3], binding.decode_config(cfg))
    token = int(ctx.step()[0][0][0])
    z = ctx.xsm_debug_get_logits()[0][0, 0]
    ctx.xsm_destroy()
    assert np.isfinite(z).sum() < vocab
    if what == "two finite":
        assert np.isfinite(z).sum() == 2 and token in some[:2]
    else:
        assert not np.isfinite(z[_ranked(z)[0]]) and token == _ranked(z)[k - 1]
