"""GPU parity at the sizes where the kernels of the launch chain change path or meet the edge of a tile."""
import numpy as np
import pytest

from paper_2507_23777_b200 import inputs

pytestmark = pytest.mark.gpu

BF16_TOL = dict(atol=2e-2, rtol=1e-2)
F32_TOL = dict(atol=2e-4, rtol=2e-4)


def _model(d=512, H=8, dh=64, f=1024, K=4, L=1, V=777, C=40, **kw):
    return dict(d_model=d, n_heads=H, d_head=dh, d_ff=f, d_cond=d, head_hidden=d, n_draft=K, n_layers=L, vocab=V, n_cond=C,
                sigma=0.02 * (1024 / d) ** 0.5, **kw)


# model, sequences, tokens of the prompt
SHAPES = {
    # projections: mma.sync up to four token rows at this width, tensor cores from five on; accumulators of four blocks up to sixteen
    # rows, of all blocks behind; tiles and remainders of token rows, these cut into parts from 49 on
    "one token row": (_model(K=0), 1, 1),
    "four token rows": (_model(K=3), 1, 1),
    "nine token rows": (_model(K=2), 3, 1),
    "seventeen token rows": (_model(K=0), 17, 1),
    "thirty-three token rows, width 640": (_model(640, 10, 64, 1280, K=2), 11, 1),
    "ninety-six token rows": (_model(K=5), 16, 1),
    "ninety-seven token rows": (_model(K=0), 97, 1),
    "a hundred and twenty-eight token rows, width 1024": (_model(1024, 16, 64, 2048, K=7), 16, 1),
    # prompts: tiles of 128 token rows, the second chunk of 2048 rows
    "prompt of 130": (_model(), 1, 130),
    "prompts of 90": (_model(), 3, 90),
    "prompt of 2100": (_model(256, 4, 64, 512), 1, 2100),
    # (a ring of two slots of activations, refilled ten times in the down projection)
    "prompt of 1100, 128 blocks of columns": (_model(256, 4, 64, 8192), 1, 1100),
    # queries projected by the cross-attention: one key tile, odd counts, keys cut over CTAs, keys that do not fit at once
    "16 condition latents": (_model(1024, 16, 64, 1024, C=16), 1, 1),
    "257 condition latents, three sequences": (_model(1024, 16, 64, 1024, K=2, C=257), 3, 1),
    "700 condition latents": (_model(1024, 16, 64, 1024, C=700), 1, 1),
    "1500 condition latents, heads of 32": (_model(256, 8, 32, 512, C=1500), 1, 1),
    "heads of 128, 600 condition latents": (_model(1024, 8, 128, 1024, C=600), 1, 1),
    "width 1280": (_model(1280, 20, 64, 1280, C=129), 1, 1),
    # keys cut over a cluster: fewer rows than CTAs, more rows than CTAs take part, tiles of 16 rows
    "one row, 1300 keys": (_model(K=0), 1, 1300),
    "eight rows, 2000 keys at room for 2700": (_model(256, 4, 64, 512, K=7, room=2700), 1, 2000),
    "five rows of two sequences, 600 keys, heads of 128": (_model(512, 4, 128, 512), 2, 600),
    "ten rows, 500 keys": (_model(K=9), 1, 500),
    # the tail: a vocabulary that is no multiple of anything, as many candidates as there can be
    "64 candidates": (_model(V=1001, verify_mode=1, k_accept=7, sample_mode=1, k_sample=64, temperature=0.9), 2, 1),
    # fp32: rows and keys beyond one chunk
    "fp32, twenty-four token rows": (_model(256, 4, 64, 512, K=3, dtype=0), 6, 1),
    "fp32, prompt of 150": (_model(256, 4, 64, 512, K=3, dtype=0), 1, 150),
}


@pytest.mark.parametrize("shape", list(SHAPES))
def test_chain_against_the_oracle(shape):
    import torch
    assert torch.cuda.is_available(), "this test needs a B200"
    from paper_2507_23777_b200 import build
    build.build()
    import parity
    over, batch, n_prompt = SHAPES[shape]
    over = dict(over)
    room = over.pop("room", n_prompt + 40)
    cfg = inputs.config(2, **over)
    cfg["max_seq_len"] = room
    tol = F32_TOL if cfg["dtype"] == 0 else BF16_TOL
    ls = parity.LockStep(cfg, batch=batch)
    ls.begin([0] + [int(t) for t in np.random.default_rng(3).integers(1, cfg["vocab"], n_prompt - 1)])
    for _ in range(2):
        ls.step(**tol)
    ls.compare_cache(**tol)
    ls.close()
