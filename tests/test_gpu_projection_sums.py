"""How much the tensor cores' sums lose.  An instruction adds sixteen products to an accumulator and cuts off what lies below its last
bit, so the error grows with the number of instructions that one accumulator takes.  Here all products are positive and near 1, with
few bits (two mantissas of eight): sixteen instructions add them up to about 2^8 and lose next to nothing, 128 lose three bits of each."""
import numpy as np
import pytest

from paper_2507_23777_b200 import inputs

pytestmark = pytest.mark.gpu

UNIT = 2.0 ** -23


def _relative_error(width, vocab, rows):
    """Mean relative error of the logits W0 g of `rows` sequences, with all of W0 and g positive and nothing else in the model."""
    import torch
    assert torch.cuda.is_available(), "this test needs a B200"
    from paper_2507_23777_b200 import binding, build
    build.build()
    cfg = inputs.config(2, d_model=width, n_heads=width // 64, d_head=64, d_ff=256, d_cond=32, head_hidden=width, n_draft=0, n_layers=1,
                        vocab=vocab, n_cond=8, max_seq_len=48)
    off = inputs.weight_offsets(cfg)
    w = np.zeros(off["__total__"][0], dtype=np.uint16)
    rng = np.random.default_rng(7)
    for name, (o, shape) in off.items():
        n = int(np.prod(shape))
        if name in ("E", "W0"):
            w[o:o + n] = inputs.f32_to_bf16_bits(rng.uniform(0.5, 1.5, n).astype(np.float32))
        elif name.endswith(("g1", "g2", "g3", "gf")):
            w[o:o + n] = inputs.f32_to_bf16_bits(rng.uniform(0.9, 1.1, n).astype(np.float32))
    ctx = binding.Context(cfg, w, max_batch=rows)
    prompt = rng.integers(0, vocab, (rows, 1))
    ctx.prefill(inputs.make_cond(cfg, rows), prompt, binding.decode_config(cfg))
    ctx.step()
    z = ctx.xsm_debug_get_logits()[0][:, 0].astype(np.float64)
    ctx.xsm_destroy()

    def view(name):
        return inputs.bf16_bits_to_f32(inputs.tensor_view(cfg, w, name)).astype(np.float64)

    x = view("E")[prompt[:, 0]]
    g = x / np.sqrt((x * x).mean(1, keepdims=True) + cfg["rms_eps"]) * view("gf")
    ref = g @ view("W0").T
    return float((np.abs(z - ref) / ref).mean())


@pytest.mark.parametrize("width,vocab,rows", [(2048, 16500, 1), (2048, 16500, 16), (1024, 16500, 5), (1024, 9000, 8)])
def test_sums_of_few_token_rows(width, vocab, rows):
    """Up to sixteen token rows an accumulator takes sixteen instructions; what is left is the rounding of 1/rms, of the lo parts and of
    the sums of the parts, half a unit each at most and in both directions (0.4 to 0.5 units; 1.9 to 20 with one accumulator)."""
    assert _relative_error(width, vocab, rows) < UNIT


@pytest.mark.parametrize("width", [1024, 2048])
def test_cutting_token_rows_does_not_lengthen_the_sums(width):
    """From 49 token rows on these are cut into parts and the columns into fewer: no worse than 48 rows, whose columns are cut as far as
    they can be (within half a unit; 1.6 and 5.5 units worse with one accumulator)."""
    whole = _relative_error(width, 3000, 48)
    for rows in (49, 80, 96, 128):
        assert _relative_error(width, 3000, rows) < whole + UNIT / 2, rows
