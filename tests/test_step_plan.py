"""How a step is cut over the chip: plans alone, no GPU."""
import pytest

import test_gpu_step_paths as paths
from paper_2507_23777_b200 import binding, build, inputs

SMS, CLUSTERS = 148, [0, 0, 74, 45, 33, 26, 22, 15, 15]      # a B200's
UMMA = 0
KIND, DOES, THREADS, CTAS, TOK, ROWS, COLUMNS, SMEM = range(8)


@pytest.fixture(scope="module", autouse=True)
def lib():
    build.build()


def plan(d, f, K, batch, prompt=0, clusters=CLUSTERS, **more):
    cfg = inputs.config(2, d_model=d, n_heads=d // 64, d_head=64, d_ff=f, d_cond=d, head_hidden=d, n_draft=K, n_layers=2, vocab=777, n_cond=40,
                        max_seq_len=512, **more)
    return binding.xsm_debug_plan(binding.model_config(cfg, batch), batch, prompt, SMS, clusters)


def _steps():
    for d in (128, 256, 384, 640, 768, 1024, 1280, 1664, 1792, 2048):
        for f in (128, 512, 1024, 2048, 4096, 8192):
            for K, batch in [(0, n) for n in range(1, 129, 5)] + [(3, 4), (4, 1), (4, 16), (5, 9), (7, 16)]:
                yield d, f, K, batch, 0
            for prompt in (8, 31, 130, 400):
                yield d, f, 4, 1, prompt


def test_cluster_projections_never_want_more_tensor_memory_than_the_sm_has():
    """An SM has 228 KB of shared memory and 512 columns of tensor memory.  A projection's CTA holds its columns while it waits for its
    cluster to have some too, so clusters of two streams could wait for each other for good if the CTAs that fit an SM's shared memory
    wanted more columns than there are."""
    seen = set()
    for case in _steps():
        stages = plan(*case)
        assert len(stages) > 0, case
        for s in stages:
            if s[KIND] == UMMA and s[CTAS] > 1:
                assert s[COLUMNS] * 228 * 1024 <= s[SMEM] * 512, (case, s)
                assert s[SMEM] <= 228 * 1024
                seen.add(int(s[COLUMNS]))
    assert seen == {32, 64, 128, 256}


def test_there_is_no_plan_for_what_is_refused():
    assert len(plan(128, 128, 4, 1)) == 2 * 7 + 3     # two layers, three kernels behind them
    assert len(plan(128, 128, 4, 26)) == 0            # 130 token rows
    assert len(plan(128, 100, 4, 1)) == 0             # d_ff no multiple of 128
    assert len(plan(128, 128, 4, 1, 100000)) == 0     # a prompt beyond the room
    assert len(plan(128, 128, 4, 8, dtype=0)) == 0    # fp32: 40 token rows


@pytest.mark.parametrize("shape", list(paths.SELECTS))
def test_shapes_of_the_step_paths_select_what_they_are_named_for(shape):
    paths.check_what_is_selected(shape, sms=SMS, clusters=CLUSTERS)
