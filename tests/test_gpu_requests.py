"""How a request ends and what its caller is told, on the hand-sized model."""
import numpy as np
import pytest

from conftest import gpu_cfg
from paper_2507_23777_b200 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def binding():
    import torch
    assert torch.cuda.is_available(), "these tests need a B200"
    from paper_2507_23777_b200 import binding, build
    build.build()
    return binding


@pytest.mark.parametrize("dtype", [0, 1])
def test_generate_reports_a_wait_that_ran_out_and_launches_no_more_steps(binding, dtype):
    """A single stage launched out of turn gives up after a shortened limit and raises the status word.  xsm_generate then
    says XSM_ERR_TIMEOUT, after the two steps that it has on their way at a time and not after all of the sixty that the
    request could take; so does every further call that synchronises, until the next prefill, which starts clean."""
    cfg = gpu_cfg(dtype=dtype, n_draft=2, sigma=0.05, max_seq_len=128)
    w = inputs.make_weights(cfg, random_gains=True)
    cond = inputs.make_cond(cfg, 1)
    dc = binding.decode_config(cfg)
    ctx = binding.Context(cfg, w)
    ctx.prefill(cond, [0], dc)
    want, _, _ = ctx.generate(60)
    ctx.prefill(cond, [0], dc)
    before = ctx.xsm_kernel_launches()
    ctx.xsm_spec_step()
    step = ctx.xsm_kernel_launches() - before
    ctx.xsm_debug_set_wait_limits(3000, 0)
    ctx.xsm_debug_launch_stage(2)
    ctx.xsm_debug_set_wait_limits(0, 0)
    before = ctx.xsm_kernel_launches()
    with pytest.raises(binding.XsmError) as e:
        ctx.generate(60)
    assert e.value.status == binding.XSM_ERR_TIMEOUT
    assert ctx.xsm_kernel_launches() - before <= 3 * step
    for call in (lambda: ctx.generate(60), lambda: ctx.xsm_debug_set_drafts([[1, 2]]), lambda: ctx.xsm_debug_set_script([[1] * 8], 1.0)):
        with pytest.raises(binding.XsmError) as e:
            call()
        assert e.value.status == binding.XSM_ERR_TIMEOUT
    toks, lens = np.zeros((1, 60), dtype=np.int32), np.zeros(1, dtype=np.int32)
    ctx.xsm_generate_host(ctx.cond_to_host(cond), np.zeros((1, 1), dtype=np.int32), dc, 60, toks, lens)
    assert lens[0] == 60 and np.array_equal(toks, want)
    ctx.xsm_destroy()


def capture(ctx, stream, calls):
    """The kernels that `calls` enqueues on the context's stream, as a graph; they do not run."""
    import torch
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        calls()
    return g


@pytest.mark.parametrize("dtype", [0, 1])
def test_a_captured_prefill_begins_a_request_at_every_replay(binding, dtype):
    """A caller captures its prefill and the first steps and replays the graph for one request after another, each of which
    xsm_generate finishes: the same tokens, lengths and counts every time.  A prefill and a request in between that are not
    captured change nothing."""
    import torch
    cfg = gpu_cfg(dtype=dtype, n_draft=2, sigma=0.05)
    w = inputs.make_weights(cfg, random_gains=True)
    cond = inputs.make_cond(cfg, 2)
    dc = binding.decode_config(cfg)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        ctx = binding.Context(cfg, w, max_batch=2)
        d_cond = ctx.cond_to_device(cond)
        d_prompt = torch.tensor([[0, 7, 9], [0, 3, 4]], dtype=torch.int32, device="cuda")

        def begin():
            ctx.xsm_prefill(d_cond, d_prompt, 3, dc)
            ctx.xsm_spec_step()
            ctx.xsm_spec_step()

        begin()
        want, _, want_st = ctx.generate(24)
        g = capture(ctx, stream, begin)
        for i in range(4):
            if i == 2:
                begin()
                ctx.generate(12)
            g.replay()
            toks, lens, st = ctx.generate(24)
            assert (lens == 24).all() and np.array_equal(toks, want), f"replay {i}"
            assert st.tokens == 48 and st.steps == want_st.steps, f"replay {i}"
        ctx.xsm_destroy()


@pytest.mark.parametrize("dtype", [0, 1])
def test_parameters_that_were_only_captured_count_as_not_stored(binding, dtype):
    """Scripted drafts are switched off in a graph that has not run yet: the next direct call still has to switch them off.
    The graph, replayed in a request with another seed, switches the script off and leaves the rest of the request's
    parameters alone.  A captured step brings the store of its own limit, a direct one behind a prefill needs none."""
    import torch
    K, T = 3, 60
    cfg = gpu_cfg(dtype=dtype, n_draft=K, sigma=0.3, max_seq_len=128, verify_mode=1, k_accept=2, sample_mode=1, k_sample=3, temperature=0.8)
    w = inputs.make_weights(cfg, random_gains=True)
    cond = inputs.make_cond(cfg, 1)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        ctx = binding.Context(cfg, w)
        script = np.tile(np.arange(T + K + 2, dtype=np.int32) % cfg["vocab"], (1, 1))

        def scripted(seed):
            ctx.prefill(cond, [0], binding.decode_config(dict(cfg, seed=seed)))
            ctx.xsm_debug_set_script(script, 1.0)

        def run(seed):
            ctx.prefill(cond, [0], binding.decode_config(dict(cfg, seed=seed)))
            return ctx.generate(T)[0]

        one, two = run(1), run(2)
        assert not np.array_equal(one, two)
        scripted(1)
        assert not np.array_equal(ctx.generate(T)[0], one)      # (the token after a rejection is the script's)
        scripted(1)
        g = capture(ctx, stream, lambda: ctx.xsm_debug_set_script(None, 0.0))
        ctx.xsm_debug_set_script(None, 0.0)
        assert np.array_equal(ctx.generate(T)[0], one)
        scripted(2)
        g.replay()
        assert np.array_equal(ctx.generate(T)[0], two)
        ctx.prefill(cond, [0], binding.decode_config(cfg))
        before = ctx.xsm_kernel_launches()
        ctx.xsm_spec_step()
        direct = ctx.xsm_kernel_launches() - before
        capture(ctx, stream, ctx.xsm_spec_step)
        assert ctx.xsm_kernel_launches() - before == 2 * direct + 1
        ctx.xsm_destroy()


@pytest.mark.parametrize("dtype", [0, 1])
def test_a_step_behind_a_prefill_that_was_only_captured_ends_in_an_error(binding, dtype, monkeypatch):
    """The workspace is full of ones.  A prefill is captured and not run; a direct step then finds the state that xsm_create
    left (no pages in the pool: XSM_ERR_CAPACITY).  Replayed, the prefill begins a request as always."""
    import torch
    cfg = gpu_cfg(dtype=dtype, n_draft=2, sigma=0.05)
    w = inputs.make_weights(cfg, random_gains=True)
    cond = inputs.make_cond(cfg, 2)
    dc = binding.decode_config(cfg)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        other = binding.Context(cfg, w, max_batch=2)
        other.prefill(cond, [0, 5], dc)
        want, _, _ = other.generate(24)
        other.xsm_destroy()
        with monkeypatch.context() as m:
            m.setattr(torch, "empty", lambda n, **kw: torch.full((n,), 255, **kw))
            ctx = binding.Context(cfg, w, max_batch=2)
        d_cond, d_prompt = ctx.cond_to_device(cond), torch.tensor([[0, 5]] * 2, dtype=torch.int32, device="cuda")
        g = capture(ctx, stream, lambda: ctx.xsm_prefill(d_cond, d_prompt, 2, dc))
        ctx.xsm_spec_step()
        with pytest.raises(binding.XsmError) as e:
            ctx.xsm_debug_get_state()
        assert e.value.status == binding.XSM_ERR_CAPACITY
        g.replay()
        toks, lens, _ = ctx.generate(24)
        assert (lens == 24).all() and np.array_equal(toks, want)
        ctx.xsm_destroy()


def test_contexts_on_streams_of_their_own_decode_as_they_do_alone(binding):
    """Five contexts, each with its thread and stream, whose projections take 32 to 256 columns of an SM's 512 of tensor memory and meet
    there."""
    import threading

    import torch
    models = []
    for d, H, f, K, batch in ((128, 2, 128, 7, 16), (256, 4, 512, 3, 1), (512, 8, 512, 0, 97), (128, 2, 256, 4, 6), (1280, 20, 512, 7, 15)):
        cfg = inputs.config(2, d_model=d, n_heads=H, d_head=64, d_ff=f, d_cond=d, head_hidden=d, n_draft=K, n_layers=2, vocab=777, n_cond=40,
                            sigma=0.02 * (1024 / d) ** 0.5, max_seq_len=96)
        models.append((cfg, batch, inputs.make_weights(cfg), inputs.make_cond(cfg, batch)))

    def request(model, stream, times):
        cfg, batch, w, cond = model
        out = []
        with torch.cuda.stream(stream):
            ctx = binding.Context(cfg, w, max_batch=batch, stream=stream)
            for _ in range(times):
                ctx.prefill(cond, [0, 3, 7], binding.decode_config(cfg))
                out.append(ctx.generate(64)[0])
            ctx.xsm_destroy()
        return out

    streams = [torch.cuda.Stream() for _ in models]
    alone = [request(m, s, 1)[0] for m, s in zip(models, streams)]
    got = [None] * len(models)

    def work(i):
        got[i] = request(models[i], streams[i], 8)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(models))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for i, want in enumerate(alone):
        assert got[i] is not None and all(np.array_equal(g, want) for g in got[i]), i


def test_a_request_that_gave_up_waiting_disturbs_no_other_context(binding):
    """One context's stages are launched out of turn and give up; kernels of another, on a stream of its own, share the SMs (and their
    tensor memory) with them all the while."""
    import threading

    import torch
    cfg = inputs.config(2, d_model=512, n_heads=8, d_head=64, d_ff=512, d_cond=512, head_hidden=512, n_draft=3, n_layers=2, vocab=777, n_cond=40,
                        max_seq_len=96)
    w, cond, dc = inputs.make_weights(cfg), inputs.make_cond(cfg, 4), binding.decode_config(cfg)
    streams = [torch.cuda.Stream() for _ in range(2)]
    with torch.cuda.stream(streams[0]):
        ctx = binding.Context(cfg, w, max_batch=4, stream=streams[0])
        ctx.prefill(cond, [0], dc)
        want = ctx.generate(64)[0]
    got = []

    def decode():
        with torch.cuda.stream(streams[0]):
            for _ in range(12):
                ctx.prefill(cond, [0], dc)
                got.append(ctx.generate(64)[0])

    with torch.cuda.stream(streams[1]):
        other = binding.Context(cfg, w, max_batch=4, stream=streams[1])
        t = threading.Thread(target=decode)
        t.start()
        for stage in (2, 5, 6, 9):
            other.prefill(cond, [0], dc)
            other.xsm_debug_set_wait_limits(3000, 0)
            other.xsm_debug_launch_stage(stage)
            with pytest.raises(binding.XsmError) as e:
                other.xsm_debug_get_state()
            assert e.value.status == binding.XSM_ERR_TIMEOUT
            other.xsm_debug_set_wait_limits(0, 0)
        other.prefill(cond, [0], dc)
        last = other.generate(64)[0]
        t.join()
        other.xsm_destroy()
    assert len(got) == 12 and all(np.array_equal(g, want) for g in got) and np.array_equal(last, want)
    ctx.xsm_destroy()
