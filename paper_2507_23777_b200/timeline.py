"""Per-stage timeline of one decoding step (xsm_debug_trace_step), as a table.

    python -m paper_2507_23777_b200.timeline --config 2 --warm 64 [--batch B] [--prompt TOKENS] [--room TOKENS]

Runs `warm` decoding steps of the chosen configuration (batch 1, a prompt of one token and the configured room unless
told otherwise), then eleven traced steps, and prints for the one in the middle by duration and every kind of stage: how
long the step spends in it (last CTA of the previous stage done -> last CTA of this stage done), how long after the
previous stage's end a CTA is past the wait for it, and how long it takes from there to its end.  Every mark is a read of
the GPU's global timer plus a store (a few hundred nanoseconds), so a traced step is slower than an untraced one; compare
shares, not totals.  A traced step is launched kernel by kernel: four ordinary steps are queued before it, so that the host is
ahead of the device as it is when recordings are replayed (else a kernel starts when the host launches it, every 4 us).
"""
from __future__ import annotations

import argparse

import numpy as np

from . import binding, build, inputs

def stage_names(cfg, n_stages: int):
    """Names of a layer's stages and of the tail's.  A layer has seven stages where the cross-attention projects its own
    queries, else eight."""
    tail = ["LM head" + (" + head blocks" if cfg["n_draft"] else "")]
    if cfg["n_draft"] and cfg.get("head_kind", 0) == 1:
        tail += ["heads' cross-attention", "heads' out-projection"]
    if cfg["n_draft"]:
        tail.append("head output projections")
    tail.append("verify / resample / commit / embed")
    cross = ["RMSNorm + cross q + cross-attention"]
    if n_stages - len(tail) == 8 * cfg["n_layers"]:
        cross = ["RMSNorm + cross q", "cross-attention"]
    return (["RMSNorm + QKV", "self-attention", "out-projection + residual"] + cross +
            ["cross out-projection + residual", "RMSNorm + gate/up + SiLU*mul", "down projection + residual"], tail)


def table(cfg, t: np.ndarray) -> str:
    t = t.astype(np.int64)
    rows, G = t.shape
    L = cfg["n_layers"]
    layer, tail = stage_names(cfg, (rows - 1) // 2)
    end_prev = t[0][t[0] > 0].max()
    acc: dict[str, list] = {}
    for p in range((rows - 1) // 2):
        a, e = t[1 + 2 * p], t[2 + 2 * p]
        name = layer[p % len(layer)] if p < len(layer) * L else tail[p - len(layer) * L]
        has = (a > 0) & (e > 0)
        if not has.any():
            continue
        acc.setdefault(name, []).append((e.max() - end_prev, (a[has] - end_prev).mean(), (e[has] - a[has]).mean(), int(has.sum())))
        end_prev = e.max()
    total = end_prev - t[0][t[0] > 0].min()
    out = [f"traced step: {total / 1e3:.1f} us (at most {G} CTAs of a stage are recorded)", f"{'stage':34s} {'n':>3s} {'us each':>8s} {'share':>7s} {'wait in':>8s} {'compute':>8s} {'CTAs':>5s}"]
    for k, v in acc.items():
        v = np.array(v, dtype=float)
        out.append(f"{k:34s} {len(v):3d} {v[:, 0].mean() / 1e3:8.2f} {100 * v[:, 0].sum() / total:6.1f}% {v[:, 1].mean() / 1e3:8.2f} {v[:, 2].mean() / 1e3:8.2f} {v[:, 3].mean():5.0f}")
    return "\n".join(out)


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--config", type=int, default=2)
    ap.add_argument("--warm", type=int, default=64)
    ap.add_argument("--batch", type=int, default=1)
    ap.add_argument("--prompt", type=int, default=1, help="tokens of the prompt (random behind the first)")
    ap.add_argument("--room", type=int, default=0, help="max_seq_len in place of the configured one")
    args = ap.parse_args()
    build.build()
    cfg = inputs.config(args.config)
    if args.room:
        cfg["max_seq_len"] = args.room
    w = inputs.make_weights(cfg)
    ctx = binding.Context(cfg, w, max_batch=args.batch)
    prompt = [cfg["bos_id"]] + [int(t) for t in np.random.default_rng(1).integers(1, cfg["vocab"], args.prompt - 1)]
    ctx.prefill(inputs.make_cond(cfg, args.batch), prompt, binding.decode_config(cfg))
    for _ in range(args.warm):
        ctx.xsm_spec_step()
    print(f"config {args.config} ({cfg['name']}), batch {args.batch}, context {int(ctx.xsm_debug_get_state()['len'][0])}")
    steps = []
    for _ in range(11):
        for _ in range(4):
            ctx.xsm_spec_step()
        steps.append(ctx.xsm_debug_trace_step())
    steps.sort(key=lambda t: int(t[-1].max()) - int(t[0][t[0] > 0].min()))
    print(table(cfg, steps[5]))
    ctx.xsm_destroy()


if __name__ == "__main__":
    main()
