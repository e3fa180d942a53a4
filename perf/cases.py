"""The work that users of this package have it do, as measurable cases: training steps of the stages
of multi-stage layerwise training, and forward passes for evaluation between stages.

A case names an architecture (the package's own configurations and the small ragged one of its
tests), the stack's depth and how many of its top layers train, the batch shape, and the options.
`prepare` builds what a training program holds before a step (a context grown to its depth by
stacking, weights, optimizer, one batch on the GPU); `run` is one call of the public entry point.
"""
from __future__ import annotations

import numpy as np
import torch

from paper_2011_13635_b200 import inputs as I
from paper_2011_13635_b200.binding import Mslt

# hidden, heads, ffn, vocab, max_pos
ARCH = {
    "tiny": (128, 2, 512, 1024, 512),
    "ragged": (192, 3, 320, 1037, 512),
    "base": (768, 12, 3072, 30522, 512),
    "large": (1024, 16, 4096, 30522, 512),
}


def _case(what, arch, dtype, layers, trainable, batch, seq, pred, shortest=0, opt="adam", nsp=False, share=1,
          loss=True):
    """shortest: 0 = every sequence is `seq` long, else lengths are uniform in [shortest, seq];
    share: layers per shared parameter block; loss: the call waits and returns the loss."""
    return dict(what=what, arch=arch, dtype=dtype, layers=layers, trainable=trainable, batch=batch, seq=seq,
                pred=pred, shortest=shortest, opt=opt, nsp=nsp, share=share, loss=loss)


def listed():
    return [
        # the package's smallest configuration, debugging and unit runs: bound by launches
        dict(_case("step", "tiny", "fp32", 2, 1, 8, 64, 10), name="tiny_stage_fp32"),
        # odd widths and lengths, everything trains, the other optimizer
        dict(_case("step", "ragged", "fp32", 3, 3, 3, 72, 7, shortest=20, opt="lamb"), name="ragged_full_fp32_lamb"),
        # first stage of BERT-Base (three layers, all of them train) in full precision
        dict(_case("step", "base", "fp32", 3, 3, 8, 128, 20), name="base_first_stage_fp32"),
        # the benchmark's headline: last stage of BERT-Base, enqueued step after step
        dict(_case("step", "base", "bf16", 12, 3, 128, 128, 20, loss=False), name="base_last_stage"),
        # the joint retraining that ends a schedule
        dict(_case("step", "base", "bf16", 12, 12, 128, 128, 20, loss=False), name="base_retraining"),
        # the paper's own per-GPU batch and objectives, second stage, LAMB
        dict(_case("step", "base", "bf16", 6, 3, 32, 128, 20, opt="lamb", nsp=True), name="base_second_stage_lamb_nsp"),
        # an uneven batch of short sequences
        dict(_case("step", "base", "bf16", 9, 3, 37, 104, 16, shortest=24), name="base_third_stage_ragged"),
        # sequences of medium length, parameters shared by groups of three layers
        dict(_case("step", "base", "bf16", 12, 6, 21, 232, 35, shortest=96, share=3, loss=False),
             name="base_shared_medium_rows"),
        # BERT-Large, three new layers on a deep frozen stack
        dict(_case("step", "large", "bf16", 24, 3, 64, 128, 20, loss=False), name="large_stage"),
        # BERT-Large on long padded sequences
        dict(_case("step", "large", "bf16", 24, 6, 16, 512, 80, shortest=256, loss=False), name="large_long_stage"),
        # evaluation of one sequence: latency
        dict(_case("forward", "base", "bf16", 12, 3, 1, 64, 10), name="base_eval_one"),
        # evaluation of a batch of long rows
        dict(_case("forward", "large", "bf16", 18, 3, 12, 384, 60, shortest=200), name="large_eval_long"),
    ]


def _between(rng, lo, hi):
    """A whole number, spread over the logarithm of [lo, hi]."""
    return min(hi, max(lo, int(round(float(np.exp(rng.uniform(np.log(lo), np.log(hi))))))))


def draw(rng):
    kind = rng.choice(["small", "small", "base", "base", "base", "large", "eval", "eval"])
    seq = 8 * _between(rng, 2, 64)
    if kind == "small":
        arch, dtype = rng.choice([("tiny", "fp32"), ("ragged", "fp32"), ("base", "fp32"), ("ragged", "bf16")])
        layers = rng.randint(1, 3)
        trainable = rng.randint(0, layers)
        tokens = _between(rng, 64, 1024)
        seq = min(seq, 128)
    elif kind == "large":
        arch, dtype = "large", "bf16"
        layers = rng.choice([6, 12, 18, 24])
        trainable = rng.choice([3, 6])
        tokens = _between(rng, 1024, 8192)
    else:
        arch, dtype = "base", "bf16"
        layers = rng.choice([3, 6, 9, 12])
        trainable = rng.choice([3, 3, layers])
        tokens = _between(rng, 512, 16384)
        if kind == "eval":
            tokens = _between(rng, 32, 8192)
    batch = max(1, tokens // seq)
    shortest = rng.choice([0, 0, max(8, seq // 4), max(8, seq // 2)])
    return _case("forward" if kind == "eval" else "step", arch, dtype, layers, trainable, batch, seq,
                 max(1, round(0.15 * seq)), shortest=shortest, opt="adam" if kind == "eval" else rng.choice(["adam", "adam", "lamb"]),
                 nsp=kind != "eval" and rng.random() < 0.25,
                 share=3 if kind == "base" and rng.random() < 0.2 else 1, loss=kind == "eval" or rng.random() < 0.5)


def _config(c):
    hidden, heads, ffn, vocab, max_pos = ARCH[c["arch"]]
    return I.StageConfig("case", hidden, heads, ffn, vocab, max_pos, c["layers"], c["trainable"], c["batch"], c["seq"],
                         c["pred"], c["dtype"], (c["shortest"], c["seq"]) if c["shortest"] else None,
                         share_group=c["share"], nsp=c["nsp"])


def prepare(case, seed):
    cfg = _config(case)
    # the stack starts at the depth of one stage and grows by copies of its top layers
    first = cfg.layers if cfg.layers <= 3 else 3 if cfg.layers % 3 == 0 else cfg.share_group
    model = Mslt.from_config(cfg, init_layers=first, max_trainable=cfg.trainable)
    shapes = I.param_shapes(cfg, first)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    count = sum(int(np.prod(s)) for s in shapes.values())
    flat = (torch.randn(count, generator=gen, device="cuda") * 0.02).cpu().numpy()
    at = 0
    for name, shape in shapes.items():
        n = int(np.prod(shape))
        w = flat[at:at + n].reshape(shape)
        model.mslt_set_param(name, w + 1.0 if name.endswith("gamma") else w)
        at += n
    while model.num_layers < cfg.layers:
        model.mslt_add_layers(min(model.num_layers, cfg.layers - model.num_layers))
    model.mslt_set_trainable(cfg.trainable)
    # learning rates of the warm-up of a stage
    lamb = case["opt"] == "lamb"
    model.mslt_set_optimizer(lr=8.8e-5 if lamb else 1e-5, lamb=int(lamb))
    tokens, lens, pos, lab = I.make_batch(cfg, seed=seed)
    segments, nsp_labels = I.make_nsp(cfg, lens, seed=seed)
    on_gpu = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    params = model._params[:16 * (model.param_bytes // (18 if case["dtype"] == "bf16" else 16))].view(torch.float32)
    n = params.numel() // 4
    state = dict(model=model, case=case, tokens=on_gpu(tokens), lens=on_gpu(lens) if case["shortest"] else None,
                 pos=on_gpu(pos), lab=on_gpu(lab), segments=on_gpu(segments), nsp_labels=on_gpu(nsp_labels))
    if case["what"] == "step":
        # the caller owns the parameter block: a step leaves weights, gradients and moments there
        grads = model.grad_buckets()
        at = [(g.data_ptr() - params.data_ptr()) // 4 for g in grads]
        state["out"] = dict(weights=params[:n], grads=grads,
                            moment1=[params[o + n:o + n + g.numel()] for o, g in zip(at, grads)],
                            moment2=[params[o + 2 * n:o + 2 * n + g.numel()] for o, g in zip(at, grads)])
    torch.cuda.synchronize()
    return state


def run(s):
    model, c = s["model"], s["case"]
    if c["what"] == "forward":
        # rows in the padding are unspecified: the hidden states come along where there is none
        hidden, logits = model.mslt_forward(s["tokens"], s["lens"], s["pos"], want_hidden=not c["shortest"])
        return dict(hidden=hidden, logits=logits)
    if c["nsp"]:
        loss = model.mslt_step_nsp(s["tokens"], s["lens"], s["segments"], s["pos"], s["lab"], s["nsp_labels"],
                                   sync=c["loss"])
    else:
        loss = model.mslt_step(s["tokens"], s["lens"], s["pos"], s["lab"], sync=c["loss"])
    return dict(s["out"], loss=loss)


def work(case):
    cfg = _config(case)
    H, F, V, L, k = cfg.hidden, cfg.ffn, cfg.vocab, cfg.layers, cfg.trainable
    E = 2 if case["dtype"] == "bf16" else 4
    lo, hi = case["shortest"] or cfg.seq, cfg.seq
    T = cfg.batch * (lo + hi) / 2                                    # tokens that are not padding
    squares = cfg.batch * ((lo + hi) ** 2 / 4 + ((hi - lo + 1) ** 2 - 1) / 12)   # sum of squared lengths
    R = cfg.batch * min(cfg.pred, max(1, round(0.15 * (lo + hi) / 2)))           # masked slots that are filled
    layer = 2 * T * (4 * H * H + 2 * H * F) + 4 * squares * H
    block = 4 * H * H + 2 * H * F + 9 * H + F
    head = H * H + 3 * H + V + (H * H + 3 * H + 2 if cfg.nsp else 0)
    emb = (V + cfg.max_pos + 2 + (2 if cfg.nsp else 0)) * H
    flops = L * layer + 2 * R * H * (H + V)
    size = (L // cfg.share_group) * block * E + head * E + V * H * E + T * H * E + 4 * cfg.batch * (cfg.seq + 2 * cfg.pred)
    if case["what"] == "forward":
        size += cfg.batch * cfg.pred * V * 4 + (0 if case["shortest"] else cfg.batch * cfg.seq * H * E)
        return dict(bytes=float(size), flops=float(flops))
    trained = (k // cfg.share_group) * block + head + (emb if k == L else 0)
    flops += 2 * k * layer + 2 * R * H * (2 * H + V)
    flops += 2 * R * H * V if k == L else -(6 * T * H * H if k else 0)
    # weights and two moments in, the same and the gradient out, and the copy that the kernels read
    size += trained * (12 + 16 + (2 if E == 2 else 0))
    return dict(bytes=float(size), flops=float(flops))


def tolerance(case):
    # bf16: two implementations that round at other places and add in another order (batched-product
    # attention, contractions on the plain ALUs) differ by 0.8e-2 to 1.2e-2 in gradients, moments and
    # logits, and this one differs from a float64 computation by 1.2e-2 to 1.4e-2.
    # fp32: gradients differ from a float64 computation by 6e-7 to 4e-6 (largest difference 2.7e-4).
    return {"rel": 0.03} if case["dtype"] == "bf16" else {"rel": 2e-5, "max": 2e-3}
