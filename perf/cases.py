"""Workloads the library is timed on: what a user of the decoding loop has it do, through the binding's public calls.

Shapes are the pairs of ``synth.CONFIGS``; the deepest targets keep their widths and lose layers (a forward's time is
proportional to the layer count), so that several contexts fit one device.  Weights, successor tables and prompts come from
the seed.  The planted successor gets a bias of +16 instead of the configurations' +8: the loop then accepts a draft
exactly where the two successor tables agree (about the configuration's share of the vocabulary), as with a confident
model, and no token hangs on a near-tie between two noise logits.

Operations
  generate  ``pacer_generate``: prompt in host memory, prefill, draft-and-verify steps until ``new`` tokens exist
  ar        ``pacer_generate_ar``: the target alone, one token per forward
  verify    ``pacer_verify``: one target forward over a full draft window (the context is filled in ``prepare``), and
            the logits a scoring program reads back
  linear    ``pacer_linear``: the stand-alone skinny product
"""
from __future__ import annotations

import dataclasses
import math

import numpy as np
import torch

from paper_2602_01274_b200 import binding, synth

DEVICE = "cuda:0"
SUCC_BIAS = 16.0
# target layers kept at most (33b: 62 -> 14, qwen: 64 -> 10, 13b: 40 -> 12; batches: 4)
LAYERS = {"tiny": 4, "7b_68m": 32, "13b_68m": 12, "33b_1b3": 14, "qwen_32b_1b5": 10}


def _gen(name, pair, layers, batch, prompt, new, window, threshold, sample=False):
    return dict(name=name, op="generate", pair=pair, layers=layers, batch=batch, prompt=prompt, new=new, window=window,
                threshold=threshold, sample=sample)


def listed():
    return [
        # the smallest loop there is: short prompt, small models; launches and fixed costs of a forward count
        _gen("loop_tiny", "tiny", 4, 1, 64, 64, 8, 0.5),
        # a chat turn at the main configuration: 512-token prompt, adaptive window
        _gen("chat_7b", "7b_68m", 32, 1, 512, 64, 16, 0.5),
        # the same pair decoding from a short prompt of odd length with rejection sampling and a fixed window
        _gen("sample_7b", "7b_68m", 16, 1, 77, 48, 8, -1.0, True),
        # summarisation: a long prompt of odd length, few new tokens
        _gen("long_prompt_7b", "7b_68m", 16, 1, 3001, 8, 8, 0.5),
        # the baseline a user compares with: plain autoregressive decoding of the target
        dict(name="ar_7b", op="ar", pair="7b_68m", layers=16, batch=1, prompt=33, new=32, window=4),
        # wider target, 1024-token prompt, a threshold that stops most windows after one block
        _gen("chat_13b", "13b_68m", 12, 1, 1024, 48, 16, 0.7),
        # grouped-query target with a large draft model and the widest window
        _gen("code_33b", "33b_1b3", 14, 1, 2048, 48, 24, 0.5),
        # grouped-query pair with a vocabulary of 151 936
        _gen("chat_qwen", "qwen_32b_1b5", 10, 1, 1024, 32, 16, 0.5),
        # eight sequences that share every forward (136 verify rows), long contexts
        _gen("batch8_long", "7b_68m", 4, 8, 2048, 32, 16, 0.5),
        # scoring a full draft window behind a long context: the verify forward alone, logits read back
        dict(name="verify_33b", op="verify", pair="33b_1b3", layers=14, batch=1, prompt=2048, new=4, window=24),
        # the stand-alone product: a small and a large one
        dict(name="linear_small", op="linear", rows=5, n=2304, k=768),
        dict(name="linear_large", op="linear", rows=17, n=4096, k=11008),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["generate"] * 6 + ["ar", "verify", "linear"])
    if op == "linear":
        k = 32 * _log_int(rng, 8, 344)
        return dict(op="linear", rows=rng.randint(1, 32), n=_log_int(rng, 256, min(32000, 4096 * 11008 // k)), k=k)
    pair = rng.choice(list(LAYERS))
    gamma_cap = synth.CONFIGS[pair].gamma_cap
    layers = rng.randint(max(2, LAYERS[pair] // 2), LAYERS[pair])
    window = 4 * rng.randint(1, gamma_cap // 4)
    if op != "generate":
        return dict(op=op, pair=pair, layers=layers, batch=1, prompt=_log_int(rng, 16, 1024), new=rng.randint(8, 32), window=window)
    batch = rng.choice([1, 1, 1, 2, 3, 4, 5, 8])
    batch = min(batch, 144 // (window + 1))
    if batch > 1:
        layers = min(layers, 4)
    return dict(op=op, pair=pair, layers=layers, batch=batch, prompt=_log_int(rng, 16, 2048 // batch), new=rng.randint(8, 48),
                window=window, threshold=rng.choice([-1.0, 0.3, 0.5, 0.5, 0.7]), sample=rng.random() < 0.25)


def _pair(case):
    cfg = synth.CONFIGS[case["pair"]]
    # a context is created for the window it will run with
    return dataclasses.replace(cfg, target=dataclasses.replace(cfg.target, n_layers=case["layers"]), batch=case["batch"],
                               n_prompt=case["prompt"], max_new=case["new"], gamma_max=case["window"], succ_bias=SUCC_BIAS)


def prepare(case, seed):
    if case["op"] == "linear":
        return dict(case=case, x=synth.normal_bf16(seed, 12, (case["rows"], case["k"]), std=1.0, device=DEVICE),
                    w=synth.normal_bf16(seed, 11, (case["n"], case["k"]), std=0.02, device=DEVICE))
    cfg = _pair(case)
    pair = synth.make_pair(cfg, seed=seed, device=DEVICE)
    ctx = binding.Context(binding.make_cfg(cfg.target, cfg.draft, cfg.batch, cfg.n_prompt + cfg.max_new + cfg.gamma_cap + 2,
                                           cfg.gamma_cap, cfg.block_b, cfg.rho, 0, cfg.succ_bias), device=DEVICE)
    binding.load_pair(ctx, pair)
    prompts = synth.make_prompts(cfg.target.vocab, cfg.batch, cfg.n_prompt, seed=seed).numpy()
    if case["op"] == "verify":
        ctx.pacer_prefill(prompts, cfg.max_new, cfg.gamma_max, -1.0)
        for _ in range(cfg.gamma_cap // cfg.block_b):
            for _ in range(cfg.block_b):
                ctx.pacer_draft_step()
            ctx.pacer_preverify()
        ctx.pacer_read_state(cfg.batch)
    return dict(case=case, cfg=cfg, ctx=ctx, prompts=prompts, seed=seed)


def run(state):
    case = state["case"]
    if case["op"] == "linear":
        return binding.pacer_linear(state["x"], state["w"])
    cfg, ctx, vocab = state["cfg"], state["ctx"], state["cfg"].target.vocab
    if case["op"] == "verify":
        ctx.pacer_verify()
        rows = cfg.gamma_cap + 1
        return ctx.pacer_read_buffer(binding.BUF_VERIFY_LOGITS, np.float32, rows * vocab)
    if case["op"] == "ar":
        tokens, _ = ctx.pacer_generate_ar(state["prompts"], cfg.max_new)
        return dict(tokens=tokens, logits=ctx.pacer_read_buffer(binding.BUF_VERIFY_LOGITS, np.float32, vocab))
    mode = binding.PACER_SAMPLE if case["sample"] else binding.PACER_GREEDY
    tokens, steps, draft_len, accept_len, _ = ctx.pacer_generate(state["prompts"], cfg.max_new, cfg.gamma_max, case["threshold"],
                                                                 mode, state["seed"])
    # with the tokens: the target's and the draft's logits of the first sequence's last step
    return dict(tokens=tokens, steps=steps, draft_len=draft_len, accept_len=accept_len,
                logits=ctx.pacer_read_buffer(binding.BUF_VERIFY_LOGITS, np.float32, vocab),
                draft_logits=ctx.pacer_read_buffer(binding.BUF_DRAFT_LOGITS, np.float32, vocab))


def work(case):
    """Bytes: the weights of a model once per forward, a prompt's weights once in all, every live key and value once per
    forward.  Flops: two per weight and row.  The number of steps follows from the share of the vocabulary on which the
    two models agree (a window that may stop early is counted as one block)."""
    if case["op"] == "linear":
        r, n, k = case["rows"], case["n"], case["k"]
        return dict(bytes=2.0 * n * k + 2.0 * r * k + 4.0 * r * n, flops=2.0 * r * n * k)
    cfg = _pair(case)
    B, n, new, p = cfg.batch, cfg.n_prompt, cfg.max_new, cfg.agree
    mb = synth.preverify_shape(cfg.draft)

    def layer_bytes(m):
        return m.streamed_weight_bytes() - 2 * m.vocab * m.d_model

    def forward(m, rows, ctx, head):
        weights = layer_bytes(m) + (2 * m.vocab * m.d_model if head else 0)
        attn = 4.0 * m.n_layers * m.d_model * ctx * rows
        return weights + B * (m.kv_bytes_per_token() * (ctx + rows)), B * (rows * weights + attn)

    def prompt(m):
        return layer_bytes(m) + B * n * m.kv_bytes_per_token(), B * (n * layer_bytes(m) + 2.0 * m.n_layers * m.d_model * n * n)

    if case["op"] == "verify":
        by, fl = forward(cfg.target, cfg.gamma_cap + 1, n, True)
        return dict(bytes=by + 4.0 * (cfg.gamma_cap + 1) * cfg.target.vocab, flops=fl)
    parts = []
    if case["op"] == "ar":
        parts = [(1, prompt(cfg.target)), (new, forward(cfg.target, 1, n + new // 2, True))]
    else:
        window = cfg.gamma_cap if case["threshold"] < 0 else cfg.block_b
        steps = max(1, round(new / sum(p ** i for i in range(window + 1))))
        ctx = n + new // 2
        parts = [(1, prompt(cfg.target)), (1, prompt(cfg.draft)), (1, prompt(mb)),
                 (steps, forward(cfg.target, window + 1, ctx, True)), (steps * window, forward(cfg.draft, 1, ctx, True)),
                 (steps * window // cfg.block_b, forward(mb, cfg.block_b, ctx, False))]
    return dict(bytes=float(sum(c * b for c, (b, _) in parts)), flops=float(sum(c * f for c, (_, f) in parts)))


def tolerance(case):
    if case["op"] == "linear":
        # bf16 inputs, fp32 sums of at most 11 008 products: an fp64 product differs by 1e-6 (5e-6 at the worst element)
        return {"rel": 4e-6, "max": 2e-5}
    # activations carry 16 mantissa bits: the logits differ from an fp64 forward's by 4e-6 (tiny) to 9e-5 (32 layers of
    # width 4096, 14 of width 7168), at the worst element 4e-4; tokens and lengths are the same
    return {"rel": 4e-4, "max": 2e-3, "differ": 0.0}
