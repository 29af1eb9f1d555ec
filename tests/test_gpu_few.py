"""Forwards of few live rows (drafts, pre-verification calls, autoregressive steps, early-stopped windows) at the edges of
their kernel: 1 to 17 live rows (8 and 16 are operand sizes, 17 is the other kernel's), fewer weight rows than blocks and
several passes per block, grouped heads, both head sizes, contexts around the key splits.  The logits of every forward (draft
steps and verify forwards of short and full windows) against the oracle's.  The activations carry 16 mantissa bits; what is
seen is at most 2.2e-5 on logits and 2.3e-6 on alpha_hat, the tolerance about four times that.  One lost remainder plane moves
the logits of these shapes by 5e-4 to 6e-3 (fp64 model with one site rounded to 8 bits; q and k of the narrow shape 3e-5)."""
import dataclasses

import numpy as np
import pytest

from oracle import pacer_oracle as orc
from paper_2602_01274_b200 import synth
from tests.common import oracle_models

pytestmark = pytest.mark.gpu
TOL, ALPHA_TOL = 1e-4, 1e-5

SHAPES = {
    # head dimension 64, fewer two-row units than blocks in the residual projections, ragged vocabulary
    "narrow": (synth.ModelShape(2, 128, 2, 1, 192, 1001), synth.ModelShape(1, 64, 1, 1, 64, 1001)),
    # head dimension 128, three heads per kv head, several passes of the gate/up projection and the LM head
    "passes": (synth.ModelShape(1, 768, 6, 2, 20480, 50000), synth.ModelShape(1, 256, 2, 2, 512, 50000)),
}

# reached by name: a target wider than 4096, whose nine and ten rows take three activation stages and eleven five; drafts whose
# gate/up projection takes one pass of 18 or 26 atoms in the variant with long passes (28: two, also there)
WIDER = {
    "stages": (synth.ModelShape(1, 4224, 33, 3, 320, 1001), synth.ModelShape(1, 64, 1, 1, 64, 1001)),
    "long18": (SHAPES["narrow"][0], synth.ModelShape(1, 256, 4, 4, 10240, 1001)),
    "long26": (SHAPES["narrow"][0], synth.ModelShape(1, 128, 2, 2, 15360, 1001)),
    "long28": (SHAPES["narrow"][0], synth.ModelShape(1, 128, 1, 1, 16576, 1001)),
}


@pytest.mark.parametrize("shape", sorted(SHAPES))
@pytest.mark.parametrize("window,n_prompt", [(4, 2), (7, 33), (8, 97), (15, 40), (16, 300)])
def test_verify_rows(shape, window, n_prompt):
    from paper_2602_01274_b200 import binding as b
    T, D = {**SHAPES, **WIDER}[shape]
    cfg = synth.PairConfig("few", T, D, agree=0.8, n_prompt=n_prompt, max_new=24, gamma_max=window, block_b=1 if window % 4 else 4)
    gpu = synth.make_pair(cfg, seed=3, device="cuda:0")
    cpu = {k: ({n: t.cpu() for n, t in v.items()} if isinstance(v, dict) else v.cpu()) for k, v in gpu.items()}
    To, Do, Bo = oracle_models(cfg, cpu)
    max_ctx = n_prompt + cfg.max_new + window + 2
    ctx = b.Context(b.make_cfg(T, D, 1, max_ctx, window, cfg.block_b, cfg.rho, 0, cfg.succ_bias))
    b.load_pair(ctx, gpu)
    prompt = synth.make_prompts(T.vocab, 1, n_prompt, seed=9).numpy()
    ctx.pacer_prefill(prompt, cfg.max_new, window, -1.0)
    o = orc.Pacer(To, Do, Bo, max_ctx, b=cfg.block_b, gamma_cap=window, t0=-1.0, rho=cfg.rho)
    o.prefill(prompt[0])
    V, blocks, rows = T.vocab, window // cfg.block_b, {}
    for k in range(blocks):
        for _ in range(cfg.block_b):
            ctx.pacer_draft_step()
        ctx.pacer_preverify()
        o.draft_block(); o.preverify()
        if k in (0, blocks - 1):
            ctx.pacer_verify()                      # 1 + the drafts so far live rows
            rows[k] = ctx.pacer_read_buffer(b.BUF_VERIFY_LOGITS, np.float32, (window + 1) * V).reshape(window + 1, V)
    o.verify()
    gamma = blocks * cfg.block_b
    assert o.stats()["min_margin_draft"] > 2 * TOL
    np.testing.assert_array_equal(ctx.pacer_read_buffer(b.BUF_DRAFTS, np.int32, window)[:gamma], o.y()[:gamma])
    p, q = o.plogits(gamma + 1), o.qlogits(gamma)
    for k, got in rows.items():                     # a row depends on the drafts before it only
        n = (k + 1) * cfg.block_b + 1
        assert np.abs(got[:n] - p[:n]).max() < TOL, k
    got = ctx.pacer_read_buffer(b.BUF_DRAFT_LOGITS, np.float32, window * V).reshape(window, V)[:gamma]
    assert np.abs(got - q).max() < TOL
    al = ctx.pacer_read_buffer(b.BUF_ALPHA, np.float32, window)[:gamma]
    assert np.abs(al - o.alpha()[:gamma]).max() < ALPHA_TOL
    ctx.close()


@pytest.mark.parametrize("shape,window", [("stages", 8), ("stages", 9), ("stages", 10), ("long18", 4), ("long26", 8), ("long28", 4)])
def test_verify_rows_of_wider_models(shape, window):
    test_verify_rows(shape, window, 9)


@pytest.mark.parametrize("batch", [1, 9, 16, 17])
def test_batched_autoregressive_rows(batch):
    """One live row per sequence: packed rows of several sequences, and one sequence too many for the kernel."""
    from paper_2602_01274_b200 import binding as b
    T, D = SHAPES["narrow"]
    cfg = synth.PairConfig("few", T, D, agree=0.8, n_prompt=21, max_new=6, gamma_max=4, batch=batch)
    gpu = synth.make_pair(cfg, seed=4, device="cuda:0")
    cpu = {k: ({n: t.cpu() for n, t in v.items()} if isinstance(v, dict) else v.cpu()) for k, v in gpu.items()}
    To, _, _ = oracle_models(cfg, cpu)
    ctx = b.Context(b.make_cfg(T, D, batch, 40, 4, 4, cfg.rho, 0, cfg.succ_bias))
    b.load_pair(ctx, gpu)
    prompts = synth.make_prompts(T.vocab, batch, cfg.n_prompt, seed=5).numpy()
    tok, _ = ctx.pacer_generate_ar(prompts, cfg.max_new)
    for s in range(batch):
        out, margin = orc.generate_ar(To, prompts[s], cfg.max_new)
        assert margin > 2 * TOL, s
        np.testing.assert_array_equal(tok[s], out, err_msg=str(s))
    ctx.close()


@pytest.mark.parametrize("n_prompt", [1279, 2600])
def test_many_key_splits(n_prompt):
    """One kv head, so that its keys are cut into 17 and 33 splits: they are merged sixteen at a time."""
    test_verify_rows("narrow", 4, n_prompt)


@pytest.mark.parametrize("vocab,batch,d_ffn", [(4, 3, 64), (16, 9, 2432), (16, 16, 64), (30, 16, 2432)])
def test_small_vocabulary_hidden_rows(vocab, batch, d_ffn):
    """Fewer LM-head rows than twice the sequences: the block that ends a sequence's draft step has none of them, without or
    with rows of the gate/up projection.  The hidden rows queued for the pre-verification model and its scores against the
    oracle's (an entry of a normalised row is a few units and passes about ten roundings to 16 mantissa bits, 2^-17 each:
    1e-4 per unit, 1e-3 is three times that for the largest)."""
    from paper_2602_01274_b200 import binding as b
    T, D = synth.ModelShape(1, 64, 1, 1, 64, vocab), synth.ModelShape(2, 64, 1, 1, d_ffn, vocab)
    cfg = synth.PairConfig("few", T, D, agree=0.8, n_prompt=7, max_new=8, gamma_max=4, batch=batch)
    gpu = synth.make_pair(cfg, seed=3, device="cuda:0", std=0.1)
    cpu = {k: ({n: t.cpu() for n, t in v.items()} if isinstance(v, dict) else v.cpu()) for k, v in gpu.items()}
    To, Do, Bo = oracle_models(cfg, cpu)
    ctx = b.Context(b.make_cfg(T, D, batch, 32, 4, 4, cfg.rho, 0, cfg.succ_bias))
    b.load_pair(ctx, gpu)
    prompts = synth.make_prompts(vocab, batch, cfg.n_prompt, seed=3).numpy()
    ctx.pacer_prefill(prompts, cfg.max_new, 4, -1.0)
    for _ in range(4):
        ctx.pacer_draft_step()
    y = ctx.pacer_read_buffer(b.BUF_DRAFTS, np.int32, batch * 4).reshape(batch, 4)
    h = ctx.pacer_read_buffer(b.BUF_HPEND, np.float32, batch * 5 * D.d_model).reshape(batch, 5, D.d_model)
    ctx.pacer_preverify()
    al = ctx.pacer_read_buffer(b.BUF_ALPHA, np.float32, batch * 4).reshape(batch, 4)
    for s in range(batch):
        o = orc.Pacer(To, Do, Bo, 32, b=4, gamma_cap=4, t0=-1.0, rho=cfg.rho)
        o.prefill(prompts[s])
        o.draft_block()
        want = o.hpend()
        o.preverify()
        assert o.stats()["min_margin_draft"] > 1.0, s
        np.testing.assert_array_equal(y[s], o.y(), err_msg=str(s))
        assert np.abs(h[s, :4] - want).max() < 1e-3, s
        assert np.abs(al[s] - o.alpha()).max() < 1e-3, s
    ctx.close()


@pytest.mark.parametrize("vocab,batch", [(5000, 1), (5000, 3), (1001, 16), (1001, 17), (30, 2)])
@pytest.mark.parametrize("mode", ["greedy", "sample"])
def test_rows_without_a_largest_logit(vocab, batch, mode):
    """Logits that are all NaN (a NaN gain of the final norm): the tokens stay inside the vocabulary (they are looked up by the
    next forward), and the loop ends.  Vocabularies at which lanes, blocks or threads have no column of a row, in the few-row
    kernel and, from 17 sequences on, in the other one."""
    from paper_2602_01274_b200 import binding as b
    shape = synth.ModelShape(1, 64, 1, 1, 64, vocab)
    cfg = synth.PairConfig("few", shape, shape, agree=0.8, n_prompt=5, max_new=6, gamma_max=4, batch=batch)
    pair = synth.make_pair(cfg, seed=3, device="cuda:0")
    for which in ("target", "draft"):
        pair[which]["normf"][3] = float("nan")
    ctx = b.Context(b.make_cfg(shape, shape, batch, 24, 4, 4, cfg.rho, 0, cfg.succ_bias))
    b.load_pair(ctx, pair)
    prompts = synth.make_prompts(vocab, batch, cfg.n_prompt, seed=3).numpy()
    m = b.PACER_SAMPLE if mode == "sample" else b.PACER_GREEDY
    tok, *_ = ctx.pacer_generate(prompts, cfg.max_new, 4, 0.5, m, 7)
    np.testing.assert_array_equal(tok, 0)
    tok, _ = ctx.pacer_generate_ar(prompts, cfg.max_new, m, 7)
    np.testing.assert_array_equal(tok, 0)
    ctx.close()


def test_nan_logit_is_never_the_largest():
    """One column of the LM head is NaN: the other columns decide, as in the oracle (which compares with `>`)."""
    from paper_2602_01274_b200 import binding as b
    T, D = SHAPES["narrow"]
    cfg = synth.PairConfig("few", T, D, agree=0.8, n_prompt=21, max_new=8, gamma_max=4)
    gpu = synth.make_pair(cfg, seed=4, device="cuda:0")
    gpu["target"]["head"][777, 5] = float("nan")
    cpu = {k: ({n: t.cpu() for n, t in v.items()} if isinstance(v, dict) else v.cpu()) for k, v in gpu.items()}
    To, _, _ = oracle_models(cfg, cpu)
    prompt = synth.make_prompts(T.vocab, 1, cfg.n_prompt, seed=5).numpy()
    out, margin = orc.generate_ar(To, prompt[0], cfg.max_new)
    assert margin > 2 * TOL
    ctx = b.Context(b.make_cfg(T, D, 1, 40, 4, 4, cfg.rho, 0, cfg.succ_bias))
    b.load_pair(ctx, gpu)
    tok, _ = ctx.pacer_generate_ar(prompt, cfg.max_new)
    np.testing.assert_array_equal(tok[0], out)
    ctx.close()
