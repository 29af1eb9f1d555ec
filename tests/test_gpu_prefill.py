"""Prompt prefill at the edges of its tiles and chunks: the last prompt through the forward kernel and the first through the
tiled GEMMs (32 / 33 rows), 128-row tiles with remainders, a batch whose sequences share a tile, more rows than a chunk,
grouped heads and both head sizes.  Everything that later steps read of a prefill (the three models' caches) is checked
through what they compute from it: target logits, drafts and alpha_hat of one block against the oracle's.  What is seen is at
most 2.2e-5 on logits and 2.3e-6 on alpha_hat, the tolerance about four times that.  One lost remainder plane moves the logits of
these shapes by 4e-4 to 7e-3 (fp64 model with one site rounded to 8 bits; q and k of the narrowest shape 1e-4)."""
import numpy as np
import pytest

from oracle import pacer_oracle as orc
from paper_2602_01274_b200 import synth
from tests.common import oracle_models

pytestmark = pytest.mark.gpu
TOL, ALPHA_TOL = 1e-4, 1e-5

SHAPES = {
    "hd64": (synth.ModelShape(2, 256, 4, 4, 320, 2048), synth.ModelShape(2, 128, 2, 1, 192, 2048)),
    # 10 and 65 blocks of 64 columns: the sums that leave the tensor cores every eight blocks end in a remainder
    "long_k": (synth.ModelShape(2, 640, 5, 5, 4160, 2048), synth.ModelShape(2, 320, 5, 1, 2112, 2048)),
    "hd128_gqa": (synth.ModelShape(2, 512, 4, 2, 1088, 2048), synth.ModelShape(1, 256, 2, 2, 512, 2048)),
}


@pytest.mark.parametrize("shape,batch,n_prompt", [
    ("hd64", 1, 33), ("hd64", 1, 34), ("hd64", 2, 18), ("hd64", 3, 44), ("hd64", 1, 129), ("hd64", 1, 130),
    ("hd64", 1, 2050), ("hd64", 5, 500), ("hd128_gqa", 1, 65), ("hd128_gqa", 1, 300), ("hd128_gqa", 4, 97),
    ("hd128_gqa", 1, 2305), ("long_k", 1, 140), ("long_k", 2, 50),
])
def test_prefill_edges(shape, batch, n_prompt, sequences=None):
    from paper_2602_01274_b200 import binding as b
    T, D = SHAPES[shape]
    cfg = synth.PairConfig("pf", T, D, agree=0.8, n_prompt=n_prompt, max_new=8, gamma_max=4, batch=batch)
    gpu = synth.make_pair(cfg, seed=6, device="cuda:0")
    cpu = {k: ({n: t.cpu() for n, t in v.items()} if isinstance(v, dict) else v.cpu()) for k, v in gpu.items()}
    To, Do, Bo = oracle_models(cfg, cpu)
    max_ctx = n_prompt + 8 + 4 + 2
    ctx = b.Context(b.make_cfg(T, D, batch, max_ctx, 4, 4, cfg.rho, 0, cfg.succ_bias))
    b.load_pair(ctx, gpu)
    prompts = synth.make_prompts(T.vocab, batch, n_prompt, seed=8).numpy()
    ctx.pacer_prefill(prompts, 8, 4, -1.0)
    for st in ctx.pacer_read_state(batch):
        assert (st["len_T"], st["len_D"], st["len_B"]) == (n_prompt - 1,) * 3
    for _ in range(4):
        ctx.pacer_draft_step()
    ctx.pacer_preverify()
    ctx.pacer_verify()
    V = T.vocab
    y = ctx.pacer_read_buffer(b.BUF_DRAFTS, np.int32, batch * 4).reshape(batch, 4)
    al = ctx.pacer_read_buffer(b.BUF_ALPHA, np.float32, batch * 4).reshape(batch, 4)
    pl = ctx.pacer_read_buffer(b.BUF_VERIFY_LOGITS, np.float32, batch * 5 * V).reshape(batch, 5, V)
    checked = 0
    for s in sequences or range(batch if n_prompt < 400 else 1):
        o = orc.Pacer(To, Do, Bo, max_ctx, b=4, gamma_cap=4, t0=-1.0, rho=cfg.rho)
        o.prefill(prompts[s])
        o.draft_block(); o.preverify(); o.verify()
        # row 0 does not depend on the drafts; the rest is comparable when no draft hangs on a tie
        assert np.abs(pl[s, 0] - o.plogits(5)[0]).max() < TOL, s
        if o.stats()["min_margin_draft"] > 2 * TOL:
            checked += 1
            np.testing.assert_array_equal(y[s], o.y()[:4])
            assert np.abs(al[s] - o.alpha()[:4]).max() < ALPHA_TOL, s
            assert np.abs(pl[s] - o.plogits(5)).max() < TOL, s
    assert checked or batch > 1
    ctx.close()
