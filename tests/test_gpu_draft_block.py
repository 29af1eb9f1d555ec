"""A block's draft forwards in one launch against the same forwards in launches of their own (which profiling asks for): tokens,
windows, accepted lengths, hidden-state scores and logits are the same to the last bit, for one sequence, for several that stop
at different blocks, for the most that one launch takes (eight, two catch-up rows each), greedy and sampled, and for models so
narrow that some blocks of the grid own no row of a projection."""
import numpy as np
import pytest

from paper_2602_01274_b200 import synth

pytestmark = pytest.mark.gpu

SHAPES = {
    "tiny": synth.CONFIGS["tiny"],
    "gqa": synth.PairConfig("gqa", synth.ModelShape(2, 512, 4, 2, 1088, 2048), synth.ModelShape(2, 768, 6, 2, 1536, 2048), agree=0.8, n_prompt=40,
                            max_new=24, gamma_max=8),
    # a draft whose gate/up projection takes the variant with long passes
    "long": synth.PairConfig("long", synth.ModelShape(2, 128, 2, 1, 192, 2048), synth.ModelShape(1, 256, 4, 4, 10240, 2048), agree=0.8, n_prompt=40,
                             max_new=24, gamma_max=8),
}


@pytest.mark.parametrize("shape,batch,window,block,sample", [
    ("tiny", 1, 8, 4, False), ("tiny", 3, 8, 4, False), ("tiny", 8, 8, 4, True), ("tiny", 2, 8, 2, False),
    ("gqa", 1, 8, 4, True), ("gqa", 4, 4, 4, False), ("gqa", 8, 8, 8, False),
    ("long", 1, 8, 4, True), ("long", 6, 8, 4, False), ("long", 8, 8, 4, False),
])
def test_one_launch_per_block(shape, batch, window, block, sample):
    from paper_2602_01274_b200 import binding as b
    cfg = SHAPES[shape]
    pair = synth.make_pair(cfg, seed=3, device="cuda:0")
    n_prompt, new = 21, 24
    prompts = synth.make_prompts(cfg.target.vocab, batch, n_prompt, seed=5).numpy()
    mode, V = (b.PACER_SAMPLE if sample else b.PACER_GREEDY), cfg.target.vocab
    runs = []
    for stamped in (False, True):
        ctx = b.Context(b.make_cfg(cfg.target, cfg.draft, batch, n_prompt + new + 8 + 2, 8, block, cfg.rho, 0, 16.0))
        b.load_pair(ctx, pair)
        if stamped:
            ctx.pacer_profile_begin()
        tok, ns, dl, al, st = ctx.pacer_generate(prompts, new, window, 0.5, mode, 11)
        runs.append([tok, ns, dl, al, ctx.pacer_read_buffer(b.BUF_DRAFT_LOGITS, np.float32, batch * 8 * V).reshape(batch, 8, V)[:, :block],
                     ctx.pacer_read_buffer(b.BUF_VERIFY_LOGITS, np.float32, V), ctx.pacer_read_buffer(b.BUF_ALPHA, np.float32, batch * 8),
                     [st[k] for k in ("n_draft_fwd", "n_mb_calls", "n_target_fwd")]])
        launches = st["n_kernel_launches"]
        if stamped:
            ctx.pacer_profile_end()
            assert launches > plain, "the two runs launched the same"
        plain = launches
        ctx.close()
    assert runs[0][7] == runs[1][7]
    for one, each in zip(*runs):
        np.testing.assert_array_equal(np.asarray(one), np.asarray(each))
