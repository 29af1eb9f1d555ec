"""Attention of a prompt at the edges of its 128-key tiles: keys that fill the tiles exactly, one key in the last tile, chunks
that begin inside a tile (three sequences share 2048 rows of a chunk, so it is 682 positions long), and caches whose memory
holds NaN behind the last key, which must not be read even where its probability is zero.  Checked like the other prompts,
through what later steps compute from the caches, with the same tolerance."""
import pytest
import torch

from tests import test_gpu_prefill as prefill

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,batch,n_prompt", [
    ("hd64", 1, 257), ("hd64", 1, 258), ("hd64", 3, 690), ("hd128_gqa", 1, 129), ("hd128_gqa", 1, 385), ("hd128_gqa", 3, 690),
])
def test_prompt_attention_edges(shape, batch, n_prompt):
    # the workspace (some 60 MB here) is likely to be cut from this block; if it is not, the case is an ordinary one
    torch.cuda.empty_cache()
    nan = torch.full((512 << 20,), 0xFF, dtype=torch.uint8, device="cuda:0")
    del nan
    prefill.test_prefill_edges(shape, batch, n_prompt)
