"""Attention of a prompt at the edges of its 128-key tiles: keys that fill the tiles exactly, one key in the last tile, chunks
that begin inside a tile (three sequences share 2048 rows of a chunk, so it is 682 positions long), several sequences of several
tiles, and caches whose memory holds NaN behind the last key, which must not be read even where its probability is zero: the
workspace is filled with NaN before the context takes it.  Checked like the other prompts, through what later steps compute from
the caches, with the same tolerance, for the first and the last sequence."""
import pytest

from tests import test_gpu_prefill as prefill
from tests.common import filled_workspaces

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,batch,n_prompt", [
    ("hd64", 1, 257), ("hd64", 1, 258), ("hd64", 3, 690), ("hd128_gqa", 1, 129), ("hd128_gqa", 1, 385), ("hd128_gqa", 3, 690),
    ("hd64", 2, 258), ("hd128_gqa", 3, 300),
])
def test_prompt_attention_edges(shape, batch, n_prompt):
    with filled_workspaces(0xFF) as sizes:
        prefill.test_prefill_edges(shape, batch, n_prompt, sequences=sorted({0, batch - 1}))
    T = prefill.SHAPES[shape][0]
    # both planes of the target's keys and values lie in a workspace that was filled
    assert max(sizes) > 2 * batch * T.kv_bytes_per_token() * n_prompt
