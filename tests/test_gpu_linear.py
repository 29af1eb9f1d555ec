"""The stand-alone skinny product at the edges of its split: 1 to 64 weight tiles per block, one to eight k slices per
cluster, row counts around the 16-row operand, ragged N, short k and activations that are not 16-byte aligned."""
import numpy as np
import pytest
import torch

from oracle import pacer_oracle as orc
from paper_2602_01274_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,N,K,offset", [
    (1, 1, 32, 0),              # one tile, one chunk
    (16, 9, 64, 0),             # a ragged second tile; fewer chunks than warps
    (17, 128, 4096, 0),         # 16 tiles: a cluster of eight k slices
    (32, 250, 2048, 0),         # 32 tiles, ragged: a cluster of four
    (7, 600, 1056, 0),          # 75 tiles over 74 or 148 blocks; 33 chunks
    (5, 8 * 148 + 1, 96, 0),    # one tile more than blocks
    (31, 8 * 148 * 8 + 8, 288, 0),   # nine tiles on one block: two tile groups
    (2, 32000, 1024, 0),        # 28 tiles per block: four tile groups
    (32, 8 * 148 * 64 + 3, 32, 0),   # more than one wave of 64-tile blocks
    (17, 1000, 512, 1), (16, 300, 2080, 3),
    (31, 8 * 148 * 2 - 5, 256, 0),   # the sums: two tiles a block (16 lanes a row), rows that do not fill the warps
    (29, 8 * 148 * 3 + 1, 96, 0),    # four tiles in some blocks, three in the others
    (13, 8 * 148 * 5 + 3, 288, 0),   # six tiles: two columns a lane, the second past the end
    (32, 8880, 512, 0),              # 15 tiles in two groups, a cluster of two
    (32, 12210, 512, 0),             # eleven tiles: no cluster
    (25, 1016, 2048, 0),             # one tile a block: eight lanes a row
])
def test_linear_split_edges(rows, N, K, offset):
    from paper_2602_01274_b200 import binding as b
    dev = "cuda:0"
    w = synth.normal_bf16(5, 13, (N, K), std=0.02, device=dev)
    x = synth.normal_bf16(6, 14, (rows * K + offset,), std=1.0, device=dev)[offset:].view(rows, K)
    y = b.pacer_linear(x, w).cpu().double().numpy()
    out = torch.full((rows, N), float("nan"), device=dev)
    if b._lib.pacer_linear_scratch_bytes(rows, N, K) <= b.PACER_LINEAR_STATIC_BYTES:
        b.pacer_linear_static(x, w, out)
        np.testing.assert_array_equal(out.cpu().double().numpy(), y)
    cols = np.unique(np.concatenate([np.arange(min(N, 24)), np.arange(max(0, N - 24), N),
                                     np.random.default_rng(N + K).integers(0, N, size=min(N, 200))]))
    ref = orc.linear(w[torch.as_tensor(cols, device=dev)].cpu(), x.float().cpu().double().numpy())
    # the inputs are exact in both: fp32 rounding of K sums and products, |x w| ~ 0.02 |x|, stays below
    # K * 2^-24 * sum|x w| / K ~ sqrt(K) * 2^-24 * 4 of the largest output
    assert np.abs(y[:, cols] - ref).max() < 2e-5 * max(1.0, np.abs(ref).max())
