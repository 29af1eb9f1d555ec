"""The stand-alone skinny product at the edges of its split: 1 to 64 weight tiles per block, one to eight k slices per
cluster, row counts around the 16-row operand, ragged N, short k and activations that are not 16-byte aligned (an odd offset:
these are always k_linear's; which aligned shapes are, tests/test_linear_plan.py).  The C entry point with the caller's scratch and
the one without it give the same bytes."""
import numpy as np
import pytest
import torch

from oracle import pacer_oracle as orc
from paper_2602_01274_b200 import synth

pytestmark = pytest.mark.gpu


def c_linear(b, x, w, short=0, offset=0):
    """(status, output) of the C entry point with the caller's scratch: `short` bytes fewer than it asks for, `offset` bytes past
    the alignment."""
    rows, K, N = x.shape[0], x.shape[1], w.shape[0]
    need = b._lib.pacer_linear_scratch_bytes(rows, N, K)
    scratch = torch.empty(need + 512, dtype=torch.uint8, device=x.device)
    y = torch.full((rows, N), float("nan"), device=x.device)
    rc = b._lib.pacer_linear(x.data_ptr(), w.data_ptr(), y.data_ptr(), rows, N, K, (scratch.data_ptr() + 255) // 256 * 256 + offset,
                             need - short, torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    return rc, y


@pytest.mark.parametrize("rows,N,K,offset", [
    (1, 1, 32, 0),              # one tile, one chunk
    (16, 9, 64, 0),             # a ragged second tile; fewer chunks than warps
    (17, 128, 4096, 0),         # k_linear, 16 tiles: a cluster of eight k slices
    (32, 250, 2048, 0),         # 32 tiles, ragged: a cluster of four
    (7, 600, 1056, 0),          # 75 tiles over 74 or 148 blocks; 33 chunks
    (5, 8 * 148 + 1, 96, 0),    # one tile more than blocks
    (31, 8 * 148 * 8 + 8, 288, 0),   # three passes of k_linear_wide
    (2, 32000, 1024, 0),        # k_linear, 28 tiles per block: four tile groups
    (32, 8 * 148 * 64 + 3, 32, 0),   # more than one wave of 64-tile blocks
    (17, 1000, 512, 1), (16, 300, 2080, 3),
    (31, 8 * 148 * 2 - 5, 256, 0), (29, 8 * 148 * 3 + 1, 96, 0), (13, 8 * 148 * 5 + 3, 288, 0), (32, 8880, 512, 0), (32, 12210, 512, 0),
    (25, 1016, 2048, 0),
    # k_linear's sums and groups: one tile a block (eight lanes a row)
    (25, 1016, 2048, 1), (5, 8 * 148 + 1, 96, 3),
    (31, 8 * 148 * 2 - 5, 256, 1),   # two tiles a block (16 lanes a row), rows that do not fill the warps
    (29, 8 * 148 * 3 + 1, 96, 3),    # four tiles in some blocks, three in the others
    (13, 8 * 148 * 5 + 3, 288, 1),   # six tiles: two columns a lane, the second past the end
    (31, 8 * 148 * 8 + 8, 288, 1),   # nine tiles on one block: two tile groups
    (32, 8880, 512, 3),              # 15 tiles in two groups, a cluster of two
    (17, 4096, 2080, 1),             # seven tiles, a cluster of two
    (32, 12210, 512, 1),             # eleven tiles: no cluster
    (16, 1536, 8960, 0), (3, 1437, 11008, 0),        # aligned, a cluster of two, three tiles
    (8, 5632, 256, 0), (1, 10251, 96, 0),            # aligned, five and ten tiles: a short k
    (17, 5627, 4096, 0), (16, 5120, 8192, 0),        # ... a long k, one slice and two
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
    rc, scratched = c_linear(b, x, w)
    assert rc == 0
    np.testing.assert_array_equal(scratched.cpu().double().numpy(), y)
    cols = np.unique(np.concatenate([np.arange(min(N, 24)), np.arange(max(0, N - 24), N),
                                     np.random.default_rng(N + K).integers(0, N, size=min(N, 200))]))
    ref = orc.linear(w[torch.as_tensor(cols, device=dev)].cpu(), x.float().cpu().double().numpy())
    # the inputs are exact in both: fp32 rounding of K sums and products, |x w| ~ 0.02 |x|, stays below
    # K * 2^-24 * sum|x w| / K ~ sqrt(K) * 2^-24 * 4 of the largest output
    assert np.abs(y[:, cols] - ref).max() < 2e-5 * max(1.0, np.abs(ref).max())


@pytest.mark.parametrize("rows,N,K", [(5, 2304, 768), (17, 4096, 11008)])
def test_scratch_that_is_too_small_or_misaligned_is_refused(rows, N, K):
    from paper_2602_01274_b200 import binding as b
    x = torch.zeros(rows, K, dtype=torch.bfloat16, device="cuda:0")
    w = torch.zeros(N, K, dtype=torch.bfloat16, device="cuda:0")
    assert c_linear(b, x, w)[0] == 0
    for kw, text in ((dict(short=1), "scratch too small"), (dict(offset=16), "misaligned pointer")):
        rc, y = c_linear(b, x, w, **kw)
        assert rc != 0 and text in b._lib.pacer_last_error(None).decode() and torch.isnan(y).all()
