"""The stand-alone product through shared memory at its edges: blocks of one and of two passes side by side, three full passes
and the first shape beyond them, odd weight rows, single rows, and k that ends inside a chunk of 64 columns, with as few as one
chunk.  Checked against the oracle with the tolerance of the other shapes."""
import pytest

from tests import test_gpu_linear as linear

pytestmark = pytest.mark.gpu
SMS = 148


@pytest.mark.parametrize("rows,N,K", [
    (1, 32 * SMS + 2, 96), (17, 32 * SMS + 3, 2080), (32, 34 * SMS - 1, 608), (8, 96 * SMS, 544), (9, 96 * SMS + 1, 544),
    (16, 2 * SMS - 1, 32), (24, 2 * SMS + 1, 160), (31, 18 * SMS + 7, 1120), (32, 16 * SMS, 4128), (15, 64 * SMS + 5, 64),
])
def test_linear_wide_edges(rows, N, K):
    linear.test_linear_split_edges(rows, N, K, 0)
