"""The stand-alone product through shared memory at its edges: one full pass and the first shape of two, three full passes and the
first shape beyond them (k_linear's), odd weight rows, single rows, k that ends inside a chunk of 64 columns, with as few as one
chunk, and the first k on its side of the lines where k_linear takes several passes.  Checked against the oracle with the tolerance of
the other shapes."""
import pytest

from tests import test_gpu_linear as linear

pytestmark = pytest.mark.gpu
SMS = 148


@pytest.mark.parametrize("rows,N,K", [
    (1, 32 * SMS + 2, 96), (17, 32 * SMS + 3, 2080), (32, 34 * SMS - 1, 608), (8, 96 * SMS, 544), (9, 96 * SMS + 1, 544),
    (16, 2 * SMS - 1, 32), (24, 2 * SMS + 1, 160), (31, 18 * SMS + 7, 1120), (32, 16 * SMS, 4128), (15, 64 * SMS + 5, 64),
    (1, 32 * SMS, 96), (32, 32 * SMS, 160), (32, 32 * SMS + 1, 160), (32, 32 * SMS + 2, 96), (7, 5632, 672), (1, 13825, 320), (16, 10240, 160),
])
def test_linear_wide_edges(rows, N, K):
    linear.test_linear_split_edges(rows, N, K, 0)
