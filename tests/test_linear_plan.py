"""The rules of the stand-alone product on the host: which kernel takes a shape (measured on both sides of each line), and what
the kernels rely on: all blocks of k_linear_wide make the same number of passes, of at most 32 weight rows each."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_01274_b200", "csrc")
SMS = 148


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    src, so = str(d / "plan.cpp"), str(d / "plan.so")
    with open(src, "w") as f:
        f.write('#include "lin_plan.h"\n'
                'extern "C" int wide(int rows, int N, int K) { return lin_wide_takes(rows, N, K, lin_plan(N, K).S); }\n'
                'extern "C" int slices(int N, int K) { return lin_plan(N, K).S; }\n'
                'extern "C" int passes(int N) { LinPasses p = lin_wide_passes(N); return p.np * 1000 + p.per; }\n')
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, "-o", so, src])
    return ctypes.CDLL(so)


@pytest.mark.parametrize("rows,N,K,slices,wide", [
    # several passes and a short k: one pass of k_linear (3.3 us, 4.5 with k_linear_wide; 3.7, 4.0; 5.1, 5.7; 4.7, 5.3) ...
    (1, 13824, 32, 1, False), (8, 5632, 256, 1, False), (17, 10240, 96, 1, False), (1, 10240, 384, 1, False),
    # ... unless there are many token rows, the passes are full, or k is longer (5.9, 5.7; 4.3, 4.0; 4.2, 4.2; 10.1, 9.5)
    (32, 10240, 32, 1, True), (1, 9472, 256, 1, True), (8, 8192, 320, 1, True), (17, 11008, 1024, 1, True),
    # two passes of 18 to 24 rows, a long k, 16 and more token rows (30.7, 35.6; 15.9, 16.5; 21.2, 23.1; 31.8, 35.6)
    (17, 5632, 11008, 1, False), (32, 5632, 4096, 1, False), (16, 5632, 8192, 1, False), (17, 5120, 11008, 2, False),
    # ... and what lies beside these (21.6, 21.3; 16.7, 15.6; 19.1, 17.8)
    (8, 5632, 8192, 1, True), (17, 5120, 4096, 2, True), (17, 8192, 4096, 1, True),
    # one pass; few weight rows that k_linear cuts; more than three passes
    (17, 4096, 11008, 2, True), (5, 2304, 768, 1, True), (1, 150, 256, 1, True), (16, 1536, 8960, 2, False), (17, 2560, 4096, 2, True),
    (1, 1185, 11008, 4, False), (17, 128, 4096, 8, False), (17, 3 * 32 * SMS + 1, 1408, 1, False),
])
def test_which_kernel_takes_a_shape(plan, rows, N, K, slices, wide):
    assert plan.slices(N, K) == slices
    assert bool(plan.wide(rows, N, K)) == wide


def test_blocks_make_the_same_number_of_passes(plan):
    for N in range(1, 3 * 32 * SMS + 1):
        np_, per = divmod(plan.passes(N), 1000)
        units = (N + 1) // 2
        blocks = min(units, SMS)
        base, rem = divmod(units, blocks)
        assert 2 <= per <= 32 and per % 2 == 0
        for b in {0, rem - 1, rem, blocks - 1} & set(range(blocks)):
            r0 = 2 * (b * base + min(b, rem))
            rows = min(N, r0 + 2 * (base + (b < rem))) - r0
            assert -(-rows // per) == np_, (N, b)
