"""The rule that picks the few-row kernel's variant, on the host: the next longer pass where it saves more than one pass for three
layers (measured on both sides, see few_plan.h)."""
import ctypes
import os
import subprocess

import pytest

from paper_2602_01274_b200 import synth

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_01274_b200", "csrc")


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    src, so = str(d / "plan.cpp"), str(d / "plan.so")
    with open(src, "w") as f:
        f.write('#include "few_plan.h"\nextern "C" int atoms(int l, int qkv, int gu, int v) { return few_pass_atoms(l, qkv, gu, v, 148); }\n')
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, "-o", so, src])
    return ctypes.CDLL(so)


S = synth.ModelShape


@pytest.mark.parametrize("shape,head,atoms", [
    (S(4, 256, 4, 4, 1024, 4096), True, 16), (S(2, 768, 12, 12, 3072, 32000), True, 16), (S(24, 2048, 16, 16, 5504, 32256), True, 16),
    (S(4, 3072, 24, 8, 8192, 32000), True, 16),           # 14 atoms of the gate/up projection
    (S(1, 4608, 36, 12, 9472, 0), False, 16),             # 16: the last of one short pass
    (S(1, 4608, 36, 12, 9480, 0), False, 24),             # 18
    (S(4, 4096, 32, 32, 11008, 32000), True, 24), (S(4, 5120, 40, 40, 13824, 32000), True, 24),
    (S(4, 5120, 40, 8, 14216, 32000), True, 26),          # 26
    (S(4, 5120, 40, 8, 17408, 32000), True, 16),          # 30: two passes in any case
    (S(14, 7168, 56, 8, 19200, 32256), True, 24), (S(3, 5120, 40, 8, 27648, 32000), True, 24),
    (S(3, 8192, 64, 8, 28672, 32000), True, 26),          # 50: four, three and two passes
    (S(28, 1536, 12, 2, 8960, 151936), True, 16),         # the LM head: three more passes, 28 layers
    (S(4, 1536, 12, 2, 8960, 151936), True, 24),          # ... four layers
    (S(1, 4096, 32, 32, 11008, 0), False, 24),            # a pre-verification layer
    (S(1, 8192, 64, 64, 1024, 0), False, 24),             # the q/k/v projection: 22 atoms
])
def test_atoms_of_a_pass(plan, shape, head, atoms):
    assert plan.atoms(shape.n_layers, shape.qkv_rows, 2 * shape.d_ffn, shape.vocab if head else 0) == atoms
