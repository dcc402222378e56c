"""GPU tests of the paired tiled schedule's token tiles above 128 (two operand buffers, results held in registers while the
next tile runs) against the CPU oracle: each tile size, full and ragged, whole tiles and tiles cut across blocks."""
import pytest

import oracle
import paper_2609_36800_b200 as bd
from paper_2609_36800_b200 import synth

from gpu_util import assert_parity, run_gemm

pytestmark = pytest.mark.gpu

# B, m, N, K                 token tile
SHAPES = [
    ((2, 81, 256, 384), 96),
    ((1, 129, 256, 384), 160),
    ((2, 160, 250, 256), 160),
    ((1, 176, 256, 640), 192),
    ((3, 192, 512, 1152), 192),
    ((1, 193, 256, 128), 128),      # two tiles, the last of 96 columns
    ((2, 512, 512, 1152), 192),     # 192, 192 and 128, cut across blocks
    ((1, 385, 256, 416), 160),      # 160, 160 and 96, K not a multiple of 128
    ((1, 1345, 256, 256), 192),     # seven tiles and one token
    ((2, 350, 512, 384), 192),
    ((80, 144, 250, 128), 160),     # more tiles than pairs of blocks: whole tiles, one behind the other
    ((1, 577, 256, 416), 160),      # K not a multiple of 128, four tiles
]


@pytest.mark.parametrize("shape,tile", SHAPES, ids=lambda s: "B%d_m%d_N%d_K%d" % s if isinstance(s, tuple) else str(s))
def test_matches_oracle(shape, tile):
    B, m, N, K = shape
    plan = bd.gemm_plan(B, m, N, K)
    assert plan["schedule"] == 4 and plan["token_tile"] == tile
    X, W, bits, alpha = synth.make_inputs(synth.Workload("t", B=B, m=m, K=K, N=N, seed=B + m + K))
    assert_parity(run_gemm(X, W, bits, alpha), oracle.gemm(X, W, bits, alpha), str(shape))
