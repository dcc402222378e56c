"""GPU parity of the 8-bit decode kernels' general form (binary16, bias, activations) at the sizes that the row-stream kernel has by
default: every instantiation by token count, the in-kernel and the pre-pass split, tiles cut across blocks in one list and in
teams, several tiles per block, whole tiles dealt in turn, ragged N."""
import pytest

import oracle
import paper_2609_36800_b200 as bd
from paper_2609_36800_b200 import synth

from gpu_util import assert_parity
from test_gpu_gemm_ex import run_ex

pytestmark = pytest.mark.gpu

# B, m, N, K               schedule (1 pre-pass split, 2 in-kernel), order (0 one list, 1 whole units, 2 teams)
SHAPES = [
    ((6, 1, 264, 1024), 2, 0),
    ((17, 2, 1400, 640), 2, 2),
    ((8, 3, 900, 512), 1, 0),
    ((4, 4, 300, 640), 2, 0),
    ((9, 4, 520, 512), 1, 0),
    ((16, 4, 1400, 1024), 1, 2),
    ((24, 4, 6400, 256), 1, 2),
    ((1, 8, 130, 2048), 2, 0),
    ((3, 8, 264, 1024), 1, 0),
    ((9, 8, 520, 512), 1, 0),
    ((32, 8, 640, 1152), 1, 2),
    ((240, 8, 890, 256), 1, 1),
]


@pytest.fixture(autouse=True)
def eight_bit_route(monkeypatch):
    monkeypatch.setenv("BITDELTA_ROW", "0")
    monkeypatch.setenv("BITDELTA_FP4", "0")      # (for the plan query and the calls without options)


@pytest.mark.parametrize("opts", [("f16", True, "none"), ("f16", True, "silu_gate"), ("bf16", False, "silu"), ("bf16", False, "none")],
                         ids=lambda o: "%s_%s_%s" % (o[0], "bias" if o[1] else "nobias", o[2]))
@pytest.mark.parametrize("shape,schedule,order", SHAPES, ids=lambda s: "B%d_m%d_N%d_K%d" % s if isinstance(s, tuple) else str(s))
def test_matches_oracle(shape, schedule, order, opts):
    B, m, N, K = shape
    dtype, bias, act = opts
    p = bd.gemm_plan(B, m, N, K)
    assert (p["schedule"], p["order"]) == (schedule, order)
    wl = synth.Workload("t", B=B, m=m, K=K, N=N, seed=B * 100 + m)
    if dtype == "f16":
        X, W, bits, alpha, b = synth.make_inputs_f16(wl)
    else:
        X, W, bits, alpha = synth.make_inputs(wl)
    b = b if bias else None
    assert_parity(run_ex(X, W, bits, alpha, b, dtype, act), oracle.gemm_ex(X, W, bits, alpha, bias=b, dtype=dtype, act=act), f"{shape} {opts}")


def test_f16_pieces_of_full_precision_activations_are_exact():
    # as test_gpu_gemm_ex's test of the delta term, on the kernel that splits the activations into pieces
    from test_gpu_gemm_ex import test_f16_delta_term_is_exact_for_full_precision_activations as check
    check()
