"""GPU tests of the tiled schedule for K that is a multiple of 32 but not of 128 (the last k-step is short, the sign words
come word by word) against the CPU oracle: each remainder, one step and an odd / even number of them, the several-tenants,
one-tenant and paired forms, tiles cut across thread blocks, ragged N, and the calls that stay on the CUDA-core kernel."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
import paper_2609_36800_b200 as bd
from paper_2609_36800_b200 import synth

from gpu_util import MAX_ABS_TOL, REL_FRO_TOL, assert_parity, errors, run_gemm, to_device, y_to_f64

pytestmark = pytest.mark.gpu

# B, m, N, K                 schedule (0 tiled, 4 on pairs, 3 CUDA-core)
SHAPES = [
    ((1, 1, 128, 160), 3),      # one token, small matrix
    ((1, 2, 128, 160), 0),      # one full step and 32 k
    ((1, 1, 1985, 544), 0),     # one token, just past the small matrices
    ((8, 1, 1026, 192), 0),     # eight tenants per unit, 64 k left, ragged N
    ((11, 3, 200, 224), 0),     # two groups of tenants, 96 k left
    ((2, 16, 127, 1056), 0),
    ((3, 20, 264, 352), 0),     # several tenants per unit, three steps
    ((6, 40, 1999, 2080), 0),   # teams, tiles cut across blocks, odd N
    ((2, 65, 128, 416), 0),     # one tenant per unit
    ((2, 130, 256, 672), 4),    # pairs, ragged token tile
    ((3, 96, 512, 1888), 4),
    ((2, 3, 96, 96), 3),
]


@pytest.mark.parametrize("shape,schedule", SHAPES, ids=lambda s: "B%d_m%d_N%d_K%d" % s if isinstance(s, tuple) else str(s))
def test_matches_oracle(shape, schedule):
    B, m, N, K = shape
    assert bd.gemm_plan(B, m, N, K)["schedule"] == schedule
    X, W, bits, alpha = synth.make_inputs(synth.Workload("t", B=B, m=m, K=K, N=N, seed=B + m + K))
    assert_parity(run_gemm(X, W, bits, alpha), oracle.gemm(X, W, bits, alpha), str(shape))


def test_products_past_the_end_of_a_row_do_not_count():
    # K = 160: what follows a row in memory is the next row; with infinities at the start of every row but the first,
    # only those rows' own outputs may be affected (each row's own infinity is at its k = 0)
    B, m, N, K = 1, 17, 4, 160
    X, W, bits, alpha = synth.make_inputs(synth.Workload("t", B=B, m=m, K=K, N=N, seed=3))
    W[1:, 0] = 0x7F80
    X[0, 1:, 0] = 0
    got = run_gemm(X, W, bits, alpha)
    assert np.isfinite(got[:, :, 0]).all()
    W[1:, 0] = 0
    assert_parity(got[:, :, :1], oracle.gemm(X, W, bits, alpha)[:, :, :1])


def test_without_scratch_the_call_runs_on_the_cuda_core_kernel():
    B, m, N, K = 2, 20, 130, 224
    wl = synth.Workload("t", B=B, m=m, K=K, N=N, seed=5)
    X, W, bits, alpha = synth.make_inputs(wl)
    d = to_device(X, W, bits, alpha)
    ref = oracle.gemm(X, W, bits, alpha)
    Y = torch.empty((B, m, N), dtype=torch.bfloat16, device="cuda")
    st = bd.load_library().bitdelta_gemm(*[ctypes.c_void_p(t.data_ptr()) for t in d], ctypes.c_void_p(Y.data_ptr()), B, m, N, K,
                                         None, 0, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == 0
    assert_parity(y_to_f64(Y), ref)
    bd.gemm_noalloc(*d, Y)          # (scratch of the library: the tiled schedule)
    max_abs, rel_fro = errors(y_to_f64(Y), ref)
    assert max_abs <= MAX_ABS_TOL and rel_fro <= REL_FRO_TOL


@pytest.mark.parametrize("act", ["none", "silu", "silu_gate"])
def test_binary16_with_options(act):
    B, m, N, K = 5, 33, 258, 736
    g = torch.Generator(device="cuda").manual_seed(7)
    X = torch.randn(B, m, K, device="cuda", generator=g).half()
    W = (torch.randn(N, K, device="cuda", generator=g) * 0.02).half()
    bits = torch.randint(-2**31, 2**31, (B, N, K // 32), device="cuda", dtype=torch.int32, generator=g)
    alpha = torch.rand(B, device="cuda", generator=g) * 0.01
    bias = torch.randn(N, device="cuda", generator=g).half()
    got = bd.gemm(X, W, bits, alpha, bias=bias, act=act).double()
    S = ((bits.unsqueeze(-1) >> torch.arange(32, device="cuda", dtype=torch.int32)) & 1).reshape(B, N, K).double() * 2 - 1
    z = X.double() @ W.double().t() + alpha.double()[:, None, None] * (X.double() @ S.transpose(1, 2)) + bias.double()
    if act == "silu":
        z = z * torch.sigmoid(z)
    elif act == "silu_gate":
        z = z[..., 0::2] * torch.sigmoid(z[..., 0::2]) * z[..., 1::2]
    assert (got - z).norm() / z.norm() <= REL_FRO_TOL and (got - z).abs().max() <= MAX_ABS_TOL
