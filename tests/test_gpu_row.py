"""GPU tests of the row-stream decode kernel against the CPU oracle and 64-bit sums: every number of tenants per activation tile
and of tiles per unit, ragged rows, K of one word group to several stages, options, exactness, values without limits; and
the same small shapes on the kernels that it stands in for."""
import numpy as np
import pytest
import torch

import oracle
import paper_2609_36800_b200 as bd
from paper_2609_36800_b200 import synth

from gpu_util import MAX_ABS_TOL, REL_FRO_TOL, assert_parity, run_gemm, to_device, y_to_f64
from test_gpu_parity import SMALL

pytestmark = pytest.mark.gpu

SHAPES = [   # B, m, N, K
    (1, 1, 1, 128), (1, 1, 512, 1024), (1, 8, 130, 1152), (2, 1, 4098, 256), (2, 5, 300, 2048), (2, 8, 149 * 16 + 2, 128),
    (3, 1, 77, 640), (3, 2, 384, 640), (4, 4, 264, 1024), (5, 3, 200, 1280), (7, 1, 4096, 384), (8, 1, 2048, 2048),
    (8, 2, 256, 3072), (9, 8, 100, 512), (16, 1, 768, 2048), (20, 7, 66, 256), (33, 1, 128, 1152), (1, 2, 1024, 14336),
]


@pytest.fixture(params=["row", "others"])
def route(request, monkeypatch):
    monkeypatch.setenv("BITDELTA_ROW", "1" if request.param == "row" else "0")
    return request.param


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "B%d_m%d_N%d_K%d" % s)
def test_matches_oracle(shape, monkeypatch):
    monkeypatch.setenv("BITDELTA_ROW", "1")
    B, m, N, K = shape
    X, W, bits, alpha = synth.make_inputs(synth.Workload("t", B=B, m=m, K=K, N=N, seed=B + m + N + K))
    n0 = bd.kernel_launch_count()
    Y = run_gemm(X, W, bits, alpha)
    assert bd.kernel_launch_count() - n0 == 1
    assert_parity(Y, oracle.gemm(X, W, bits, alpha), str(shape))


@pytest.mark.parametrize("shape", [s for s in SMALL if s[1] <= 8], ids=lambda s: "B%d_m%d_N%d_K%d" % s)
def test_small_shapes_on_the_other_kernels(shape, monkeypatch):
    monkeypatch.setenv("BITDELTA_ROW", "0")
    B, m, N, K = shape
    X, W, bits, alpha = synth.make_inputs(synth.Workload("t", B=B, m=m, K=K, N=N, seed=B * 1000 + m))
    assert_parity(run_gemm(X, W, bits, alpha), oracle.gemm(X, W, bits, alpha), str(shape))


def test_default_route():
    assert bd.gemm_row_stream(1, 1, 4096, 4096) and bd.gemm_row_stream(2, 8, 11008, 4096) and bd.gemm_row_stream(8, 1, 2048, 2048)
    assert not bd.gemm_row_stream(8, 1, 4096, 4096) and not bd.gemm_row_stream(1, 9, 512, 512) and not bd.gemm_row_stream(1, 1, 512, 544)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16])
@pytest.mark.parametrize("act", ["none", "silu", "silu_gate"])
@pytest.mark.parametrize("shape", [(1, 1, 258, 384), (4, 2, 1000, 1152), (6, 3, 130, 256)], ids=str)
def test_options(shape, act, dtype, route):
    B, m, N, K = shape
    g = torch.Generator(device="cuda").manual_seed(N)
    X = torch.randn(B, m, K, device="cuda", generator=g).to(dtype)
    W = (torch.randn(N, K, device="cuda", generator=g) * 0.02).to(dtype)
    bits = torch.randint(-2**31, 2**31, (B, N, K // 32), device="cuda", dtype=torch.int32, generator=g)
    alpha = torch.rand(B, device="cuda", generator=g) * 0.01
    bias = torch.randn(N, device="cuda", generator=g).to(dtype)
    got = bd.gemm(X, W, bits, alpha, bias=bias, act=act).double()
    assert bd.last_device_status()[0] == 0
    S = ((bits.unsqueeze(-1) >> torch.arange(32, device="cuda", dtype=torch.int32)) & 1).reshape(B, N, K).double() * 2 - 1
    z = X.double() @ W.double().t() + alpha.double()[:, None, None] * (X.double() @ S.transpose(1, 2)) + bias.double()
    if act == "silu":
        z = z * torch.sigmoid(z)
    elif act == "silu_gate":
        z = z[..., 0::2] * torch.sigmoid(z[..., 0::2]) * z[..., 1::2]
    assert (got - z).norm() / z.norm() <= REL_FRO_TOL
    # (beyond |z| = 8 the result's own bf16 rounding, 2^-9 |z|, passes the absolute gate)
    assert ((got - z).abs() <= torch.clamp(z.abs() * 2.0**-8, min=MAX_ABS_TOL)).all()


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16])
def test_one_hot_activations_give_the_signs_exactly(dtype, monkeypatch):
    # x = e_k for every k of two words, W = 0, alpha = 1: every sign of the words in its place
    monkeypatch.setenv("BITDELTA_ROW", "1")
    N, K = 70, 1280
    for k0 in (0, 96, 1216):
        for half in range(8):
            ks = torch.arange(k0 + 8 * half, k0 + 8 * half + 8, device="cuda")
            X = torch.zeros(1, 8, K, device="cuda", dtype=dtype)
            X[0, torch.arange(8, device="cuda"), ks] = 1
            bits = torch.randint(-2**31, 2**31, (1, N, K // 32), device="cuda", dtype=torch.int32)
            Y = bd.gemm(X, torch.zeros(N, K, device="cuda", dtype=dtype), bits, torch.ones(1, device="cuda"))
            want = ((bits[0][:, ks // 32] >> (ks % 32).int()) & 1) * 2 - 1
            assert torch.equal(Y[0].t().float(), want.float())


def test_large_small_and_non_finite_activations(monkeypatch):
    monkeypatch.setenv("BITDELTA_ROW", "1")
    B, m, N, K = 2, 4, 130, 512
    rng = np.random.default_rng(3)
    x = rng.standard_normal((B, m, K)).astype(np.float32)
    x[0, 0] = 2.0**100
    x[0, 1, ::2] = 2.0**-130
    x[0, 2] = 3.0                                  # (a mean: the offsets' sums do not cancel)
    x[1, 0, 7] = np.inf
    x[1, 1, 9] = 2.0**125                          # (finite, but 17 of them are not: those outputs term by term)
    x[1, 2, 11] = np.nan
    w = (0.02 * rng.standard_normal((N, K))).astype(np.float32)
    bits = rng.integers(0, 2**32, size=(B, N, K // 32), dtype=np.uint32)
    alpha = np.array([0.5, 0.001], dtype=np.float32)
    X, W = synth.f32_to_bf16_bits(x), synth.f32_to_bf16_bits(w)
    got = run_gemm(X, W, bits, alpha)
    with np.errstate(invalid="ignore"):
        ref = oracle.gemm(X, W, bits, alpha)
    assert np.isnan(got[1, 2]).all()
    assert np.array_equal(np.isinf(got[1, 0]), np.isinf(ref[1, 0])) and np.array_equal(np.sign(got[1, 0]), np.sign(ref[1, 0]), equal_nan=True)
    fin = [(0, 0), (0, 1), (0, 2), (0, 3), (1, 1), (1, 3)]
    for b, t in fin:
        # one output rounding (2^-9) and the sums' 2^-20 of the largest magnitude that enters them
        scale = np.abs(ref[b, t]) * 2.0**-8 + np.abs(x[b, t].astype(np.float64)).max() * K * 2.0**-20
        assert (np.abs(got[b, t] - ref[b, t]) <= scale + 1e-30).all(), (b, t)


def test_no_workspace_is_still_refused():
    wl = synth.Workload("t", B=1, m=1, K=256, N=256, seed=1)
    d = to_device(*synth.make_inputs(wl))
    out = torch.empty(1, 1, 256, dtype=torch.bfloat16, device="cuda")
    with pytest.raises(bd.BitDeltaError):
        bd.gemm(*d, out=out, workspace=torch.empty(16, dtype=torch.uint8, device="cuda"))
    ws = bd.make_workspace(1, 1, 256, 256)
    a = y_to_f64(bd.gemm(*d, out=out, workspace=ws))
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        bd.gemm(*d, out=out, workspace=ws)
    out.zero_()
    g.replay()
    assert np.array_equal(y_to_f64(out), a)
