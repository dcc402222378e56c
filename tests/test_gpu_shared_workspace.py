"""GPU test: calls of one shape that take different plans (decode, wide range; on pairs of blocks or not) may share a workspace.
Each leaves partial results in it, none may leave them where another counts arrivals."""
import pytest
import torch

import paper_2609_36800_b200 as bd

from gpu_util import MAX_ABS_TOL, REL_FRO_TOL

pytestmark = pytest.mark.gpu


def _inputs(B, m, N, K):
    g = torch.Generator(device="cuda").manual_seed(B + m + N)
    X = torch.randn(B, m, K, device="cuda", generator=g).bfloat16()
    W = (torch.randn(N, K, device="cuda", generator=g) * 0.02).bfloat16()
    bits = torch.randint(-2**31, 2**31, (B, N, K // 32), device="cuda", dtype=torch.int32, generator=g)
    alpha = torch.rand(B, device="cuda", generator=g) * 0.01
    S = ((bits.unsqueeze(-1) >> torch.arange(32, device="cuda", dtype=torch.int32)) & 1).reshape(B, N, K).double() * 2 - 1
    return (X, W, bits, alpha), X.double() @ W.double().t() + alpha.double()[:, None, None] * (X.double() @ S.transpose(1, 2))


def _check(args, ref, ws, what, **kw):
    out = torch.full(ref.shape, float("nan"), dtype=torch.bfloat16, device="cuda")
    d = bd.gemm(*args, out=out, workspace=ws, **kw).double() - ref
    assert d.abs().max() <= MAX_ABS_TOL and d.norm() / ref.norm() <= REL_FRO_TOL, what


# Decode in two groups of four tenants, wide range in one of eight: 259 and 130 arrival counters, i.e. more and less than 1 KB;
# the wide-range plan's first block has less than a tile of eight steps, so it writes the first slot of partial results.
@pytest.mark.parametrize("shape", [(5, 10, 16512, 1024), (8, 12, 16500, 1024)], ids=str)
def test_decode_and_wide_range(shape, monkeypatch):
    monkeypatch.setenv("BITDELTA_ROW", "0")
    args, ref = _inputs(*shape)
    ws = bd.make_workspace(*shape)
    for i in range(3):
        _check(args, ref, ws, f"decode {i}")
        _check(args, ref, ws, f"wide range {i}", wide_range=True)


# 130 tokens are one token tile on pairs and two on single blocks: 131 and 261 arrival counters
@pytest.mark.parametrize("shape", [(1, 130, 16640, 2048), (1, 130, 16600, 2016)], ids=str)
def test_pairs_and_single_blocks(shape, monkeypatch):
    args, ref = _inputs(*shape)
    ws = bd.make_workspace(*shape)
    for i in range(3):
        monkeypatch.setenv("BITDELTA_PAIR", "1")
        _check(args, ref, ws, f"pairs {i}")
        monkeypatch.setenv("BITDELTA_PAIR", "0")
        _check(args, ref, ws, f"single blocks {i}")
