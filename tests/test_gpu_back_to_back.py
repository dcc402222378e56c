"""GPU test: many calls in a row of the tiled forms, on two workspaces in turn, give the same bits.  An arrival counter that is not
back at zero, or a stage, sign-word slot or operand buffer handed over too early, would show in some of them."""
import pytest
import torch

import paper_2609_36800_b200 as bd

from gpu_util import MAX_ABS_TOL, REL_FRO_TOL

pytestmark = pytest.mark.gpu

# B, m, N, K                     form
SHAPES = [
    (8, 37, 4096, 4096),       # several tenants per unit, three issuers, teams, tiles cut across blocks
    (6, 40, 1999, 2080),       # ... and sign words copied word by word, odd N
    (3, 160, 1024, 1152),      # pairs of blocks, 160-token tiles cut across pairs
    (2, 130, 512, 2080),       # ... with a short last step
    (3, 70, 640, 1056),        # single blocks, one tenant per unit, short last step
]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "B%d_m%d_N%d_K%d" % s)
def test_calls_in_a_row_give_the_same_bits(shape):
    B, m, N, K = shape
    g = torch.Generator(device="cuda").manual_seed(K)
    X = torch.randn(B, m, K, device="cuda", generator=g).bfloat16()
    W = (torch.randn(N, K, device="cuda", generator=g) * 0.02).bfloat16()
    bits = torch.randint(-2**31, 2**31, (B, N, K // 32), device="cuda", dtype=torch.int32, generator=g)
    alpha = torch.rand(B, device="cuda", generator=g) * 0.01
    spaces = [bd.make_workspace(B, m, N, K) for _ in range(2)]
    outs = [torch.full((B, m, N), float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(10)]
    first = bd.gemm(X, W, bits, alpha, out=torch.empty_like(outs[0]), workspace=spaces[0])
    S = ((bits[0].unsqueeze(-1) >> torch.arange(32, device="cuda", dtype=torch.int32)) & 1).reshape(N, K).double() * 2 - 1
    ref = X[0].double() @ W.double().t() + alpha[0].double() * (X[0].double() @ S.t())
    assert (first[0].double() - ref).abs().max() <= MAX_ABS_TOL and (first[0].double() - ref).norm() / ref.norm() <= REL_FRO_TOL
    for _ in range(30):
        for i, out in enumerate(outs):
            out.fill_(float("nan")) if i == 0 else None
            bd.gemm(X, W, bits, alpha, out=out, workspace=spaces[i % 2])
        assert all(torch.equal(out.view(torch.int16), first.view(torch.int16)) for out in outs)
    assert bd.last_device_status()[0] == 0
