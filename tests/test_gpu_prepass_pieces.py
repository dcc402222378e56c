"""GPU test of the 8-bit decode kernels' pre-pass: one activation per token row, W_base zero, scale one, so the output is the activation
with a sign, which only exact pieces give back."""
import pytest
import torch

import paper_2609_36800_b200 as bd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,K", [(8, 128), (5, 384), (16, 256)])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16])
def test_every_mantissa_is_exact(dtype, m, K, monkeypatch):
    monkeypatch.setenv("BITDELTA_FP4", "0")
    monkeypatch.setenv("BITDELTA_ROW", "0")
    B, N = 24, 130
    assert bd.gemm_plan(B, m, N, K)["schedule"] == 1
    # every mantissa (binary16: an odd stride through them) at every exponent whose last bit is 2^-16 (e5m2's smallest value) or more
    bits_, top = (7, 15) if dtype == torch.bfloat16 else (10, 15)
    mant = torch.arange(0, 2**bits_, 1 if bits_ == 7 else 13, dtype=torch.float64)
    x = torch.cat([(1 + mant / 2**bits_) * 2.0**e for e in range(-16 + bits_, top + 1)] + [torch.zeros(1, dtype=torch.float64)])
    x = torch.cat([x, -x]).to(dtype).cuda()
    g = torch.Generator(device="cuda").manual_seed(m + K)
    words = torch.randint(-2**31, 2**31, (B, N, K // 32), device="cuda", dtype=torch.int32, generator=g)
    sign = ((words.unsqueeze(-1) >> torch.arange(32, device="cuda", dtype=torch.int32)) & 1).reshape(B, N, K) * 2 - 1
    W, alpha = torch.zeros(N, K, device="cuda", dtype=dtype), torch.ones(B, device="cuda")
    out, ws = torch.empty(B, m, N, device="cuda", dtype=dtype), bd.make_workspace(B, m, N, K)
    for i in range(0, x.numel(), B * m):
        v = torch.zeros(B * m, device="cuda", dtype=dtype)
        v[:x[i:i + B * m].numel()] = x[i:i + B * m]
        k = (torch.arange(B * m, device="cuda") * 7 + i) % K
        X = torch.zeros(B * m, K, device="cuda", dtype=dtype)
        X[torch.arange(B * m, device="cuda"), k] = v
        bd.gemm(X.view(B, m, K), W, words, alpha, out=out, workspace=ws)
        s = sign.gather(2, k.view(B, 1, m).expand(B, N, m)).transpose(1, 2).to(dtype)
        assert torch.equal(out, s * v.view(B, m, 1))
    assert bd.last_device_status()[0] == 0
