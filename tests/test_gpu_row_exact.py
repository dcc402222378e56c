"""GPU tests of the row-stream decode kernel's sums: exact wherever every partial sum has a binary32 value, whatever the mean of the
activations, and as fast with infinities or NaN among the activations as without."""
import pytest
import torch

import paper_2609_36800_b200 as bd

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def row_route(monkeypatch):
    monkeypatch.setenv("BITDELTA_ROW", "1")


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16])
@pytest.mark.parametrize("shape", [(1, 1, 300, 14336), (2, 8, 264, 14336), (4, 2, 130, 11008), (8, 1, 130, 14336), (5, 3, 66, 4096), (6, 4, 40, 4224)], ids=str)
def test_sums_of_positive_activations_are_exact(shape, dtype):
    # Activations are positive integers of eight bits, a third of them times sixteen (binary16: all of it times 2^-6): a warp's part
    # of a sum stays below 1792 * 4080 < 2^23 units, so +-x adds up without rounding in any order.  The base term takes two of
    # tenant 0's activations, which are 1 and 1, times minus the high and the middle part of the delta's sum, so that the output
    # is what remains, exactly.  (Sums of larger multiples of x, 17 of them for one, leave binary32's 24 bits.)
    B, m, N, K = shape
    g = torch.Generator(device="cuda").manual_seed(K + B)
    unit = 1.0 if dtype == torch.bfloat16 else 2.0**-6
    X = torch.randint(128, 256, (B, m, K), device="cuda", generator=g).double()
    X *= torch.where(torch.rand(B, m, K, device="cuda", generator=g) < 0.67, 16.0, 1.0) * unit
    X[0, 0, 5] = X[0, 0, 77] = 1
    bits = torch.randint(-2**31, 2**31, (B, N, K // 32), device="cuda", dtype=torch.int32, generator=g)
    S = ((bits[0].unsqueeze(-1) >> torch.arange(32, device="cuda", dtype=torch.int32)) & 1).reshape(N, K).double() * 2 - 1
    d = S @ X[0, 0]
    high = d.to(dtype)
    middle = (d - high.double()).to(dtype)
    W = torch.zeros(N, K, device="cuda", dtype=dtype)
    W[:, 5], W[:, 77] = -high, -middle
    out = bd.gemm(X.to(dtype), W, bits, torch.ones(B, device="cuda"))
    assert torch.equal(out[0, 0].double(), d - high.double() - middle.double())


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_non_finite_activations_do_not_slow_the_call(value):
    B, m, N, K = 1, 1, 4096, 4096
    g = torch.Generator(device="cuda").manual_seed(1)
    X = torch.randn(B, m, K, device="cuda", generator=g).bfloat16()
    W = (torch.randn(N, K, device="cuda", generator=g) * 0.02).bfloat16()
    bits = torch.randint(-2**31, 2**31, (B, N, K // 32), device="cuda", dtype=torch.int32, generator=g)
    alpha, out, ws = torch.rand(B, device="cuda"), torch.empty(B, m, N, device="cuda", dtype=torch.bfloat16), bd.make_workspace(B, m, N, K)

    def us(x):
        best = float("inf")
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(50):
                bd.gemm(x, W, bits, alpha, out=out, workspace=ws)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b) * 20)
        return best

    bad = X.clone()
    bad[0, 0, 3] = value
    us(X)
    usual = us(X)
    assert us(bad) <= 2 * usual      # (40 times as long with every such output summed again by one thread)
    assert not torch.isfinite(out).any()
