"""Which kernel a call runs on: the queries of the C ABI (CPU), and what the calls themselves show on a GPU."""
import pytest
import torch

import paper_2609_36800_b200 as bd


def test_the_query_takes_the_options_of_the_call():
    shape = (4, 1, 4096, 4096)       # the 4-bit kernel's clusters are ahead, the 8-bit kernel is not
    assert not bd.gemm_row_stream(*shape)
    for options in (dict(fp16=True), dict(bias=True), dict(act="silu"), dict(act="silu_gate"), dict(fp16=True, bias=True, act="silu_gate")):
        assert bd.gemm_row_stream(*shape, **options), options
        assert not bd.gemm_row_stream(*shape, wide_range=True, **options)
    assert bd.gemm_row_stream(1, 1, 512, 512) and not bd.gemm_row_stream(1, 1, 512, 512, wide_range=True)
    assert not bd.gemm_row_stream(1, 9, 512, 512, fp16=True) and not bd.gemm_row_stream(1, 1, 512, 544, bias=True)


@pytest.mark.gpu
@pytest.mark.parametrize("row", ["0", "1"])
@pytest.mark.parametrize("options", [dict(bias=True), dict(act="silu"), dict(act="silu_gate")], ids=str)
def test_calls_clamp_and_flag_large_activations_as_the_query_says(options, row, monkeypatch):
    # 2^17 in one activation: the 8-bit decode kernels clamp it in the delta and flag the call, the row-stream kernel takes it as it is
    monkeypatch.setenv("BITDELTA_ROW", row)
    B, m, N, K = 3, 2, 264, 512
    g = torch.Generator(device="cuda").manual_seed(1)
    X = torch.randn(B, m, K, device="cuda", generator=g).bfloat16()
    X[1, 0, 7] = 2.0**17
    W = (torch.randn(N, K, device="cuda", generator=g) * 0.02).bfloat16()
    bits = torch.randint(-2**31, 2**31, (B, N, K // 32), device="cuda", dtype=torch.int32, generator=g)
    bias = torch.randn(N, device="cuda", generator=g).bfloat16() if options.get("bias") else None
    bd.last_device_status()
    bd.gemm(X, W, bits, torch.ones(B, device="cuda"), bias=bias, act=options.get("act", "none"))
    assert bd.gemm_row_stream(B, m, N, K, **options) == (row == "1")
    assert bd.last_device_status()[0] == (0 if row == "1" else bd.binding.STATUS_RANGE)


@pytest.mark.parametrize("shape,plain,options", [   # B, m, N, K
    ((19, 5, 3642, 512), False, False), ((9, 6, 7192, 512), False, False), ((10, 5, 3274, 1024), True, True),   # eight, ten, five rounds
    ((12, 1, 1220, 3200), False, False), ((9, 1, 1550, 2432), False, True),                                      # a second round of six units
    ((2, 8, 5632, 11008), False, False), ((2, 6, 8192, 8192), False, True), ((2, 8, 11008, 14336), True, True),  # rounds partly empty, full
    ((2, 4, 8192, 8192), True, True), ((1, 8, 8192, 8192), True, True),
], ids=str)
def test_row_stream_range(shape, plain, options):
    assert bd.gemm_row_stream(*shape) == plain
    assert bd.gemm_row_stream(*shape, fp16=True, bias=True, act="silu_gate") == options
