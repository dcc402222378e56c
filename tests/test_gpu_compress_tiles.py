"""GPU tests of the compress step where its tiles of 8192 elements end: whole and partial last tiles, one word, more tiles than blocks, more
tenants than are staged at once, and both."""
import numpy as np
import pytest
import torch

import oracle
import paper_2609_36800_b200 as bd
from paper_2609_36800_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 1, 32), (2, 255, 32), (2, 256, 32), (3, 257, 32), (1, 2369, 1024), (2, 300, 8192 + 96), (33, 17, 512), (35, 2400, 1024)], ids=str)
def test_tile_edges(shape):
    B, N, K = shape
    fine, W = synth.make_fine_weights(B, N, K, seed=B + N + K)
    up = lambda a: torch.from_numpy(a.view(np.int16)).cuda().view(torch.bfloat16)
    # (results and one word behind them: nothing is written past the end)
    bits = torch.full((B * N * (K // 32) + 1,), 0x5A5A5A5A, dtype=torch.int32, device="cuda")
    alpha = torch.empty(B, device="cuda")
    bd.compress(up(fine), up(W), bits=bits[:-1].view(B, N, K // 32), alpha=alpha)
    ref_bits, ref_alpha = oracle.compress(fine, W)
    assert bd.last_device_status()[0] == 0 and bits[-1].item() == 0x5A5A5A5A
    assert np.array_equal(bits[:-1].cpu().numpy().view(np.uint32).reshape(ref_bits.shape), ref_bits)
    # |delta| in fp32 (2^-24 each), four of them added in fp32 (3 * 2^-24), the rest in double
    assert np.allclose(alpha.cpu().numpy(), ref_alpha, rtol=1e-6, atol=0)
