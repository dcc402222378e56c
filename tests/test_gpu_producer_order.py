"""GPU tests of the order between products and compress calls on the same buffers.  A product queued behind a compress call, with other work in
between, fetches sign words and scales before the kernel ahead of it has ended unless it is told not to; a compress call queued behind a
product or another compress call is launched early, too, and has to wait before it writes.  Everything is queued behind a kernel that idles for a while, so
that each call finds the one before it still running or not yet begun."""
import numpy as np
import pytest
import torch

import oracle
import paper_2609_36800_b200 as bd
from paper_2609_36800_b200 import synth

from gpu_util import assert_parity, y_to_f64

pytestmark = pytest.mark.gpu

ROUNDS = 4
IDLE_CYCLES = 3_000_000   # 1.5 ms: longer than the host takes to queue a round

# B, m, N, K           kernel of the product
SHAPES = [
    (2, 1, 256, 512),    # row-stream; a matrix of sixteen compress tiles
    (3, 2, 4096, 2048),  # 4-bit decode, clusters; more tiles than blocks
    (5, 8, 2048, 4096),  # 8-bit decode, pre-pass
    (2, 48, 256, 384),   # tiled
    (1, 130, 256, 512),  # tiled on pairs
]


def up(a):
    return torch.from_numpy(a.view(np.int16)).cuda().view(torch.bfloat16)


class Call:
    """Buffers of one product whose signs come from compress, rewritten each round, and what each round should give."""

    def __init__(self, B, m, N, K):
        rng = np.random.default_rng(B + m + N)
        X = synth.f32_to_bf16_bits(rng.standard_normal((B, m, K), dtype=np.float32))
        # (smaller weights where K is long, as in the down projections: outputs stay below 8, where rounding to bfloat16 alone is 1.6e-2)
        base = np.float32(0.02 if K <= 4096 else 0.01) * rng.standard_normal((N, K), dtype=np.float32)
        W = synth.f32_to_bf16_bits(base)
        fine = [synth.f32_to_bf16_bits(base + 0.004 * rng.standard_normal((B, N, K), dtype=np.float32)) for _ in range(ROUNDS)]
        self.X, self.W, self.fine = up(X), up(W), [up(f) for f in fine]
        self.bits = torch.zeros((B, N, K // 32), dtype=torch.int32, device="cuda")
        self.alpha = torch.zeros(B, device="cuda")
        self.outs = [torch.zeros((B, m, N), dtype=torch.bfloat16, device="cuda") for _ in range(ROUNDS)]
        self.ws = bd.make_workspace(B, m, N, K)
        self.refs = [oracle.gemm(X, W, *oracle.compress(f, W)) for f in fine]

    def product(self, out):
        bd.gemm(self.X, self.W, self.bits, self.alpha, out=out, workspace=self.ws)

    def check(self, what):
        assert bd.last_device_status()[0] == 0
        for r in range(ROUNDS):
            assert_parity(y_to_f64(self.outs[r]), self.refs[r], f"{what}, round {r}")


def elsewhere():
    """A product of other weights, on buffers of its own."""
    g = torch.Generator(device="cuda").manual_seed(1)
    X, W = torch.randn(2, 1, 512, device="cuda", generator=g).bfloat16(), torch.randn(256, 512, device="cuda", generator=g).bfloat16()
    bits, alpha = torch.zeros(2, 256, 16, dtype=torch.int32, device="cuda"), torch.ones(2, device="cuda")
    out, ws = torch.empty(2, 1, 256, dtype=torch.bfloat16, device="cuda"), bd.make_workspace(2, 1, 256, 512)
    return lambda: bd.gemm(X, W, bits, alpha, out=out, workspace=ws)


@pytest.mark.parametrize("shape", SHAPES, ids=str)
def test_product_on_another_stream_in_between(shape):
    call, other = Call(*shape), elsewhere()
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(a):
        torch.cuda._sleep(IDLE_CYCLES)
        for r in range(ROUNDS):
            bd.compress(call.fine[r], call.W, bits=call.bits, alpha=call.alpha)
            with torch.cuda.stream(b):
                other()
            call.product(call.outs[r])
    torch.cuda.synchronize()
    call.check("two streams")


@pytest.mark.parametrize("shape", SHAPES, ids=str)
def test_product_behind_an_event_of_the_producer(shape):
    call, other = Call(*shape), elsewhere()
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(a):
        torch.cuda._sleep(IDLE_CYCLES)
    for r in range(ROUNDS):
        with torch.cuda.stream(a):
            a.wait_stream(b)   # (the product before has read the buffers)
            bd.compress(call.fine[r], call.W, bits=call.bits, alpha=call.alpha)
            other()            # (... on the producer's own stream)
        with torch.cuda.stream(b):
            b.wait_stream(a)
            call.product(call.outs[r])
    torch.cuda.synchronize()
    call.check("event")


@pytest.mark.parametrize("shape", SHAPES, ids=str)
def test_captured_with_a_product_elsewhere_during_the_capture(shape):
    call, other = Call(*shape), elsewhere()
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    fine, out = call.fine[0].clone(), torch.empty_like(call.outs[0])
    with torch.cuda.stream(a):
        call.product(out)
    with torch.cuda.stream(b):
        other()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=a, capture_error_mode="relaxed"):
        bd.compress(fine, call.W, bits=call.bits, alpha=call.alpha)
        with torch.cuda.stream(b):
            other()
        call.product(out)
    torch.cuda.synchronize()
    with torch.cuda.stream(a):
        torch.cuda._sleep(IDLE_CYCLES)
        for r in range(ROUNDS):
            fine.copy_(call.fine[r])
            graph.replay()
            call.outs[r].copy_(out)
    torch.cuda.synchronize()
    call.check("captured")
    # the recorded product does not speak for the stream itself: eager calls on it afterwards
    call.bits.zero_()
    torch.cuda.synchronize()
    with torch.cuda.stream(a):
        torch.cuda._sleep(IDLE_CYCLES)
        for r in range(ROUNDS):
            bd.compress(call.fine[r], call.W, bits=call.bits, alpha=call.alpha)
            call.product(call.outs[r])
    torch.cuda.synchronize()
    call.check("after the capture")


# Few blocks and a long K: the compress call that follows has room to begin while the product runs
BEHIND = SHAPES + [(2, 1, 128, 14336), (3, 8, 128, 8192), (2, 48, 128, 8192)]


@pytest.mark.parametrize("shape", BEHIND, ids=str)
def test_compress_waits_for_the_product_that_reads_what_it_overwrites(shape):
    call = Call(*shape)
    alone = []
    for r in range(ROUNDS):
        bd.compress(call.fine[r], call.W, bits=call.bits, alpha=call.alpha)
        torch.cuda.synchronize()
        call.product(call.outs[r])
        torch.cuda.synchronize()
        alone.append((call.bits.clone(), call.alpha.clone(), call.outs[r].clone()))
    call.check("alone")
    for out in call.outs:
        out.zero_()
    bd.compress(call.fine[0], call.W, bits=call.bits, alpha=call.alpha)
    torch.cuda.synchronize()
    torch.cuda._sleep(IDLE_CYCLES)
    for r in range(ROUNDS):
        call.product(call.outs[r])
        bd.compress(call.fine[(r + 1) % ROUNDS], call.W, bits=call.bits, alpha=call.alpha)
    torch.cuda.synchronize()
    for r in range(ROUNDS):
        assert torch.equal(call.outs[r], alone[r][2]), r
    assert torch.equal(call.bits, alone[0][0]) and torch.equal(call.alpha, alone[0][1])
    assert bd.last_device_status()[0] == 0


@pytest.mark.parametrize("B,N,K", [(1, 8, 32), (5, 130, 1056), (8, 600, 4096), (40, 64, 1024)])
def test_compress_calls_in_a_row_share_buffers(B, N, K):
    # one buffer of sign words and one of partial sums (the allocator hands the same one out again) for all, a scale buffer each
    g = torch.Generator(device="cuda").manual_seed(N)
    W = (torch.randn(N, K, device="cuda", generator=g) * 0.02).bfloat16()
    fine = [(W + torch.randn(B, N, K, device="cuda", generator=g) * 0.004 * (r + 1)).bfloat16() for r in range(6)]
    alone = []
    for f in fine:
        alone.append(bd.compress(f, W))
        torch.cuda.synchronize()
    bits = torch.empty(B, N, K // 32, dtype=torch.int32, device="cuda")
    alphas = torch.zeros(6, B, device="cuda")
    torch.cuda.synchronize()
    torch.cuda._sleep(IDLE_CYCLES)
    for r, f in enumerate(fine):
        bd.compress(f, W, bits=bits, alpha=alphas[r])
    torch.cuda.synchronize()
    for r in range(6):
        assert torch.equal(alphas[r], alone[r][1]), r
    assert torch.equal(bits, alone[-1][0])
    # ... and one scale buffer for all, copied out behind each call
    copies = []
    torch.cuda._sleep(IDLE_CYCLES)
    for f in fine:
        bd.compress(f, W, bits=bits, alpha=alphas[0])
        copies.append((bits.clone(), alphas[0].clone()))
    torch.cuda.synchronize()
    for (b, a), (rb, ra) in zip(copies, alone):
        assert torch.equal(b, rb) and torch.equal(a, ra)
    assert bd.last_device_status()[0] == 0
