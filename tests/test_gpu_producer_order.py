"""GPU tests of a product queued behind a compress call that writes its sign words and scales, with other work in between: the product fetches
both before the kernel ahead of it has ended unless it is told not to.  Everything is queued behind a kernel that idles for a while, so
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
        base = 0.02 * rng.standard_normal((N, K), dtype=np.float32)
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
