"""When the memory of a weight or a rotation may be released: while a stream is being captured, while launches still read it."""
import numpy as np
import pytest
import torch

from paper_2506_13472_b200 import binding as rb
from paper_2506_13472_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture()
def ctx():
    c = rb.Context(0)
    yield c
    c.close()


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def weight(ctx, key, d_in=512, d_out=384):
    return ctx.quantize(dev(synth.weights(d_in, d_out, seed=61, key=key, outlier_frac=0.01)), None, bits=4, k_salient=128)


def test_free_and_quantize_during_a_relaxed_capture(ctx):
    """In relaxed mode a program may release and build operands while it captures launches on another stream (an object that
    the garbage collector finds is enough): the capture stays valid."""
    w, gone = weight(ctx, "stays"), weight(ctx, "goes")
    r = ctx.rotation_create(torch.eye(512, device="cuda").half())
    x = torch.randn((64, 512), device="cuda").half()
    y = torch.empty((64, 384), dtype=torch.float16, device="cuda")
    want = ctx.linear(x, w).clone()
    W = dev(synth.weights(512, 256, seed=61, key="new", outlier_frac=0.01))
    new_want = {k: v.cpu() for k, v in ctx.quantize(W, None, bits=4, k_salient=128).export().items()}
    torch.cuda.synchronize()
    graph, capture, other = torch.cuda.CUDAGraph(), torch.cuda.Stream(), torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=capture, capture_error_mode="relaxed"):
        ctx.linear(x, w, out=y)
        gone.free()
        r.free()
        new = ctx.quantize(W, None, bits=4, k_salient=128, stream=other)
        ctx.linear(x, w, out=y)
    y.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert ctx.last_status() == rb.ROSAQ_OK
    assert torch.equal(y, want)
    got = new.export()
    assert all(torch.equal(got[k].cpu(), new_want[k]) for k in new_want)


def test_free_waits_for_launches_that_read_the_operand(ctx):
    """Freeing an operand right behind launches on a stream of their own returns when they are through: what is quantized next
    may get the same memory."""
    x = torch.randn((2048, 4096), device="cuda").half()
    side = torch.cuda.Stream()
    W = [torch.randn((4096, 4096), device="cuda").half() * 0.02 for _ in range(2)]
    want = [ctx.linear(x, ctx.quantize(v, None, bits=4, k_salient=128)).clone() for v in W]
    for k in range(4):
        w = ctx.quantize(W[k % 2], None, bits=4, k_salient=128)
        torch.cuda.synchronize()
        ys = [torch.empty((2048, 4096), dtype=torch.float16, device="cuda") for _ in range(8)]
        done = torch.cuda.Event()
        with torch.cuda.stream(side):
            for y in ys:
                ctx.linear(x, w, out=y)
            done.record()
        w.free()
        assert done.query()
        ctx.quantize(W[1 - k % 2], None, bits=4, k_salient=128)
        torch.cuda.synchronize()
        assert all(torch.equal(y, want[k % 2]) for y in ys)
    assert ctx.last_status() == rb.ROSAQ_OK
