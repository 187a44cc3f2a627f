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


def test_captured_launches_outlive_the_workspace_they_used(ctx):
    """A workspace grows when a later call or plan needs more.  Launches captured before -- a linear whose rotated activations
    lie in it, pair tiles and a plan whose partial tiles do -- replay on the one they were captured with."""
    d = 1024
    rot = ctx.rotation_create((torch.randn((d, d), device="cuda") / d ** 0.5).half())
    w, wide = weight(ctx, "ws", d, d), weight(ctx, "wsw", d, 11008)
    x, xp = torch.randn((64, d), device="cuda").half(), torch.randn((520, d), device="cuda").half()
    y, yp, xr, yl = (torch.empty(s, dtype=torch.float16, device="cuda") for s in ((64, d), (520, 11008), (64, d), (64, d)))
    plan = ctx.plan_create(64, [(x, None, rot, xr), (None, 0, w, yl)])

    def launches():
        ctx.linear(x, w, rot, out=y)
        ctx.linear(xp, wide, out=yp)
        plan.run()

    launches()
    want = [t.clone() for t in (y, yp, yl)]
    graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(side), torch.cuda.graph(graph, stream=side):
        launches()
    big = torch.randn((6000, d), device="cuda").half()
    for m in (2100, 3000, 6000):                                     # 4.3, 6.1, 12.3 MB of rotated activations
        ctx.linear(big[:m], w, rot)
    # twelve operations one after the other, each with partial tiles in every CTA: more of them than the context starts with
    # (768 of 64 KB on 148 SMs)
    xl = torch.randn((128, d), device="cuda").half()
    outs = [torch.empty((128, d), dtype=torch.float16, device="cuda") for _ in range(12)]
    ctx.plan_create(128, [(xl if k == 0 else None, None if k == 0 else k - 1, w, o) for k, o in enumerate(outs)]).run()
    filler = [torch.full((1 << 22,), float("nan"), device="cuda") for _ in range(8)]
    for _ in range(2):
        for t in (y, yp, yl):
            t.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip((y, yp, yl), want))
    assert ctx.last_status() == rb.ROSAQ_OK
    del filler
