"""One to eight tokens on the kernel of 32-column slices, at the edges of its cut: fewer units than warps, fp16 and quantized units in
one ring, a ragged last tile and slices past it, several weights, more slices than SMs, every depth of the ring of an all-fp16
operand, the head-wise rotation; and the token counts where the dispatch leaves it.  Every column against the per-call tcgen05
kernel (implementation 3: the same fp16 weights and fp32 sums in another order, one rounding to fp16: 2e-4 as elsewhere), sampled
columns against the oracle, nothing written outside, the same bits again, also from a captured chain of launches."""
import numpy as np
import pytest
import torch

from oracle import rosaq_oracle as orc
from paper_2506_13472_b200 import binding as rb
from paper_2506_13472_b200 import synth
from tests import helpers as H

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = rb.Context(0)
    yield c
    c.close()


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def same(a, b):
    return torch.equal(a.view(torch.int16), b.view(torch.int16))


@pytest.mark.parametrize("M,d_in,widths,bits", [
    (1, 128, [128], 4),                 # four fp16 units, no quantized group
    (3, 256, [200], 3),                 # five units for eight warps; a slice with eight columns and one past the last
    (8, 1152, [1000], 4),               # uneven units, every row of x' its own
    (5, 1536, [384, 72, 136], 3),       # three weights
    (2, 1024, [16384], 4),              # more slices than SMs: three CTAs of a launch on an SM
    (8, 5120, [5120], 4),               # x' leaves no room for the second CTA: the tcgen05 kernel
    (9, 512, [512], 4),                 # past its tokens
    (3, 11008, [72], 4),                # few slices, the longest K of INT4 that stays ...
    (4, 11008, [72], 4),                # ... the tcgen05 kernel
    (2, 11008, [200], 3),               # the same for INT3
    (3, 11008, [200], 3),
])
def test_linear(ctx, M, d_in, widths, bits):
    Ws = [synth.weights(d_in, n, seed=17, key=f"small{n}", outlier_frac=0.01) for n in widths]
    ws = [ctx.quantize(dev(W), None, bits=bits, k_salient=128) for W in Ws]
    rng = synth.rng_for(17, "x", M, d_in)
    xa, xb = (dev(rng.standard_normal((M, d_in)).astype(np.float16)) for _ in range(2))
    bufs = [torch.full((M + 1, (n + 23) // 8 * 8), 7.0, dtype=torch.float16, device="cuda") for n in widths]
    outs = [b[:M, :n] for b, n in zip(bufs, widths)]
    ctx.set_linear_impl(3)
    ref = [y.clone() for y in ctx.linear_multi(xa, ws)]
    ctx.set_linear_impl(0)
    got = [y.clone() for y in ctx.linear_multi(xa, ws, outs=outs)]
    for b, n in zip(bufs, widths):
        assert torch.all(b[M:] == 7.0) and torch.all(b[:, n:] == 7.0)
    want_b = [y.clone() for y in ctx.linear_multi(xb, ws)]
    x = xa.clone()
    ys = [torch.empty((M, n), dtype=torch.float16, device="cuda") for n in widths]
    side, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.stream(side), torch.cuda.graph(graph, stream=side):
        for _ in range(3):                                                               # chained launches
            ctx.linear_multi(x, ws, outs=ys)
    for src, want in ((xa, got), (xb, want_b), (xa, got)):
        x.copy_(src)
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        assert all(same(y, w) for y, w in zip(ys, want))
    assert ctx.last_status() == rb.ROSAQ_OK
    for y, r, W, n in zip(got, ref, Ws, widths):
        assert H.rel_fro(y.cpu().numpy(), r.cpu().numpy()) <= 2e-4
        cols = synth.sample_columns(n, 24, 17, f"small{n}")
        qd = H.oracle_quantized(W, None, None, bits, 128, cols=cols)
        assert H.rel_fro(y.cpu().numpy()[:, cols], orc.forward(xa.cpu().numpy(), qd, None)) <= H.REL_TOL_Y


@pytest.mark.parametrize("M,d,head", [(1, 512, False), (8, 2048, False), (3, 5120, False), (8, 5120, False), (7, 1024, True), (1, 4096, True)])
def test_rotation(ctx, M, d, head):
    rng = synth.rng_for(18, "rot", M, d)
    if head:
        q = rng.standard_normal((d // 128, 128, 128)).astype(np.float32) / 128 ** 0.5
        perm = rng.permutation(d).astype(np.int32)
        r = ctx.rotation_create(dev(q.astype(np.float16)), dev(perm))
    else:
        r = ctx.rotation_create(dev((rng.standard_normal((d, d)) / d ** 0.5).astype(np.float16)))
    x = dev(rng.standard_normal((M, d)).astype(np.float16))
    ctx.set_linear_impl(3)
    ref = ctx.rotate(x, r).clone()
    ctx.set_linear_impl(0)
    got = ctx.rotate(x, r)
    assert same(got, ctx.rotate(x, r))
    assert H.rel_fro(got.cpu().numpy(), ref.cpu().numpy()) <= 2e-4
    # rotation and linear in one call: the chain of the two launches gives what the two calls give
    w = ctx.quantize(dev(synth.weights(d, 384, seed=19, key="chain", outlier_frac=0.01)), None, bits=4, k_salient=128)
    assert same(ctx.linear(x, w, rotation=r), ctx.linear(got, w))
    assert ctx.last_status() == rb.ROSAQ_OK


@pytest.mark.parametrize("kind,d,widths,bits", [
    ("dense", 128, [128], 4),              # eight CTAs
    ("dense", 512, [200], 4),              # a slice with eight columns, one past the last
    ("heads", 384, [72, 384, 1000], 3),
    ("dense", 2048, [2688], 3),            # 148 CTAs, the most on 148 SMs; one tile more below
    ("dense", 2048, [2696], 4),
    ("heads", 2304, [136], 4),             # seven tokens are the most with one launch
])
def test_rotation_and_linears_in_one_launch(ctx, kind, d, widths, bits):
    """A small rotated call is one launch (unless it is captured): the bits of the rotation and the linears called one by one, with
    other calls in between, with values that are no numbers, and behind a call that gave up."""
    rng = synth.rng_for(21, "onelaunch", d)
    if kind == "dense":
        r = ctx.rotation_create(dev((rng.standard_normal((d, d)) / d ** 0.5).astype(np.float16)))
    else:
        r = ctx.rotation_create(dev((rng.standard_normal((d // 128, 128, 128)) / 128 ** 0.5).astype(np.float16)))
    ws = [ctx.quantize(dev(synth.weights(d, n, 21, f"onelaunch{i}", outlier_frac=0.01)), None, bits=bits, k_salient=128) for i, n in enumerate(widths)]
    for M in (1, 3, 8, 2, 8):
        x = dev(rng.standard_normal((M, d)).astype(np.float16))
        if M == 2:
            x[0, 5], x[1, 7] = float("inf"), float("nan")
        xr = ctx.rotate(x, r)
        want = ctx.linear_multi(xr, ws)
        if M == 3:
            old = ctx.set_wait_limit(1)
            ctx.linear_multi(x, ws, r)
            ctx.set_wait_limit(old)
            status = ctx.last_status()                     # (the smallest may be done before the second poll)
            assert status == rb.ROSAQ_ERR_TIMEOUT or (status == rb.ROSAQ_OK and widths != [2688])
        for _ in range(3):
            assert all(same(y, v) for y, v in zip(ctx.linear_multi(x, ws, r), want))
            assert same(ctx.linear(x, ws[0], r), want[0])
        y, graph, side = torch.empty_like(want[0]), torch.cuda.CUDAGraph(), torch.cuda.Stream()
        torch.cuda.synchronize()
        with torch.cuda.stream(side), torch.cuda.graph(graph, stream=side):
            ctx.linear(x, ws[0], r, out=y)
        graph.replay()
        torch.cuda.synchronize()
        assert same(y, want[0]) and same(ctx.linear(x, ws[0], r), want[0])
    assert ctx.last_status() == rb.ROSAQ_OK


@pytest.mark.parametrize("M,d_in,widths,bits", [
    (1, 4736, [4736], 4),               # 40 units: eight warps, the most slices with an SM each ...
    (1, 4864, [4472, 136], 4),          # ... 41: sixteen, the last round nearly empty; the most slices, a ragged tile, two weights
    (1, 4864, [4600, 136], 4),          # one tile more: eight
    (1, 4864, [4744], 4),
    (2, 4096, [328], 3),                # 35 and
    (7, 4224, [328], 3),                # 36 units of INT3
    (5, 13824, [2048], 4),              # x' of the most tokens next to the rings of sixteen warps,
    (8, 11008, [4096], 3),              # of one token more than that: eight
    (8, 6144, [4096], 4),
])
def test_long_k_on_sixteen_warps(ctx, M, d_in, widths, bits):
    """The line between eight and sixteen warps per slice, and a rotated call on either side of it, which is one launch on the near one:
    the bits of two calls."""
    test_linear(ctx, M, d_in, widths, bits)
    rng = synth.rng_for(23, "sixteen", d_in)
    r = ctx.rotation_create(dev((rng.standard_normal((d_in // 128, 128, 128)) / 128 ** 0.5).astype(np.float16)))
    w = ctx.quantize(dev(synth.weights(d_in, 72, 23, "sixteen", outlier_frac=0.01)), None, bits=bits, k_salient=128)
    x = dev(rng.standard_normal((2, d_in)).astype(np.float16))
    assert same(ctx.linear(x, w, rotation=r), ctx.linear(ctx.rotate(x, r), w))
    assert ctx.last_status() == rb.ROSAQ_OK
