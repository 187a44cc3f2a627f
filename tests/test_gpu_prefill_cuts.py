"""The prefill tiles (implementation 5) in each way a launch can be cut: a cluster of one to four pairs of CTAs per tile,
equal shares with the exchange through L2 (two and more holders of a tile), the all-fp16 operand, several weights in one
launch; ragged token counts and widths; and the head-wise rotation written in column order and moved inside its rows.
Sampled columns against the oracle, every column against the per-call kernels (implementation 3: the same sums in another
order, one rounding to fp16: 2e-4 as elsewhere), the same bits again, also when a captured launch is replayed on other input."""
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
    (200, 1024, [384], 4),              # a cluster of several pairs per tile
    (255, 896, [1160], 3),              # ragged tokens, a last tile without a second column tile, groups that do not divide evenly
    (33, 1152, [6000], 4),              # narrow token tile, one pair per tile
    (300, 384, [512, 200, 136], 4),     # three weights, two token blocks
    (520, 1024, [11008, 1000], 3),      # equal shares
    (260, 2048, [10496], 4),            # equal shares, two holders of most tiles
    (300, 24576, [136], 4),             # equal shares, 37 holders of each tile
])
def test_prefill_cuts(ctx, M, d_in, widths, bits):
    Ws = [synth.weights(d_in, n, seed=91, key=f"cut{n}", outlier_frac=0.01) for n in widths]
    ws = [ctx.quantize(dev(W), None, bits=bits, k_salient=128) for W in Ws]
    rng = synth.rng_for(91, "x", M, d_in)
    xa, xb = (dev(rng.standard_normal((M, d_in)).astype(np.float16)) for _ in range(2))
    bufs = [torch.full((M + 1, n + 16), 7.0, dtype=torch.float16, device="cuda") for n in widths]
    outs = [b[:M, :n] for b, n in zip(bufs, widths)]
    ctx.set_linear_impl(3)
    ref = [y.clone() for y in ctx.linear_multi(xa, ws)]
    ctx.set_linear_impl(5)
    try:
        got = [y.clone() for y in ctx.linear_multi(xa, ws, outs=outs)]
        for b, n in zip(bufs, widths):
            assert torch.all(b[M:] == 7.0) and torch.all(b[:, n:] == 7.0)              # nothing written outside
        want_b = [y.clone() for y in ctx.linear_multi(xb, ws)]
        x = xa.clone()
        ys = [torch.empty((M, n), dtype=torch.float16, device="cuda") for n in widths]
        side = torch.cuda.Stream()
        graph = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.stream(side), torch.cuda.graph(graph, stream=side):
            for _ in range(2):                                                           # chained launches
                ctx.linear_multi(x, ws, outs=ys)
        for src, want in ((xa, got), (xb, want_b), (xa, got)):
            x.copy_(src)
            torch.cuda.synchronize()
            graph.replay()
            torch.cuda.synchronize()
            assert all(same(y, w) for y, w in zip(ys, want))
    finally:
        ctx.set_linear_impl(0)
    assert ctx.last_status() == rb.ROSAQ_OK
    for y, r, W, n in zip(got, ref, Ws, widths):
        assert H.rel_fro(y.cpu().numpy(), r.cpu().numpy()) <= 2e-4
        cols = synth.sample_columns(n, 24, 91, f"cut{n}")
        qd = H.oracle_quantized(W, None, None, bits, 128, cols=cols)
        assert H.rel_fro(y.cpu().numpy()[:, cols], orc.forward(xa.cpu().numpy(), qd, None)) <= H.REL_TOL_Y


@pytest.mark.parametrize("M", [5, 200, 300])
@pytest.mark.parametrize("d,heads", [(512, 1), (640, 1), (512, 4), (384, 3), (768, 2)])
def test_rotations_at_prefill_sizes(ctx, M, d, heads):
    """Dense and head-wise rotations, with and without a column order: heads of 128 channels in pairs, an odd number of them
    (not a pair's operand), heads of three groups.  Implementations 5 and 0 against the oracle; untouched columns."""
    rng = synth.rng_for(92, "rot", d, heads)
    dh = d // heads
    Rb = np.stack([synth.orthogonal_qr(dh, rng) for _ in range(heads)]).astype(np.float16)
    x = rng.standard_normal((M, d)).astype(np.float16)
    for perm in (None, rng.permutation(d).astype(np.int32)):
        rot = ctx.rotation_create(dev(Rb if heads > 1 else Rb[0]), None if perm is None else dev(perm))
        full = np.zeros((d, d))
        for h in range(heads):
            full[h * dh:(h + 1) * dh, h * dh:(h + 1) * dh] = Rb[h].astype(np.float64)
        ref = x.astype(np.float64) @ (full if perm is None else full[:, perm])
        for impl in (0, 5):
            ctx.set_linear_impl(impl)
            try:
                buf = torch.full((M, d + 8), 7.0, dtype=torch.float16, device="cuda")
                ctx.rotate(dev(x), rot, out=buf[:, :d])
                assert torch.all(buf[:, d:] == 7.0)
                assert H.rel_fro(buf[:, :d].cpu().numpy(), ref) <= 1e-3
            finally:
                ctx.set_linear_impl(0)
        rot.free()
    assert ctx.last_status() == rb.ROSAQ_OK


def test_few_tiles_of_a_long_k_stay_on_the_per_call_kernel(ctx):
    """Where a launch has one or two tiles of many groups the exchange of the pair tiles costs more than the launch on the
    per-call kernel (11.7 us against 17 to 43 at 160 tokens); the same kernel gives the same bits as implementation 3."""
    for d_in, widths in ((13824, [128]), (11008, [384]), (13824, [128, 128, 128, 128])):
        rng = synth.rng_for(93, "longk", d_in)
        ws = [ctx.quantize(dev(synth.weights(d_in, n, seed=93, key=f"longk{i}", outlier_frac=0.01)), None, bits=4, k_salient=128)
              for i, n in enumerate(widths)]
        for M in (129, 160, 300):
            x = dev(rng.standard_normal((M, d_in)).astype(np.float16))
            ctx.set_linear_impl(3)
            ref = [y.clone() for y in ctx.linear_multi(x, ws)]
            ctx.set_linear_impl(0)
            assert all(same(y, r) for y, r in zip(ctx.linear_multi(x, ws), ref))
    assert ctx.last_status() == rb.ROSAQ_OK


@pytest.mark.parametrize("d", [512, 1536])
def test_column_order_scattered_or_moved(ctx, d):
    """Either side of the sizes where the column order is no longer written by the epilogue but by a second launch: the same
    sums, so the same bits as the scattering kernel (implementation 3)."""
    rng = synth.rng_for(94, "order", d)
    q = np.stack([synth.orthogonal_qr(128, rng) for _ in range(d // 128)]).astype(np.float16)
    rot = ctx.rotation_create(dev(q), dev(rng.permutation(d).astype(np.int32)))
    for M in (16, 17, 22, 23, 54, 55, 64, 100, 128):
        x = dev(rng.standard_normal((M, d)).astype(np.float16))
        ctx.set_linear_impl(3)
        ref = ctx.rotate(x, rot).clone()
        ctx.set_linear_impl(0)
        assert same(ctx.rotate(x, rot), ref), M
    assert ctx.last_status() == rb.ROSAQ_OK


@pytest.mark.parametrize("d,M", [(512, 9), (512, 33), (512, 1184), (512, 1185), (1152, 128), (1152, 129), (4096, 64), (4096, 65), (5120, 48), (128, 40)])
def test_column_order_in_tiles_of_sixteen_tokens(ctx, d, M):
    """Up to one CTA per SM (of sixteen tokens and one head; two per SM where the heads are few) and behind it, ragged last tiles: the columns
    of the rotation without an order, moved; the rows behind the batch and the columns behind the last one stay untouched."""
    rng = synth.rng_for(95, "tiles", d, M)
    q = dev((rng.standard_normal((d // 128, 128, 128)) / 128 ** 0.5).astype(np.float16))
    perm = rng.permutation(d).astype(np.int32)
    x = dev(rng.standard_normal((M, d)).astype(np.float16))
    ctx.set_linear_impl(3)
    want = ctx.rotate(x, ctx.rotation_create(q))[:, torch.from_numpy(perm).cuda().long()]
    ctx.set_linear_impl(0)
    buf = torch.full((M + 1, d + 8), 7.0, dtype=torch.float16, device="cuda")
    rot = ctx.rotation_create(q, dev(perm))
    for _ in range(2):
        ctx.rotate(x, rot, out=buf[:M, :d])
    assert same(buf[:M, :d].contiguous(), want.contiguous())
    assert torch.all(buf[M:] == 7.0) and torch.all(buf[:, d:] == 7.0)
    assert ctx.last_status() == rb.ROSAQ_OK


@pytest.mark.parametrize("M", [257, 600, 1570, 1793])
def test_last_token_block_of_its_own_size(ctx, M):
    """Token blocks of 160 and 128, 224 and 160, 256 and 64, 256 and 32: equal shares of uneven units (64 to 128 tiles of 512 channels) and, for
    the head-wise rotation, clusters."""
    d, n = 512, 4096
    rng = synth.rng_for(97, "last", M)
    x = dev(rng.standard_normal((M, d)).astype(np.float16))
    w = ctx.quantize(dev(synth.weights(d, n, seed=97, key="last", outlier_frac=0.01)), None, bits=4, k_salient=128)
    xw = dev(rng.standard_normal((M, n)).astype(np.float16))
    dense = ctx.rotation_create(dev((rng.standard_normal((n, n)) / n ** 0.5).astype(np.float16)))
    heads = ctx.rotation_create(dev((rng.standard_normal((n // 128, 128, 128)) / 128 ** 0.5).astype(np.float16)))
    for call, args in ((ctx.linear, (x, w)), (ctx.rotate, (xw, dense)), (ctx.rotate, (xw, heads))):
        ctx.set_linear_impl(3)
        ref = call(*args).clone()
        ctx.set_linear_impl(5)
        buf = torch.full((M + 1, n + 8), 7.0, dtype=torch.float16, device="cuda")
        runs = []
        for _ in range(2):
            call(*args, out=buf[:M, :n])
            runs.append(buf[:M, :n].clone())
        ctx.set_linear_impl(0)
        assert same(runs[0], runs[1]) and torch.all(buf[M:] == 7.0) and torch.all(buf[:, n:] == 7.0)
        assert H.rel_fro(runs[0].cpu().numpy(), ref.cpu().numpy()) <= 2e-4
    assert ctx.last_status() == rb.ROSAQ_OK


@pytest.mark.parametrize("d_in,n,M", [(1408, 9000, 1300), (1280, 10672, 300), (896, 3000, 520), (384, 4768, 1782), (256, 6840, 1127)])
def test_equal_shares_without_short_ends(ctx, d_in, n, M):
    """Shares that would end with the first groups of a tile end with the tile before it, where a tile has three groups and more (here 11, 10,
    7, 3 and 2; shares of 7 to 29 groups)."""
    rng = synth.rng_for(98, "ends", d_in, M)
    x = dev(rng.standard_normal((M, d_in)).astype(np.float16))
    w = ctx.quantize(dev(synth.weights(d_in, n, seed=98, key="ends", outlier_frac=0.01)), None, bits=4, k_salient=128)
    ctx.set_linear_impl(3)
    ref = ctx.linear(x, w).clone()
    ctx.set_linear_impl(5)
    runs = [ctx.linear(x, w).clone() for _ in range(2)]
    ctx.set_linear_impl(0)
    assert ctx.last_status() == rb.ROSAQ_OK
    assert same(runs[0], runs[1])
    assert (runs[0].double() - ref.double()).norm() <= 2e-4 * ref.double().norm()
