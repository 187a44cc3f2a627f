"""rosaq_calib_cov where few tiles make a cluster of CTAs share each tile's tokens: every split count of the three kernels
(pairs, single CTAs, fp32), ragged tokens and widths, two accumulated calls, the same bits on a second run."""
import numpy as np
import pytest
import torch

from oracle import rosaq_oracle as orc
from paper_2506_13472_b200 import binding as rb
from paper_2506_13472_b200 import synth
from tests import helpers as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,n_tokens,d,n_blocks", [
    (np.float16, 2100, 512, 1),       # single CTAs, 8 splits
    (np.float16, 1030, 768, 1),       # 4 splits (tokens), columns past the last whole tile
    (np.float16, 1500, 1032, 1),      # pairs, 4 splits, d no multiple of 64
    (np.float16, 600, 1288, 1),       # pairs, 2 splits
    (np.float16, 2049, 640, 5),       # head blocks of 128, 8 splits
    (np.float16, 515, 1024, 2),       # two blocks of 512
    (np.float32, 1001, 256, 1),       # fp32, 8 splits, mirrored shares
    (np.float32, 300, 384, 3),        # 4 splits
    (np.float16, 700, 96, 2),         # narrow blocks on the fp32 kernel
    (np.float16, 300, 704, 8),        # head blocks that start inside a block of 64 channels: 88 channels,
    (np.float16, 90, 576, 4),         # 144 (two row tiles),
    (np.float16, 200, 4160, 8),       # 520 (pairs)
    (np.float32, 70, 136, 1),         # one split
    (np.float32, 515, 2048, 1)])      # 136 tiles in two: steps of eight, mirrored shares
def test_calib_cov_splits(dtype, n_tokens, d, n_blocks):
    X = synth.ActivationLaw(d, 1.0, seed=47, key=f"covs{d}").sample(n_tokens, "X", dtype)
    dh, half = d // n_blocks, n_tokens // 2 // 8 * 8
    Xd = torch.from_numpy(X).cuda()
    ctx = rb.Context(0)
    try:
        runs = []
        for _ in range(2):
            Cg = torch.zeros((n_blocks, dh, dh), dtype=torch.float32, device="cuda")
            ctx.calib_cov(Xd, Cg, n_blocks)
            ctx.calib_cov(Xd[half:], Cg, n_blocks)
            runs.append(Cg.cpu().numpy())
        assert ctx.last_status() == rb.ROSAQ_OK
    finally:
        ctx.close()
    assert np.array_equal(runs[0].view(np.uint32), runs[1].view(np.uint32))
    Cref = orc.cov(X, n_blocks).reshape(n_blocks, dh, dh) + orc.cov(X[half:], n_blocks).reshape(n_blocks, dh, dh)
    got = runs[0].astype(np.float64)
    assert np.all(np.abs(got - Cref) <= H.cov_tolerance(Cref, n_tokens) + 1e-30)
    assert np.array_equal(got, np.swapaxes(got, -1, -2))


def test_calib_cov_reads_what_the_launch_before_wrote():
    """The fp32 kernel is chained to the launch before it, which may still be writing its input when it starts: rotation and
    Gram matrix of narrow blocks from a captured chain, the same bits as with a synchronization in between."""
    M, d, nb = 600, 256, 8
    ctx = rb.Context(0)
    try:
        rng = synth.rng_for(48, "chain")
        rot = ctx.rotation_create(torch.from_numpy(synth.orthogonal_qr(d, rng).astype(np.float16)).cuda(),
                                  torch.from_numpy(rng.permutation(d).astype(np.int32)).cuda())
        xs = [torch.from_numpy(rng.standard_normal((M, d)).astype(np.float16)).cuda() for _ in range(4)]
        xr, Cg = torch.empty((M, d), dtype=torch.float16, device="cuda"), torch.zeros((nb, d // nb, d // nb), device="cuda")
        want = []
        for x in xs:
            ctx.rotate(x, rot, out=xr)
            torch.cuda.synchronize()
            ctx.calib_cov(xr, Cg, nb)
            want.append(Cg.clone())
        x, out = xs[0].clone(), [torch.empty_like(Cg) for _ in xs]
        side, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.stream(side), torch.cuda.graph(graph, stream=side):
            for src, o in zip(xs, out):
                x.copy_(src)
                ctx.rotate(x, rot, out=xr)
                ctx.calib_cov(xr, Cg, nb)
                o.copy_(Cg)
        for _ in range(3):
            xr.fill_(float("nan"))
            Cg.zero_()
            graph.replay()
            torch.cuda.synchronize()
            assert all(torch.equal(o, w) for o, w in zip(out, want))
        assert ctx.last_status() == rb.ROSAQ_OK
    finally:
        ctx.close()


def test_a_long_calib_cov_does_not_use_up_the_waits_of_the_launch_behind_it():
    """Eight CTAs that take 10 ms leave the other SMs to the launch behind them, whose waits last a few hundred microseconds:
    it must not start counting before the Gram matrix is nearly complete."""
    ctx = rb.Context(0)
    try:
        X = torch.ones((1 << 20, 64), device="cuda")
        Cg = torch.zeros((64, 64), device="cuda")
        W = synth.weights(1024, 512, seed=49, key="behind", outlier_frac=0.01)
        w = ctx.quantize(torch.from_numpy(W).cuda(), None, bits=4, k_salient=128)
        x = torch.randn((64, 1024), device="cuda").half()
        y = torch.empty((64, 512), dtype=torch.float16, device="cuda")
        want = ctx.linear(x, w).clone()
        plan = ctx.plan_create(64, [(x, None, w, y)])
        ctx.calib_cov(X[:64], Cg)
        old = ctx.set_wait_limit(300)
        try:
            for run in (lambda: ctx.linear(x, w, out=y), plan.run):
                Cg.zero_()
                y.zero_()
                torch.cuda.synchronize()
                ctx.calib_cov(X, Cg)
                run()
                assert ctx.last_status() == rb.ROSAQ_OK
                assert torch.all(Cg == 1 << 20) and (y - want).norm() <= 2e-4 * want.norm()
        finally:
            ctx.set_wait_limit(old)
    finally:
        ctx.close()


@pytest.mark.parametrize("n_tokens,n_blocks", [(509, 14), (509, 15), (7, 1), (17, 2), (515, 14), (519, 15)])
def test_calib_cov_either_step_of_the_fp32_kernel(n_tokens, n_blocks):
    """The fp32 kernel steps through sixteen tokens at a time where an SM has one CTA (up to 118 of them on 148 SMs), else through eight:
    both sides of the line (515 and 519 tokens in eight parts: 112 and 120 CTAs; 509 only in four), tokens that fill no whole step, one
    step, less than one."""
    d = 128 * n_blocks
    X = synth.ActivationLaw(d, 1.0, seed=49, key=f"covk{d}").sample(n_tokens, "X", np.float32)
    ctx = rb.Context(0)
    try:
        Cg = torch.zeros((n_blocks, 128, 128), dtype=torch.float32, device="cuda")
        ctx.calib_cov(torch.from_numpy(X).cuda(), Cg, n_blocks)
        assert ctx.last_status() == rb.ROSAQ_OK
    finally:
        ctx.close()
    Cref = orc.cov(X, n_blocks).reshape(n_blocks, 128, 128)
    got = Cg.cpu().numpy().astype(np.float64)
    assert np.all(np.abs(got - Cref) <= H.cov_tolerance(Cref, n_tokens) + 1e-30)
    assert np.array_equal(got, np.swapaxes(got, -1, -2))


@pytest.mark.parametrize("n_tokens,d,n_blocks", [(130, 3000, 1), (64, 3072, 1), (200, 4608, 2), (1, 4104, 1), (1919, 3000, 1), (1921, 3000, 1)])
def test_calib_cov_more_tiles_than_pairs(n_tokens, d, n_blocks):
    """78 to 153 tiles for the 74 pairs of 148 SMs: pairs that take a second and a third tile while the first is added to C (78 tiles: from 961
    tokens, both calls of the last case, on).  A C that does
    not lie on 32 bytes takes the kernel with a pair per tile, whose bits it has to give; tokens and channels that fill no whole tile."""
    dh = d // n_blocks
    X = (torch.randn((n_tokens, d), generator=torch.Generator().manual_seed(51)) * torch.linspace(2, 0.1, d)).half().cuda()
    ctx = rb.Context(0)
    try:
        got = []
        for off in (0, 4):
            C = torch.empty(n_blocks * dh * dh + 8, device="cuda")[off:off + n_blocks * dh * dh].view(n_blocks, dh, dh)
            assert C.data_ptr() % 32 == 4 * off
            C.fill_(0.5)
            ctx.calib_cov(X, C, n_blocks)
            ctx.calib_cov(X[:n_tokens // 2 + 1], C, n_blocks)
            got.append(C)
        assert ctx.last_status() == rb.ROSAQ_OK
    finally:
        ctx.close()
    assert torch.equal(got[0], got[1]) and torch.equal(got[0], got[0].transpose(1, 2))
    Xd = X.double().view(n_tokens, n_blocks, dh).transpose(0, 1)
    Xh = Xd[:, :n_tokens // 2 + 1]
    want = Xd.transpose(1, 2) @ Xd + Xh.transpose(1, 2) @ Xh
    diag = want.diagonal(dim1=1, dim2=2)
    bound = (n_tokens / 16 + 12) * 2.0 ** -23 * (diag[:, :, None] * diag[:, None, :]).sqrt() + 1e-6   # (0.5 and two sums rounded)
    assert torch.all((got[0].double() - 0.5 - want).abs() <= bound)


@pytest.mark.parametrize("d", [768, 2048, 3328])
def test_calib_cov_behind_one_that_gave_up(d):
    """A Gram matrix that gives up (its epilogue waits for hundreds of microseconds, with a limit of one poll), on single CTAs, on a
    pair per tile and on pairs that take tiles in turn, where one CTA may give up long before the other.  The status says so, both leave, and the next call gives the bits of the first."""
    X = (torch.randn((32768, d), generator=torch.Generator().manual_seed(53)) * 0.5).half().cuda()
    ctx = rb.Context(0)
    try:
        def gram(x):
            C = torch.zeros((d, d), device="cuda")
            ctx.calib_cov(x, C)
            return C

        want = gram(X[:1000])
        assert ctx.last_status() == rb.ROSAQ_OK
        for _ in range(3):
            old = ctx.set_wait_limit(1)
            try:
                gram(X)
            finally:
                ctx.set_wait_limit(old)
            assert ctx.last_status() == rb.ROSAQ_ERR_TIMEOUT
            assert torch.equal(gram(X[:1000]), want)
            assert ctx.last_status() == rb.ROSAQ_OK
    finally:
        ctx.close()


def test_calib_cov_of_values_that_are_no_numbers():
    """A NaN and an infinity in one channel each, on the pairs that take tiles in turn (91 tiles): their rows and columns of C hold nothing
    finite, everything else has the bits that it has without them."""
    n_tokens, d = 200, 3328
    X = torch.randn((n_tokens, d), generator=torch.Generator().manual_seed(54)).half().cuda()
    X[5, 100], X[150, 3000] = 0, 0
    ctx = rb.Context(0)
    try:
        want = torch.zeros((d, d), device="cuda")
        ctx.calib_cov(X, want)
        X[5, 100], X[150, 3000] = float("nan"), float("inf")
        C = torch.zeros((d, d), device="cuda")
        ctx.calib_cov(X, C)
        assert ctx.last_status() == rb.ROSAQ_OK
    finally:
        ctx.close()
    keep = torch.ones(d, dtype=torch.bool, device="cuda")
    keep[100] = keep[3000] = False
    assert torch.equal(C[keep][:, keep], want[keep][:, keep])
    assert torch.all(torch.isnan(C[100])) and torch.all(torch.isnan(C[:, 100]))
    assert not torch.any(torch.isfinite(C[3000])) and not torch.any(torch.isfinite(C[:, 3000]))
