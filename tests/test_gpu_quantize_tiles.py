"""rosaq_quantize at the edges of its 128 x 128 tiles, bit for bit against the oracle: head blocks that are no
multiple of a tile, a column order next to a dense R, fp16 rotations, scaled weights, widths that leave a partial tile
or no aligned row, and a weight wide enough for several slabs of the head-wise path."""
import numpy as np
import pytest
import torch

from oracle import rosaq_oracle as orc
from paper_2506_13472_b200 import binding as rb
from paper_2506_13472_b200 import synth
from tests import helpers as H

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("heads,dh,d_out,perm,half,scaled,bits", [
    (1, 512, 200, True, False, False, 4),      # dense R with a column order: a tile gathers its columns of R
    (1, 256, 129, False, True, True, 3),       # fp16 R, scaled, odd width: no aligned rows
    (4, 96, 136, False, False, False, 3),      # head blocks narrower than a tile
    (2, 192, 264, True, False, True, 4),       # ... and 1.5 tiles, with a column order and a scale
    (4, 128, 128, False, True, False, 4),      # head blocks of one tile, fp16 R, in place
    (4, 128, 8328, True, False, False, 3),     # two slabs of W'
])
def test_quantize_tile_edges_bit_exact(heads, dh, d_out, perm, half, scaled, bits):
    d = heads * dh
    rng = synth.rng_for(81, "tiles", heads, dh, d_out)
    Rb = np.stack([synth.orthogonal_qr(dh, rng) for _ in range(heads)]).astype(np.float16 if half else np.float32)
    p = rng.permutation(d).astype(np.int32) if perm else None
    W = synth.weights(d, d_out, seed=81, key=f"tiles{d}x{d_out}", outlier_frac=0.01)
    scale = (0.5 + rng.random(d)).astype(np.float32) if scaled else None
    cols = np.asarray(sorted({0, d_out - 1, min(127, d_out - 1), min(128, d_out - 1)} | set(rng.integers(0, d_out, 60).tolist())), np.int32)
    Wf = W if scale is None else orc.scale_rows_f32(W, scale)
    Wp = orc.rotate_weights_f32(Rb.astype(np.float32) if heads > 1 or perm else Rb[0].astype(np.float32), Wf, p, cols)
    qd = orc.quantize(Wp, bits, 128, 128)
    qd["qw"], qd["cols"] = orc.pack(qd["codes"], bits), cols
    ctx = rb.Context(0)
    try:
        for _ in range(2):                      # the second one gets the memory of the first
            w = ctx.quantize(dev(W), dev(Rb if heads > 1 else Rb[0]), None if p is None else dev(p), bits=bits, k_salient=128,
                             in_scale=None if scale is None else dev(scale))
            H.assert_export_matches(H.export_to_numpy(w.export()), qd)
            w.free()
        assert ctx.last_status() == rb.ROSAQ_OK
    finally:
        ctx.close()


@pytest.mark.parametrize("heads,half,off", [(1, False, 1), (1, False, 2), (1, True, 1), (1, True, 3), (2, False, 3), (2, True, 2)])
def test_rotation_on_any_element(heads, half, off):
    """R at an address that is no multiple of four elements (a view into a larger buffer)."""
    dh, d_out = 256 // heads, 136
    rng = synth.rng_for(82, "offset", heads, half)
    Rb = np.stack([synth.orthogonal_qr(dh, rng) for _ in range(heads)]).astype(np.float16 if half else np.float32)
    W = synth.weights(256, d_out, seed=82, key="offset", outlier_frac=0.01)
    q = dev(np.concatenate([np.zeros(off, Rb.dtype), Rb.ravel()]))[off:].view(heads, dh, dh)
    assert q.data_ptr() % (8 if half else 16)
    qd = H.oracle_quantized(W, Rb.astype(np.float32) if heads > 1 else Rb[0].astype(np.float32), None, 4, 128)
    ctx = rb.Context(0)
    try:
        w = ctx.quantize(dev(W), q if heads > 1 else q[0], None, bits=4, k_salient=128)
        H.assert_export_matches(H.export_to_numpy(w.export()), qd)
        assert ctx.last_status() == rb.ROSAQ_OK
    finally:
        ctx.close()


@pytest.mark.parametrize("bits", [3, 4])
def test_nan_inside_a_group(bits):
    """NaNs behind the first row of a group are no extremes: scale, zero-point and the other rows' codes as in one scan down
    the column, wherever the threads of a column start.  (A NaN has no code; the kernel stores 0.)"""
    d, d_out = 384, 140
    W = synth.weights(d, d_out, seed=83, key="nan", outlier_frac=0.01)
    for n, row in enumerate((1, 31, 32, 33, 64, 65, 95, 96, 127)):
        W[128 + row, n] = np.nan
        W[256 + row, 130 + n] = np.nan
    W[128 + 32:128 + 64, 20] = np.nan
    W[256 + 1:384, 21] = np.nan
    qd = orc.quantize(W.astype(np.float32), bits, 128, 128)
    codes = np.where(np.isnan(W[128:].astype(np.float32)), 0, qd["codes"]).astype(np.uint8)
    qd["qw"], qd["cols"] = orc.pack(codes, bits), np.arange(d_out)
    ctx = rb.Context(0)
    try:
        H.assert_export_matches(H.export_to_numpy(ctx.quantize(dev(W), None, bits=bits, k_salient=128).export()), qd)
    finally:
        ctx.close()


def test_more_head_blocks_than_a_grid_dimension_holds():
    """70016 head blocks of one channel: R is a diagonal of signs, so W' is W with the signs, in a column order."""
    d, d_out = 70016, 8
    rng = synth.rng_for(84, "blocks", d)
    sign = rng.choice(np.asarray([-1.0, 1.0], np.float32), d)
    p = rng.permutation(d).astype(np.int32)
    W = synth.weights(d, d_out, seed=84, key="blocks", outlier_frac=0.01)
    qd = orc.quantize((W.astype(np.float32) * sign[:, None])[p], 4, 128, 128)
    qd["qw"], qd["cols"] = orc.pack(qd["codes"], 4), np.arange(d_out)
    ctx = rb.Context(0)
    try:
        w = ctx.quantize(dev(W), dev(sign.reshape(d, 1, 1)), dev(p), bits=4, k_salient=128)
        H.assert_export_matches(H.export_to_numpy(w.export()), qd)
    finally:
        ctx.close()
