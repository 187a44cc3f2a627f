"""Performance cases: what a user of librosaq has it do, through the public binding.

Five kinds of work, at LLaMA-7B and LLaMA-13B shapes (the ones of `synth.LLAMA_7B` / `LLAMA_13B`), at the tiny
shape the tests start from, and over the sizes between:

  linear     one rotated linear y = (x R) W': a projection called on its own
  layer      the linears of a decoder layer as separate calls, the way a model with attention and an activation
             function between them issues them: rotation + q/k/v, rotation + o, rotation + gate/up, down.  Few
             tokens are decoding, hundreds to thousands are a prompt
  plan       the same ten operations as one rosaq_plan launch (decode batches)
  calibrate  one chunk of the calibration stream: C += X^T X
  quantize   rotate, quantize and pack linears of a layer and export them, as when a checkpoint is written

Activations and weights follow the laws of `synth` (power-law spectrum mixed by Householder reflections, Gaussian
weights with amplified input channels), drawn on the GPU from the seed; rotations are the exact eigenvectors of
those laws, per-head ones with the column order by eigenvalue.
"""
import math

import torch

from paper_2506_13472_b200 import binding, synth

GROUP = 128          # quantization group, the only one the library takes
SALIENT = 128        # fp16 channels
HEAD = 128           # head dimension of both model shapes

_ctx = None


def _context():
    """One context per process, as a program that serves a model keeps it."""
    global _ctx
    if _ctx is None:
        _ctx = binding.Context(0)
    return _ctx


# ---------------------------------------------------------------------------------------------- the cases
def listed():
    d7, f7 = synth.LLAMA_7B["d"], synth.LLAMA_7B["ffn"]
    d13, f13 = synth.LLAMA_13B["d"], synth.LLAMA_13B["ffn"]
    return [
        # the smallest call: latency of one rotated linear of the tiny configuration
        dict(name="linear_tiny_m4", kind="linear", d_in=512, d_out=512, m=4, bits=4, rotation="dense"),
        # one linear over a ragged batch, un-rotated input, a width that is no multiple of a column tile
        dict(name="linear_ragged_m77_int3", kind="linear", d_in=2944, d_out=5000, m=77, bits=3, rotation="none"),
        # one user generating text: every weight is read for one token
        dict(name="layer_7b_m1", kind="layer", d=d7, f=f7, m=1, bits=4),
        # a decode batch on the larger model
        dict(name="layer_13b_m64", kind="layer", d=d13, f=f13, m=64, bits=4),
        # decode batches as one launch per layer: the headline configuration, and INT3 at a smaller batch
        dict(name="plan_7b_m64", kind="plan", d=d7, f=f7, m=64, bits=4),
        dict(name="plan_7b_m16_int3", kind="plan", d=d7, f=f7, m=16, bits=3),
        # a short prompt (or a mixed batch), a prompt chunk, a long prompt
        dict(name="layer_7b_m200_int3", kind="layer", d=d7, f=f7, m=200, bits=3),
        dict(name="layer_13b_m512", kind="layer", d=d13, f=f13, m=512, bits=4),
        dict(name="layer_7b_m1900", kind="layer", d=d7, f=f7, m=1900, bits=4),
        # calibration: a chunk of the 13B stream, and the per-head Gram matrices of the o_proj input
        dict(name="calibrate_13b_16384", kind="calibrate", tokens=16384, d=d13, blocks=1, fp32=False),
        dict(name="calibrate_heads_4096", kind="calibrate", tokens=4096, d=d7, blocks=d7 // HEAD, fp32=False),
        # offline: one linear of each kind (dense R; per-head R with its column order; scaled, un-rotated)
        dict(name="quantize_7b_q_o_down", kind="quantize", d=d7, f=f7, bits=4, linears="q,o,down"),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _mult(v, step):
    return max(step, int(round(v / step)) * step)


# a drawn layer costs no more than the listed prompt of 1900 tokens
_LAYER_LIMIT = 1900 * (6 * synth.LLAMA_7B["d"] ** 2 + 3 * synth.LLAMA_7B["d"] * synth.LLAMA_7B["ffn"])


def draw(rng):
    kind = rng.choice(["linear", "linear", "layer", "layer", "plan", "plan", "calibrate", "calibrate", "quantize"])
    bits = rng.choice([4, 4, 3])
    if kind == "linear":
        d_in = _mult(_log_uniform(rng, 256, 13824), GROUP)
        return dict(kind=kind, d_in=d_in, d_out=_mult(_log_uniform(rng, 128, 13824), 8), m=_log_uniform(rng, 1, 1900), bits=bits,
                    rotation=rng.choice(["none", "dense", "heads"]) if d_in <= 5120 else "none")
    if kind == "quantize":
        d = _mult(_log_uniform(rng, 512, 4096), HEAD)
        return dict(kind=kind, d=d, f=_mult(d * rng.uniform(2.0, 2.7), GROUP), bits=bits,
                    linears=rng.choice(["q", "o", "down", "q,o,down"]))
    if kind == "calibrate":
        if rng.random() < 0.3:                              # fp32 activations, as the tiny configuration has them
            d = _mult(_log_uniform(rng, 256, 2048), HEAD)
            return dict(kind=kind, tokens=_log_uniform(rng, 200, 4096), d=d, blocks=rng.choice([1, d // HEAD]), fp32=True)
        d = _mult(_log_uniform(rng, 512, 5120), HEAD)
        return dict(kind=kind, tokens=_log_uniform(rng, 500, 16384), d=d, blocks=rng.choice([1, 1, d // HEAD]), fp32=False)
    d = _mult(_log_uniform(rng, 512, 5120), HEAD)
    f = _mult(d * rng.uniform(2.0, 2.75), GROUP)
    if kind == "plan":
        return dict(kind=kind, d=d, f=f, m=_log_uniform(rng, 1, 128), bits=bits)
    most = min(2048, _LAYER_LIMIT // (6 * d * d + 3 * d * f))
    return dict(kind=kind, d=d, f=f, m=_log_uniform(rng, 1, most), bits=bits)


# ---------------------------------------------------------------------------------------------- inputs
class _Draw:
    """Seeded draws on the GPU."""

    def __init__(self, seed):
        self.g = torch.Generator(device="cuda").manual_seed(int(seed))

    def normal(self, *shape):
        return torch.randn(shape, device="cuda", generator=self.g)

    def law(self, d, exponent):
        """(square roots of the spectrum, reflection vectors) of a power-law covariance."""
        lam = torch.arange(1, d + 1, device="cuda", dtype=torch.float32).pow(-exponent)
        v = self.normal(8, d)
        return lam.sqrt(), v / v.norm(dim=1, keepdim=True)

    def weight(self, d_in, d_out):
        """fp16 [d_in][d_out], N(0, 0.02^2), one input channel in a hundred ten times larger."""
        w = self.normal(d_in, d_out) * 0.02
        rows = torch.randperm(d_in, device="cuda", generator=self.g)[: max(1, d_in // 100)]
        w[rows] *= 10.0
        return w.half()


def _reflect(z, vs):
    for v in vs:
        z = z - 2.0 * torch.outer(z @ v, v)
    return z


def _dense_input(dr, m, d, dtype=torch.float16):
    """(x [m][d], R fp32 [d][d]): activations of a power-law spectrum and their principal directions."""
    s, vs = dr.law(d, 1.0)
    x = _reflect(dr.normal(m, d) * s, vs).to(dtype)
    return x, _reflect(torch.eye(d, device="cuda"), vs).T.contiguous()


def _heads_input(dr, m, d, dtype=torch.float16):
    """(x, R fp32 [heads][128][128], perm): an exponent per head, columns of all heads by falling eigenvalue."""
    heads = d // HEAD
    expo = torch.rand(heads, device="cuda", generator=dr.g) * 0.7 + 0.8
    lam = torch.arange(1, HEAD + 1, device="cuda", dtype=torch.float32)[None, :].pow(-expo[:, None])
    q = torch.linalg.qr(dr.normal(heads, HEAD, HEAD))[0]
    z = dr.normal(heads, m, HEAD) * lam.sqrt()[:, None, :]
    x = torch.bmm(z, q.transpose(1, 2)).permute(1, 0, 2).reshape(m, d).to(dtype).contiguous()
    perm = torch.argsort(lam.reshape(-1), descending=True, stable=True).to(torch.int32)
    return x, q.contiguous(), perm


def _scaled_input(dr, m, d):
    """(x D^-1, D): the un-rotated down projection's input; D by the rule of `pca.channel_scale`."""
    s, vs = dr.law(d, 1.0)
    mean = _reflect(dr.normal(512, d) * s, vs).abs().mean(dim=0)
    scale = mean.sqrt()
    scale = (scale / (scale.max() * scale.min()).sqrt()).contiguous()
    return (_reflect(dr.normal(m, d) * s, vs) / scale).half(), scale


def _layer_state(c, dr):
    ctx, d, f, m, bits = _context(), c["d"], c["f"], c["m"], c["bits"]
    st = dict(ctx=ctx)
    st["x_attn"], r_attn = _dense_input(dr, m, d)
    st["x_o"], r_o, perm = _heads_input(dr, m, d)
    st["x_mlp"], r_mlp = _dense_input(dr, m, d)
    st["x_down"], scale = _scaled_input(dr, m, f)
    st["r_attn"], st["r_mlp"] = ctx.rotation_create(r_attn.half()), ctx.rotation_create(r_mlp.half())
    st["r_o"] = ctx.rotation_create(r_o.half(), perm)
    for n in ("q", "k", "v"):
        st[n] = ctx.quantize(dr.weight(d, d), r_attn, bits=bits, k_salient=SALIENT)
    st["o"] = ctx.quantize(dr.weight(d, d), r_o, perm, bits=bits, k_salient=SALIENT)
    for n in ("gate", "up"):
        st[n] = ctx.quantize(dr.weight(d, f), r_mlp, bits=bits, k_salient=SALIENT)
    st["down"] = ctx.quantize(dr.weight(f, d), None, bits=bits, k_salient=SALIENT, in_scale=scale)
    return st


def prepare(case, seed):
    c, dr = case, _Draw(seed)
    ctx = _context()
    if c["kind"] == "linear":
        d, rot, perm = c["d_in"], None, None
        if c["rotation"] == "dense":
            x, rot = _dense_input(dr, c["m"], d)
        elif c["rotation"] == "heads":
            x, rot, perm = _heads_input(dr, c["m"], d)
        else:
            x, _ = _scaled_input(dr, c["m"], d)
        w = ctx.quantize(dr.weight(d, c["d_out"]), rot, perm, bits=c["bits"], k_salient=SALIENT)
        return dict(kind=c["kind"], ctx=ctx, x=x, w=w, r=None if rot is None else ctx.rotation_create(rot.half(), perm))
    if c["kind"] == "layer":
        return dict(_layer_state(c, dr), kind=c["kind"])
    if c["kind"] == "plan":
        st = dict(_layer_state(c, dr), kind=c["kind"])
        m, d, f = c["m"], c["d"], c["f"]
        out = lambda n: torch.empty((m, n), dtype=torch.float16, device="cuda")  # noqa: E731
        xr = [out(d) for _ in range(3)]
        st["y"] = {n: out(f if n in ("gate", "up") else d) for n in ("q", "k", "v", "o", "gate", "up", "down")}
        y = st["y"]
        st["plan"] = ctx.plan_create(m, [
            (st["x_attn"], None, st["r_attn"], xr[0]), (st["x_mlp"], None, st["r_mlp"], xr[1]), (st["x_o"], None, st["r_o"], xr[2]),
            (st["x_down"], None, st["down"], y["down"]),
            (None, 0, st["q"], y["q"]), (None, 0, st["k"], y["k"]), (None, 0, st["v"], y["v"]), (None, 2, st["o"], y["o"]),
            (None, 1, st["gate"], y["gate"]), (None, 1, st["up"], y["up"])])
        return st
    if c["kind"] == "calibrate":
        d, nb = c["d"], c["blocks"]
        dtype = torch.float32 if c["fp32"] else torch.float16
        x = _dense_input(dr, c["tokens"], d, dtype)[0] if nb == 1 else _heads_input(dr, c["tokens"], d, dtype)[0]
        return dict(kind=c["kind"], ctx=ctx, x=x, blocks=nb, gram=torch.zeros((nb, d // nb, d // nb), device="cuda"))
    st, d, f = dict(kind=c["kind"], ctx=ctx, todo=[]), c["d"], c["f"]
    for n in c["linears"].split(","):
        job = dict(bits=c["bits"], k_salient=SALIENT)
        if n == "q":
            job.update(W=dr.weight(d, d), q=_dense_input(dr, 1, d)[1])
        elif n == "o":
            _, rot, perm = _heads_input(dr, 1, d)
            job.update(W=dr.weight(d, d), q=rot, perm=perm)
        else:
            job.update(W=dr.weight(f, d), in_scale=_scaled_input(dr, 1, f)[1])
        st["todo"].append(job)
    return st


# ---------------------------------------------------------------------------------------------- one pass
def run(state):
    s, ctx = state, state["ctx"]
    if s["kind"] == "linear":
        return ctx.linear(s["x"], s["w"], s["r"])
    if s["kind"] == "layer":
        q, k, v = ctx.linear_multi(s["x_attn"], [s["q"], s["k"], s["v"]], s["r_attn"])
        o = ctx.linear(s["x_o"], s["o"], s["r_o"])
        gate, up = ctx.linear_multi(s["x_mlp"], [s["gate"], s["up"]], s["r_mlp"])
        down = ctx.linear(s["x_down"], s["down"])
        return dict(q=q, k=k, v=v, o=o, gate=gate, up=up, down=down)
    if s["kind"] == "plan":
        s["plan"].run()
        return s["y"]
    if s["kind"] == "calibrate":
        return ctx.calib_cov(s["x"], s["gram"], s["blocks"])
    out = []
    for job in s["todo"]:
        w = ctx.quantize(**job)
        out.append(w.export())
        w.free()
    return out


# ---------------------------------------------------------------------------------------------- bounds
def _weight_bytes(d_in, d_out, bits):
    return SALIENT * d_out * 2 + (d_in - SALIENT) * d_out * bits // 8 + (d_in - SALIENT) // GROUP * d_out * 4


def _linear_work(d_in, d_out, m, bits):
    return _weight_bytes(d_in, d_out, bits) + 2 * m * (d_in + d_out), 2 * m * d_in * d_out


def _rotation_work(d, blocks, m):
    """The operand R; its input is what the linear is given and its output stays inside the call."""
    return 2 * d * (d // blocks), 2 * m * d * (d // blocks)


def work(case):
    c = case
    if c["kind"] == "linear":
        parts = [_linear_work(c["d_in"], c["d_out"], c["m"], c["bits"])]
        if c["rotation"] != "none":
            parts.append(_rotation_work(c["d_in"], 1 if c["rotation"] == "dense" else c["d_in"] // HEAD, c["m"]))
    elif c["kind"] in ("layer", "plan"):
        d, f, m, bits = c["d"], c["f"], c["m"], c["bits"]
        parts = [_linear_work(d, 3 * d, m, bits), _linear_work(d, d, m, bits), _linear_work(d, 2 * f, m, bits),
                 _linear_work(f, d, m, bits), _rotation_work(d, 1, m), _rotation_work(d, d // HEAD, m), _rotation_work(d, 1, m)]
    elif c["kind"] == "calibrate":
        n, d, dh = c["tokens"], c["d"], c["d"] // c["blocks"]
        # C is symmetric: half of the products determine it
        parts = [(n * d * (4 if c["fp32"] else 2) + 2 * 4 * d * dh, n * d * (dh + 1))]
    else:
        d, f, parts = c["d"], c["f"], []
        for n in c["linears"].split(","):
            d_in, dh = (f, 0) if n == "down" else (d, d if n == "q" else HEAD)
            parts.append((2 * d_in * d + 4 * d_in * max(dh, 1) + _weight_bytes(d_in, d, c["bits"]), 2 * d_in * max(dh, 1) * d))
    return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}


def tolerance(case):
    """About four times what the path shows against the same sums in 64 bits."""
    if case["kind"] == "quantize":
        return "exact"            # codes, scales and zeros follow one fp32 chain and one IEEE formula
    if case["kind"] == "calibrate":
        # fp32 sums; from fp16 activations the tensor core cuts its accumulator once per 16 tokens, an error that
        # grows with the tokens (9e-5 at 16384, 1.2e-5 at 4096)
        rel = 2e-5 if case["fp32"] else max(5e-5, 3.6e-4 * case["tokens"] / 16384)
        return {"rel": rel, "max": 4 * rel}
    # fp16 x R, fp16 weights, fp16 y: 2.1e-4 to 3.1e-4, at most one unit in the last place of y (1e-3)
    return {"rel": 1.2e-3, "max": 4e-3}
