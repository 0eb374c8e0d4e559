"""Performance cases of the FlashDecoder library: what its users have it do, at the sizes of
its own configurations and around them.

Whole calls: decoding a clip chunk by chunk through a stream handle (from device or from pinned
host memory), decoding several streams through the stacked batch, one streaming training step.
Layers, each through its kernel-level call: attention over the rolling cache, the fused QKV
projection, a block's MLP (norm, up, down; bf16 or e4m3, GELU or gated), the pixel head, and the
row-wise backward of the head. ``exact`` evaluates the same mathematics with torch in 64 bits.
"""
from __future__ import annotations

import math
import types

import numpy as np
import torch

from paper_2607_14898_gb300 import flashdec as fd

F64 = torch.float64
DEV = "cuda"
EXACT_FLOPS = 4e12  # 64-bit work above this takes longer than a check is worth


# ------------------------------------------------------------------ the cases
def _model(**kw):
    """Shape of a decoder; the defaults are the 480p configuration (60 x 104 latents of 16
    channels, patch 2: 1560 tokens; 16 heads on 4 KV groups, window 4, 4 frames per chunk)."""
    c = dict(channels=16, lat_h=60, lat_w=104, patch=2, hidden=1024, groups=4, blocks=24,
             refine=2, window=4, r_t=4, vae=8, gated=False, qk_norm=False, fp8=False,
             one_first=False, u8=False, chunks=5)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest stream a user decodes: two chunks of a 64-token frame, 2 blocks of width
        # 256; every kernel is a few microseconds, so launches and their latency count
        dict(name="decode_tiny", kind="decode", host=False,
             **_model(lat_h=8, lat_w=8, patch=1, hidden=256, groups=2, blocks=2, refine=0,
                      window=2, r_t=1, chunks=2)),
        # the flagship: a 480p stream through the full 24 + 2 block model; five chunks, so the
        # four-chunk caches fill and evict
        dict(name="decode_480p", kind="decode", host=False, **_model()),
        # serving: eight independent 480p streams, stacked, one model
        dict(name="batch_480p_x8", kind="batch", streams=8, **_model(chunks=2)),
        # one training step of the 480p model over a clip of two latent frames (8 pixel frames)
        dict(name="train_480p", kind="train", **_model(chunks=2)),
        # a small odd training step: 130 tokens per frame (padded rows, keys not a multiple of
        # 8), window 3 over five chunks
        dict(name="train_small_odd", kind="train",
             **_model(lat_h=20, lat_w=26, hidden=256, groups=2, blocks=2, refine=1, window=3)),
        # one backbone attention layer of a 480p chunk over its full cache
        dict(name="attn_480p", kind="attention", rows=1560, keys=6240, heads=16, groups=4),
        # the largest attention layer: 720p refinement, 14400 queries over 57600 keys
        dict(name="attn_720p_refine", kind="attention", rows=14400, keys=57600, heads=16,
             groups=4),
        # the QKV projection with norm, rotary embedding and cache append, 480p backbone chunk
        dict(name="qkv_480p", kind="qkv", grid_h=30, grid_w=52, frames=1, window=4, step=5,
             hidden=1024, heads=16, groups=4, qk_norm=False),
        # the MLP half of a 480p backbone block: norm, up with GELU, down into the residual
        dict(name="mlp_480p", kind="mlp", rows=1560, hidden=1024, ratio=4, gated=False, fp8=False),
        # the same of the widest layout, gated, with e4m3 products
        dict(name="mlp_xl_fp8", kind="mlp", rows=1560, hidden=1536, ratio=4, gated=True, fp8=True),
        # the pixel head of a 720p chunk (4 frames of 3600 tokens) into uint8 frames
        dict(name="head_720p_u8", kind="head", grid_h=45, grid_w=80, frames=4, hidden=1024, rs=16,
             u8=True),
        # the loss and the row-wise backward of the head, a 480p chunk of 4 frames
        dict(name="head_bwd_480p", kind="head_bwd", grid_h=30, grid_w=52, frames=4, hidden=1024,
             rs=16),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _draw_model(rng, kind):
    hidden = 128 * rng.choice([2, 2, 4, 6, 8, 12] if kind != "train" else [2, 2, 4, 6, 8])
    heads = hidden // 64
    wan22 = rng.random() < 0.3  # 48-channel, 16x latents at patch 1, against 16-channel, 8x
    patch = 1 if wan22 else rng.choice([1, 2, 2])
    gh, gw = _log_int(rng, 4, 45), _log_int(rng, 4, 80)
    c = _model(channels=48 if wan22 else 16, lat_h=gh * patch, lat_w=gw * patch, patch=patch,
               hidden=hidden, groups=rng.choice([g for g in (1, 2, 3, 4) if heads % g == 0]),
               blocks=rng.randint(1, 4), refine=rng.randint(0, 2), window=rng.randint(1, 4),
               r_t=rng.choice([1, 2, 4, 4]), vae=16 if wan22 else 8, gated=rng.random() < 0.4,
               qk_norm=rng.random() < 0.2, one_first=rng.random() < 0.2, chunks=rng.randint(1, 5))
    if kind == "train":
        c["chunks"] = rng.randint(1, 3 if gh * gw > 1000 else 6)
    else:
        c["u8"] = rng.random() < 0.4
        c["fp8"] = rng.random() < 0.2
    return c


def draw(rng):
    kind = rng.choice(["decode", "decode", "batch", "train", "train", "attention", "attention",
                       "qkv", "mlp", "mlp", "head", "head_bwd"])
    if kind == "decode":
        return dict(kind=kind, host=rng.random() < 0.3, **_draw_model(rng, kind))
    if kind == "batch":
        return dict(kind=kind, streams=rng.randint(2, 8), **_draw_model(rng, kind))
    if kind == "train":
        return dict(kind=kind, **_draw_model(rng, kind))
    if kind == "attention":
        groups = rng.randint(1, 4)
        rows = _log_int(rng, 64, 14400)
        return dict(kind=kind, rows=rows, keys=rows * rng.randint(1, 4) - rng.choice([0, 0, 1, 7]),
                    heads=groups * rng.choice([1, 2, 4, 6]), groups=groups)
    hidden = 128 * rng.choice([2, 4, 6, 8, 12])
    gh, gw = _log_int(rng, 3, 45), _log_int(rng, 5, 80)
    frames = rng.choice([1, 2, 4])
    if kind == "qkv":
        heads = hidden // 64
        return dict(kind=kind, grid_h=gh, grid_w=gw, frames=frames, window=rng.randint(1, 4),
                    step=rng.randint(0, 40), hidden=hidden, heads=heads,
                    groups=rng.choice([g for g in (1, 2, 3, 4) if heads % g == 0]),
                    qk_norm=rng.random() < 0.3)
    if kind == "mlp":
        return dict(kind=kind, rows=_log_int(rng, 33, 14400), hidden=hidden, ratio=4,
                    gated=rng.random() < 0.5, fp8=rng.random() < 0.4)
    if kind == "head":
        return dict(kind=kind, grid_h=gh, grid_w=gw, frames=frames, hidden=hidden,
                    rs=rng.choice([8, 16]), u8=rng.random() < 0.5)
    return dict(kind=kind, grid_h=gh, grid_w=gw, frames=frames, hidden=hidden,
                rs=rng.choice([8, 16]))


# ------------------------------------------------------------------ shapes and inputs
def _config(c):
    return types.SimpleNamespace(
        latent_channels=c["channels"], latent_h=c["lat_h"], latent_w=c["lat_w"],
        patch=c["patch"], hidden=c["hidden"], heads=c["hidden"] // 64, kv_groups=c["groups"],
        mlp_ratio=4, n_blocks=c["blocks"], n_refine=c["refine"], window=c["window"],
        r_t=c["r_t"], vae_spatial=c["vae"], out_channels=3, out_u8=c["u8"],
        mlp_gated=c["gated"], qk_norm=c["qk_norm"], mlp_fp8=c["fp8"],
        first_chunk_frames=1 if c["one_first"] else 0, rope_mode="abs", norm_eps=1e-6,
        rope_base=10000.0)


def _dims(c):
    gh, gw, rs = c["lat_h"] // c["patch"], c["lat_w"] // c["patch"], c["vae"] * c["patch"]
    return types.SimpleNamespace(
        gh=gh, gw=gw, L=gh * gw, rs=rs, D=c["hidden"], N=c["hidden"] // 64, G=c["groups"],
        cin=c["channels"] * c["patch"] ** 2, qkv=c["hidden"] + 128 * c["groups"],
        up=(8 if c["gated"] else 4) * c["hidden"], out=3 * rs * rs)


def _layout(c):
    """(name, shape) of the weight blob's tensors, in the order of include/flashdec.h."""
    d = _dims(c)
    D = d.D

    def block(p):
        return [(p + "n1", (D,)), (p + "wqkv", (d.qkv, D)), (p + "bqkv", (d.qkv,)),
                (p + "gk", (64,)), (p + "g2", (64,)), (p + "wo", (D, D)), (p + "bo", (D,)),
                (p + "n2", (D,)), (p + "w1", (d.up, D)), (p + "b1", (d.up,)),
                (p + "w2", (D, 4 * D)), (p + "b2", (D,))]
    out = [("we", (D, d.cin)), ("be", (D,))]
    for b in range(c["blocks"]):
        out += block(f"B{b}.")
    out += [("nf", (D,)), ("wt", (c["r_t"] * D, D)), ("bt", (c["r_t"] * D,))]
    for b in range(c["refine"]):
        out += block(f"R{b}.")
    return out + [("nh", (D,)), ("wh1", (D, D)), ("bh1", (D,)), ("wh2", (d.out, D)),
                  ("bh2", (d.out,))]


def _gen(seed, stream):
    return torch.Generator(device=DEV).manual_seed(seed * 1009 + stream)


def _randn(shape, gen, scale=1.0, dtype=torch.float32):
    return (torch.randn(shape, generator=gen, device=DEV) * scale).to(dtype)


def _gain(n, gen):
    return 1 + 0.02 * torch.randn(n, generator=gen, device=DEV)


def _blob(c, seed):
    """Random-init weights N(0, 0.02^2), gains 1 + N(0, 0.02^2), as one bf16 tensor."""
    layout = _layout(c)
    flat = _randn(sum(math.prod(s) for _, s in layout), _gen(seed, 1), 0.02)
    off = 0
    for name, shape in layout:
        n = math.prod(shape)
        if name.rsplit(".", 1)[-1] in ("n1", "n2", "gk", "g2", "nf", "nh"):
            flat[off:off + n] += 1.0
        off += n
    return flat.to(torch.bfloat16)


def _latents(c, seed, n):
    return _randn((n, c["channels"], c["lat_h"], c["lat_w"]), _gen(seed, 2))


def _targets(c, seed):
    """Pixels in [-1, 1], away from the decoder's near-zero outputs."""
    d, g = _dims(c), _gen(seed, 3)
    shape = (c["chunks"], 3, c["r_t"], d.gh * d.rs, d.gw * d.rs)
    mag = torch.rand(shape, generator=g, device=DEV) * 0.7 + 0.3
    return torch.where(torch.rand(shape, generator=g, device=DEV) < 0.5, mag, -mag)


def _weights(c, seed):
    return fd.Weights(_config(c), _blob(c, seed).view(torch.int16).cpu().numpy().view(np.uint16))


def _pixel_buffers(c, n_chunks, host=False):
    d = _dims(c)
    out = []
    for t in range(n_chunks):
        frames = 1 if c["one_first"] and t == 0 else c["r_t"]
        shape = (3, frames, d.gh * d.rs, d.gw * d.rs)
        dtype = torch.uint8 if c["u8"] else torch.float32
        out.append(torch.zeros(shape, dtype=dtype, pin_memory=True) if host
                   else torch.zeros(shape, dtype=dtype, device=DEV))
    return out


def _row_blocks(gate, up):
    """Gate and up rows interleaved in blocks of 32, the row order of the gated epilogues."""
    n = gate.shape[0]
    return torch.stack([gate.reshape(n // 32, 32, *gate.shape[1:]),
                        up.reshape(n // 32, 32, *up.shape[1:])], 1).reshape(2 * n, *gate.shape[1:])


def _inputs(c, seed):
    """The tensors of a layer case."""
    g, kind, s = _gen(seed, 4), c["kind"], types.SimpleNamespace()
    if kind == "attention":
        pitch = (c["keys"] + 127) // 128 * 128
        s.q = _randn((c["rows"], c["heads"] * 64), g, 0.6, torch.bfloat16)
        s.k = torch.zeros(c["groups"], pitch, 64, dtype=torch.bfloat16, device=DEV)
        s.k[:, :c["keys"]] = _randn((c["groups"], c["keys"], 64), g)
        s.vt = torch.zeros(c["groups"], 64, pitch, dtype=torch.float16, device=DEV)
        s.vt[:, :, :c["keys"]] = _randn((c["groups"], 64, c["keys"]), g)
        s.pitch = pitch
    elif kind == "qkv":
        M, D = c["grid_h"] * c["grid_w"] * c["frames"], c["hidden"]
        n = (c["heads"] + 2 * c["groups"]) * 64
        s.a = _randn((M, D), g, 1.0, torch.bfloat16)
        s.w, s.b = _randn((n, D), g, 0.02, torch.bfloat16), _randn((n,), g, 0.02)
        s.gk, s.g2 = _gain(64, g), _gain(64, g)
        s.pitch = (c["window"] * M + 127) // 128 * 128
    elif kind == "mlp":
        M, D = c["rows"], c["hidden"]
        Dm = c["ratio"] * D
        s.h, s.gain = _randn((M, D), g), _gain(D, g)
        w1 = _randn((2 * Dm if c["gated"] else Dm, D), g, 0.02)
        s.b1 = _randn((w1.shape[0],), g, 0.02)
        w2, s.b2 = _randn((D, Dm), g, 0.02), _randn((D,), g, 0.02)
        if c["fp8"]:
            # e4m3 weights with one power-of-two scale, e4m3 activations with static scales
            s.ws, s.su, s.sh = 2.0 ** -11, 2.0 ** -4, 2.0 ** -5
            q = [(w / s.ws).clamp(-448, 448).to(torch.float8_e4m3fn) for w in (w1, w2)]
            s.w1, s.w2 = (x.view(torch.uint8) for x in q)
            s.w1f, s.w2f = (x.to(torch.float32) * s.ws for x in q)
            s.cs1 = torch.full((w1.shape[0],), s.su * s.ws, device=DEV)
            s.cs2 = torch.full((D,), s.sh * s.ws, device=DEV)
        else:
            s.w1, s.w2 = w1.to(torch.bfloat16), w2.to(torch.bfloat16)
            s.w1f, s.w2f = s.w1, s.w2
        if c["gated"]:
            s.w1 = _row_blocks(s.w1[:Dm], s.w1[Dm:]).contiguous()
            s.b1b = _row_blocks(s.b1[:Dm], s.b1[Dm:]).contiguous()
        else:
            s.b1b = s.b1
    elif kind == "head":
        M, D, n = c["grid_h"] * c["grid_w"] * c["frames"], c["hidden"], 3 * c["rs"] ** 2
        s.h, s.gain = _randn((M, D), g), _gain(D, g)
        s.w1, s.b1 = _randn((D, D), g, 0.02, torch.bfloat16), _randn((D,), g, 0.02)
        s.w2, s.b2 = _randn((n, D), g, 0.05, torch.bfloat16), _randn((n,), g, 0.02)
    else:  # head_bwd
        M, D, n = c["grid_h"] * c["grid_w"] * c["frames"], c["hidden"], 3 * c["rs"] ** 2
        s.f = _randn((M, n), g, 0.1)
        s.target = torch.rand(3, c["frames"], c["grid_h"] * c["rs"], c["grid_w"] * c["rs"],
                              generator=g, device=DEV) * 2 - 1
        s.z, s.da = _randn((M, D), g, 0.6), _randn((M, D), g, 1e-3)
        s.x, s.gain, s.dy = _randn((M, D), g), _gain(D, g), _randn((M, D), g, 1e-3)
    return s


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind in ("decode", "batch", "train"):
        s = types.SimpleNamespace(case=c, w=_weights(c, seed))
        cfg = _config(c)
        if kind == "train":
            s.trainer = fd.Trainer(cfg, s.w, c["chunks"])
            s.z, s.x = _latents(c, seed, c["chunks"]), _targets(c, seed)
            s.loss = torch.zeros(1, device=DEV)
            s.grads = torch.zeros(s.trainer.grad_elems, device=DEV)
            return s
        n = c.get("streams", 1)
        s.dec = [fd.Decoder(cfg, s.w) for _ in range(n)]
        z = _latents(c, seed, n * c["chunks"])
        host = c.get("host", False)
        if host:
            z = z.cpu().pin_memory()
        s.z = [[z[i * c["chunks"] + t] for t in range(c["chunks"])] for i in range(n)]
        s.pix = [_pixel_buffers(c, c["chunks"], host) for _ in range(n)]
        if kind == "batch":
            s.batch = fd.Batch(cfg, s.w, n)
        return s
    s = _inputs(c, seed)
    s.case = c
    s.err = torch.zeros(1, dtype=torch.int32, device=DEV)
    if kind == "attention":
        s.out = torch.empty_like(s.q)
        s.ws = torch.empty(max(16, fd.attention_workspace_bytes(c["rows"], c["heads"], c["groups"],
                                                                c["keys"])),
                           dtype=torch.uint8, device=DEV)
    elif kind == "qkv":
        M = s.a.shape[0]
        s.q = torch.empty(M, c["heads"] * 64, dtype=torch.bfloat16, device=DEV)
        s.k = torch.zeros(c["groups"], s.pitch, 64, dtype=torch.bfloat16, device=DEV)
        s.vt = torch.zeros(c["groups"], 64, s.pitch, dtype=torch.float16, device=DEV)
        s.rope = torch.empty(c["frames"], 12, 2, device=DEV)
        fd.op_rope_table(c["step"], c["frames"], 10000.0, s.rope)
    elif kind == "mlp":
        M, D, t = c["rows"], c["hidden"], torch.uint8 if c["fp8"] else torch.bfloat16
        s.u = torch.empty(M, D, dtype=t, device=DEV)
        s.hid = torch.empty(M, c["ratio"] * D, dtype=t, device=DEV)
        s.w1f = s.w2f = None
    elif kind == "head":
        s.u, s.a = (torch.empty(s.h.shape, dtype=torch.bfloat16, device=DEV) for _ in range(2))
        s.pix = torch.empty(3, c["frames"], c["grid_h"] * c["rs"], c["grid_w"] * c["rs"],
                            dtype=torch.uint8 if c["u8"] else torch.float32, device=DEV)
    elif kind == "head_bwd":
        s.df, s.loss = torch.empty_like(s.f), torch.zeros(1, device=DEV)
        s.dz, s.dz16 = torch.empty_like(s.z), torch.empty_like(s.z, dtype=torch.bfloat16)
        s.dx, s.dg = torch.empty_like(s.x), torch.empty_like(s.gain)
    return s


# ------------------------------------------------------------------ one pass
def run(s):
    c, kind = s.case, s.case["kind"]
    if kind == "decode":
        dec = s.dec[0]
        dec.reset()
        if c["host"]:
            dec.decode_sequence_host(s.z[0], s.pix[0])
        else:
            for z, pix in zip(s.z[0], s.pix[0]):
                dec.decode_chunk(z, pix)
        return s.pix[0]
    if kind == "batch":
        for dec in s.dec:
            dec.reset()
        for t in range(c["chunks"]):
            s.batch.decode(s.dec, [z[t] for z in s.z], [p[t] for p in s.pix])
        return s.pix
    if kind == "train":
        s.trainer.step(s.z, s.x, s.loss, s.grads)
        return {"loss": s.loss, "grads": s.grads}
    if kind == "attention":
        fd.op_attention(s.q, s.k, s.vt, c["heads"], c["groups"], s.pitch, c["keys"], s.out,
                        workspace=s.ws, err=s.err)
        return s.out
    if kind == "qkv":
        fd.op_qkv(s.a, s.w, s.b, s.gk, s.g2, c["heads"], c["groups"], c["grid_h"] * c["grid_w"],
                  c["grid_w"], c["frames"], c["window"], c["step"], 1e-6, 10000.0, s.rope, s.q,
                  s.k, s.vt, s.pitch, err=s.err, qk_norm=c["qk_norm"])
        return {"q": s.q, "k": s.k, "vt": s.vt}
    if kind == "mlp":
        up = fd.EPI_SWIGLU if c["gated"] else fd.EPI_GELU
        if c["fp8"]:
            fd.op_rmsnorm_e4m3(s.h, s.gain, 1e-6, 1 / s.su, s.u)
            fd.op_linear_e4m3(up, s.u, s.w1, s.cs1, s.b1b, s.hid, 1 / s.sh, err=s.err)
            fd.op_linear_e4m3(fd.EPI_RESID, s.hid, s.w2, s.cs2, s.b2, s.h, err=s.err)
        else:
            fd.op_rmsnorm(s.h, s.gain, 1e-6, s.u)
            fd.op_linear(up, s.u, s.w1, s.b1b, s.hid, err=s.err)
            fd.op_linear(fd.EPI_RESID, s.hid, s.w2, s.b2, s.h, err=s.err)
        return {"u": s.u, "hid": s.hid, "h": s.h}
    if kind == "head":
        fd.op_rmsnorm(s.h, s.gain, 1e-6, s.u)
        fd.op_linear(fd.EPI_GELU, s.u, s.w1, s.b1, s.a, err=s.err)
        fd.op_linear_pixel(s.a, s.w2, s.b2, c["frames"], c["grid_h"], c["grid_w"], 3, c["rs"],
                           fd.DTYPE_U8 if c["u8"] else fd.DTYPE_F32, s.pix, err=s.err)
        return {"u": s.u, "a": s.a, "pix": s.pix}
    fd.op_l1_pixel_bwd(s.f, s.target, c["frames"], c["grid_h"], c["grid_w"], 3, c["rs"], s.df,
                       s.loss)
    fd.op_gelu_bwd(s.z, s.da, s.dz, s.dz16)
    fd.op_rmsnorm_bwd(s.x, s.gain, s.dy, 1e-6, s.dx, s.dg)
    return {"df": s.df, "loss": s.loss, "dz": s.dz, "dz16": s.dz16, "dx": s.dx, "dg": s.dg}


# ------------------------------------------------------------------ work of a pass
def _model_work(c, train):
    """FLOPs of the products and attention over the clip; bytes of weights (once per chunk when
    streaming), inputs, outputs and of the caches read and written."""
    d, T, r = _dims(c), c["chunks"], c["r_t"]
    params = sum(math.prod(s) for _, s in _layout(c))
    block = d.D * (d.qkv + d.D + d.up + 4 * d.D)
    flops = bytes_ = 0.0
    for t in range(T):
        n = min(t + 1, c["window"])
        flops += 2 * d.L * (d.cin * d.D + c["blocks"] * block + r * d.D * d.D)
        flops += 2 * r * d.L * (c["refine"] * block + d.D * d.D + d.D * d.out)
        flops += 4 * d.L * n * d.L * d.D * (c["blocks"] + c["refine"] * r * r)
        bytes_ += 256 * d.G * n * d.L * (c["blocks"] + c["refine"] * r)
        bytes_ += 4 * d.L * d.cin + r * d.L * d.out * (1 if c["u8"] and not train else 4)
    if train:
        return {"bytes": bytes_ + params * (2 + 4), "flops": 3 * flops}
    n = c.get("streams", 1)
    return {"bytes": n * bytes_ + T * params * 2, "flops": n * flops}


def work(case):
    c, kind = case, case["kind"]
    if kind in ("decode", "batch", "train"):
        return _model_work(c, kind == "train")
    if kind == "attention":
        return {"bytes": 4 * c["rows"] * c["heads"] * 64 + 256 * c["groups"] * c["keys"],
                "flops": 4 * c["rows"] * c["keys"] * c["heads"] * 64}
    D = c["hidden"]
    M = c["rows"] if kind == "mlp" else c["grid_h"] * c["grid_w"] * c["frames"]
    if kind == "qkv":
        n = (c["heads"] + 2 * c["groups"]) * 64
        return {"bytes": 2 * (M * D + n * D + M * n), "flops": 2 * M * n * D}
    if kind == "mlp":
        Dm, e = c["ratio"] * D, 1 if c["fp8"] else 2
        n = (3 if c["gated"] else 2) * Dm * D
        return {"bytes": 8 * M * D + e * (n + M * D + M * Dm), "flops": 2 * M * n}
    n = 3 * c["rs"] ** 2
    if kind == "head":
        return {"bytes": M * (4 * D + 4 * D + n * (1 if c["u8"] else 4)) + 2 * D * (D + n),
                "flops": 2 * M * D * (D + n)}
    return {"bytes": M * (3 * 4 * n + (4 + 4 + 4 + 2) * D + 3 * 4 * D), "flops": M * (n + 40 * D)}


# ------------------------------------------------------------------ the same in 64 bits
def _rms(x, g):
    return x * torch.rsqrt(x.square().mean(-1, keepdim=True) + 1e-6) * g


def _gelu(x):
    return 0.5 * x * (1 + torch.erf(x / math.sqrt(2.0)))


def _silu(x):
    return x * torch.sigmoid(x)


def _angles(frames, gh, gw):
    """Rotation angles [frames gh gw][32] of the tokens of the given temporal indices: 12
    temporal, 10 row, 10 column pairs."""
    def inv(n):
        return 10000.0 ** (-torch.arange(n, dtype=F64, device=DEV) / n)
    f = torch.as_tensor(frames, dtype=F64, device=DEV)
    y, x = (torch.arange(n, dtype=F64, device=DEV) for n in (gh, gw))
    shape = (len(frames), gh, gw)
    t = (f[:, None] * inv(12))[:, None, None].expand(*shape, 12)
    r = (y[:, None] * inv(10))[None, :, None].expand(*shape, 10)
    col = (x[:, None] * inv(10))[None, None].expand(*shape, 10)
    return torch.cat([t, r, col], -1).reshape(-1, 32)


def _rotate(x, a):
    """x [heads][rows][64], interleaved pairs rotated by a [rows][32]."""
    e, o, cs, sn = x[..., 0::2], x[..., 1::2], a.cos(), a.sin()
    return torch.stack([e * cs - o * sn, e * sn + o * cs], -1).flatten(-2)


def _attend(q, k, v):
    """q [N][rows][64] over k, v [G][keys][64], a bounded block of rows at a time."""
    hpg, step = q.shape[0] // k.shape[0], max(1, (1 << 27) // k.shape[1])
    out = []
    for n in range(q.shape[0]):
        kk, vv = k[n // hpg], v[n // hpg]
        out.append(torch.cat([torch.softmax(p @ kk.T / 8, -1) @ vv
                              for p in q[n].split(step)]))
    return torch.stack(out)


def _project(u, w, b, heads, groups, gk, g2, qk_norm, ang):
    x = (u @ w.T + b).reshape(u.shape[0], heads + 2 * groups, 64).transpose(0, 1)
    q, k, v = x[:heads], x[heads:heads + groups], x[heads + groups:]
    k = _rms(k, gk)
    if qk_norm:
        q = _rms(q, g2)
    else:
        v = _rms(v, g2)
    return _rotate(q, ang), _rotate(k, ang), v


def _mlp64(u, w1, b1, w2, b2, gated):
    z = u @ w1.T + b1
    if gated:
        n = z.shape[1] // 2
        a = _silu(z[:, :n]) * z[:, n:]
    else:
        a = _gelu(z)
    return a, a @ w2.T + b2


def _decode64(c, P, z):
    """The decoder of Algorithm 1 on a clip: unclamped pixels of every chunk."""
    d, r, W = _dims(c), c["r_t"], c["window"]
    cache = {}

    def block(p, h, ang):
        q, k, v = _project(_rms(h, P[p + "n1"]), P[p + "wqkv"], P[p + "bqkv"], d.N, d.G,
                           P[p + "gk"], P[p + "g2"], c["qk_norm"], ang)
        cache[p] = (cache.get(p, []) + [(k, v)])[-W:]
        o = _attend(q, *(torch.cat(t, 1) for t in zip(*cache[p])))
        h = h + o.transpose(0, 1).reshape(h.shape) @ P[p + "wo"].T + P[p + "bo"]
        return h + _mlp64(_rms(h, P[p + "n2"]), P[p + "w1"], P[p + "b1"], P[p + "w2"],
                          P[p + "b2"], c["gated"])[1]

    out = []
    for t in range(len(z)):
        x = torch.nn.functional.pixel_unshuffle(z[t].to(F64)[None], c["patch"])[0]
        h = x.reshape(d.cin, d.L).T @ P["we"].T + P["be"]
        ang = _angles([t], d.gh, d.gw)
        for b in range(c["blocks"]):
            h = block(f"B{b}.", h, ang)
        e = _rms(h, P["nf"]) @ P["wt"].T + P["bt"]
        h = e.reshape(d.L, r, d.D).transpose(0, 1).reshape(r * d.L, d.D)
        ang = _angles([t * r + i for i in range(r)], d.gh, d.gw)
        for b in range(c["refine"]):
            h = block(f"R{b}.", h, ang)
        f = _gelu(_rms(h, P["nh"]) @ P["wh1"].T + P["bh1"]) @ P["wh2"].T + P["bh2"]
        frames = 1 if c["one_first"] and t == 0 else r
        f = f.reshape(r, d.gh, d.gw, d.out)[:frames].permute(0, 3, 1, 2)
        out.append(torch.nn.functional.pixel_shuffle(f, d.rs).transpose(0, 1))
    return out


def exact(case, seed):
    c, kind = case, case["kind"]
    if work(c)["flops"] > EXACT_FLOPS or c.get("fp8") and kind != "mlp":
        return None
    if kind in ("decode", "batch", "train"):
        if kind != "train" and c["u8"]:
            return None
        flat, P, off = _blob(c, seed).to(F64).requires_grad_(kind == "train"), {}, 0
        for name, shape in _layout(c):
            n = math.prod(shape)
            P[name] = flat[off:off + n].view(shape)
            off += n
        z = _latents(c, seed, c.get("streams", 1) * c["chunks"])
        if kind == "train":
            d, x = _dims(c), _targets(c, seed).to(F64)
            if c["chunks"] * d.N * (c["window"] * d.L ** 2) * (
                    c["blocks"] + c["refine"] * c["r_t"] ** 2) > 3e9:
                return None  # the probabilities of every layer, kept for the backward
            pix = _decode64(c, P, z)
            total = sum(p.numel() for p in pix)
            loss = sum((p - t[:, :p.shape[1]]).abs().sum() for p, t in zip(pix, x)) / total
            loss.backward()
            return {"loss": loss.detach()[None], "grads": flat.grad}
        with torch.no_grad():
            pix = [[p.clamp(-1, 1) for p in _decode64(c, P, z[i:i + c["chunks"]])]
                   for i in range(0, len(z), c["chunks"])]
        return pix[0] if kind == "decode" else pix
    s = _inputs(c, seed)
    with torch.no_grad():
        if kind == "attention":
            n, q = c["keys"], s.q.to(F64).reshape(c["rows"], c["heads"], 64).transpose(0, 1)
            o = _attend(q, s.k[:, :n].to(F64), s.vt[:, :, :n].to(F64).transpose(1, 2))
            return o.transpose(0, 1).reshape(c["rows"], -1)
        if kind == "qkv":
            M, first = s.a.shape[0], c["step"] * c["frames"]
            ang = _angles(list(range(first, first + c["frames"])), c["grid_h"], c["grid_w"])
            q, k, v = _project(s.a.to(F64), s.w.to(F64), s.b.to(F64), c["heads"], c["groups"],
                               s.gk.to(F64), s.g2.to(F64), c["qk_norm"], ang)
            ring = torch.zeros(2, c["groups"], s.pitch, 64, dtype=F64, device=DEV)
            at = c["step"] % c["window"] * M
            ring[0, :, at:at + M], ring[1, :, at:at + M] = k, v
            return {"q": q.transpose(0, 1).reshape(M, -1), "k": ring[0],
                    "vt": ring[1].transpose(1, 2).contiguous()}
        if kind == "mlp":
            h = s.h.to(F64)
            u = _rms(h, s.gain.to(F64))
            a, y = _mlp64(u, s.w1f.to(F64), s.b1.to(F64), s.w2f.to(F64), s.b2.to(F64),
                          c["gated"])
            return {"u": None, "hid": None, "h": h + y} if c["fp8"] else \
                {"u": u, "hid": a, "h": h + y}
        if kind == "head":
            u = _rms(s.h.to(F64), s.gain.to(F64))
            a = _gelu(u @ s.w1.to(F64).T + s.b1.to(F64))
            f = a @ s.w2.to(F64).T + s.b2.to(F64)
            f = f.reshape(c["frames"], c["grid_h"], c["grid_w"], -1).permute(0, 3, 1, 2)
            pix = torch.nn.functional.pixel_shuffle(f, c["rs"]).transpose(0, 1).clamp(-1, 1)
            return {"u": u, "a": a, "pix": None if c["u8"] else pix}
        f = s.f.to(F64).reshape(c["frames"], c["grid_h"], c["grid_w"], -1).permute(0, 3, 1, 2)
        diff = torch.nn.functional.pixel_shuffle(f, c["rs"]).transpose(0, 1) - s.target.to(F64)
        df = torch.nn.functional.pixel_unshuffle(diff.sign().transpose(0, 1), c["rs"])
        z, x, gain, dy = (t.to(F64) for t in (s.z, s.x, s.gain, s.dy))
        dz = s.da.to(F64) * (0.5 * (1 + torch.erf(z / math.sqrt(2.0)))
                             + z * torch.exp(-0.5 * z * z) / math.sqrt(2 * math.pi))
        rr = torch.rsqrt(x.square().mean(-1, keepdim=True) + 1e-6)
        dx = rr * dy * gain - x * rr ** 3 * (dy * gain * x).mean(-1, keepdim=True)
        return {"df": df.permute(0, 2, 3, 1).reshape(s.f.shape) / s.f.numel(),
                "loss": diff.abs().mean()[None], "dz": dz, "dz16": dz, "dx": dx,
                "dg": (dy * x * rr).sum(0)}
