"""The streaming training step on the GPU (fd_train_step, Sec. 3.3 "Training--Inference
Consistency", Sec. 3.5 Eq. loss) against the oracle's explicit backward of the same step
(oracle.backward.training_step_explicit, itself pinned to autograd of the streaming decode, to
the masked full-clip pass and to central differences): the L1 loss and the gradient of every
decoder parameter."""
import numpy as np
import pytest
import torch

import oracle
import synth
from oracle.backward import training_step_explicit
import oracle.backward as oracle_bwd

pytestmark = pytest.mark.gpu

fdp = pytest.importorskip("paper_2607_14898_gb300.flashdec")

# Bars. The GPU runs every product on bf16 operands (the forward's and the backward's) with fp32
# accumulation; the fp64 oracle with only its forward operands rounded to bf16 / fp16 already
# moves the gradients by up to 0.49 % (per tensor, relative L2; median 0.16-0.28 %; measured on
# tiny, tiny_rt, tiny_qk and small), and the backward's own roundings add about as much again.
# The per-tensor bar is 4x that worst movement; the bar on the median over the tensors is 2x the
# worst movement (the GB300 measures worst 0.72-1.50 %, median 0.42-0.48 %).
GRAD_REL = 2e-2      # per tensor: ||g_gpu - g|| / ||g||
GRAD_REL_MEDIAN = 1e-2
LOSS_REL = 1e-3


@pytest.fixture(scope="module", autouse=True)
def _setup(torch_threads):
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    fdp.lib()


def gpu_step(cfg, w, z, x):
    W = fdp.Weights(cfg, fdp.pack_blob(cfg, w))
    tr = fdp.Trainer(cfg, W, len(z))
    lat = torch.from_numpy(np.ascontiguousarray(np.stack(z))).cuda()
    # the step's target layout has r_t frames per chunk; a one-frame chunk 0 is padded with
    # NaN, which the step must not read
    rt = cfg.r_t
    x = [np.concatenate([c, np.full(c.shape[:1] + (rt - c.shape[1],) + c.shape[2:], np.nan,
                                    np.float32)], axis=1) if c.shape[1] < rt else c for c in x]
    tgt = torch.from_numpy(np.ascontiguousarray(np.stack(x))).cuda()
    loss = torch.zeros(1, device="cuda")
    grads = torch.full((tr.grad_elems,), float("nan"), device="cuda")
    tr.step(lat, tgt, loss, grads)
    assert tr.status() == fdp.FD_OK
    out = float(loss.item()), grads.cpu().double()
    tr.close()
    W.close()
    return out


def split(cfg, flat):
    out, off = {}, 0
    for name, shape, _ in synth.weight_layout(cfg):
        n = int(np.prod(shape))
        out[name] = flat[off:off + n].reshape(shape)
        off += n
    assert off == flat.numel()
    return out


@pytest.mark.parametrize("name", ["tiny", "tiny_rt", "tiny_qk", "small", "train_480p_grid",
                                  "tiny_gated", "small_f1", "tiny_xl"])
def test_training_step_matches_the_oracle(name):
    """Loss and every parameter's gradient of one step over the preset's clip. The targets keep
    0.3 away from zero, so that no pixel sits near the kink of |x_hat - x| (the outputs of the
    seeded decoder stay well inside [-0.3, 0.3]). train_480p_grid has the 480p token grid (1560
    tokens per frame, padded to 1664 rows; 3120 refined rows per chunk) at reduced width and
    depth: the padding, the fused forward's key maps and the band at the product's token count.
    tiny_gated, small_f1 and tiny_xl carry the XL layout's gated-SiLU MLP and the one-frame
    first chunk (whose loss covers the (T - 1) r_t + 1 frames the clip decodes to)."""
    cfg = synth.PRESETS[name]
    w, z = synth.make_weights(cfg), synth.make_latents(cfg)
    x = synth.make_target_pixels(cfg, min_abs=0.3)
    loss_ref, g_ref = training_step_explicit(cfg, w, z, x)
    loss, flat = gpu_step(cfg, w, z, x)
    g = split(cfg, flat)
    assert abs(loss - loss_ref) <= LOSS_REL * abs(loss_ref), (loss, loss_ref)
    rel = {}
    for k, ref in g_ref.items():
        ref = ref.reshape(g[k].shape)
        assert torch.isfinite(g[k]).all(), k
        rel[k] = float((g[k] - ref).norm() / max(float(ref.norm()), 1e-30))
    worst = max(rel, key=rel.get)
    print(f"{name}: loss {loss:.6f} (oracle {loss_ref:.6f}); gradient rel. error median "
          f"{np.median(list(rel.values())):.2e}, worst {rel[worst]:.2e} ({worst})")
    assert rel[worst] <= GRAD_REL, (worst, rel[worst])
    assert np.median(list(rel.values())) <= GRAD_REL_MEDIAN


def test_training_step_is_deterministic_and_refuses_other_layouts():
    """Two steps on the same inputs give the same bits (no order-dependent sums); FP8 MLPs
    (the inference-only lossy setting) are refused at creation."""
    cfg = synth.PRESETS["tiny_rt"]
    w, z = synth.make_weights(cfg), synth.make_latents(cfg)
    x = synth.make_target_pixels(cfg, min_abs=0.3)
    a = gpu_step(cfg, w, z, x)
    b = gpu_step(cfg, w, z, x)
    assert a[0] == b[0] and torch.equal(a[1], b[1])
    for other in (synth.PRESETS["small_fp8"], synth.PRESETS["tiny_gated_fp8"]):
        W = fdp.Weights(other, fdp.pack_blob(other, synth.make_weights(other)))
        with pytest.raises(fdp.FdError) as e:
            fdp.Trainer(other, W, 2)
        assert e.value.code == 2
        W.close()


# ------------------------------------------------------------------ single kernels of the step
def test_rmsnorm_backward_kernel():
    """fd_op_rmsnorm_bwd against the oracle's written-out derivative (oracle.backward), ragged
    row counts, the widths of the configs."""
    from oracle.backward import rms_norm_bwd
    from helpers import randn
    for M, D in ((520, 256), (130, 1024)):
        x = randn((M, D), M + D, 2.0)
        g = 1 + randn((D,), M + D + 1, 0.02)
        dy = randn((M, D), M + D + 2)
        dx = torch.empty(M, D, device="cuda")
        dg = torch.empty(D, device="cuda")
        fdp.op_rmsnorm_bwd(torch.from_numpy(x).cuda(), torch.from_numpy(g).cuda(),
                           torch.from_numpy(dy).cuda(), 1e-6, dx, dg)
        torch.cuda.synchronize()
        want_dx, want_dg = rms_norm_bwd(torch.from_numpy(x).double(), torch.from_numpy(g).double(),
                                        1e-6, torch.from_numpy(dy).double())
        for got, want, what in ((dx, want_dx, "dx"), (dg, want_dg, "dg")):
            err = float((got.cpu().double() - want).abs().max() / want.abs().max())
            assert err < 2e-5, (M, D, what, err)


def test_gelu_backward_kernel():
    """fd_op_gelu_bwd against GELU'(z) = Phi(z) + z phi(z) of the oracle, on a grid through the
    kink region and the tails; the bf16 copy is the rounding of the fp32 result."""
    from oracle.backward import gelu_bwd
    z = torch.linspace(-9, 9, 4097, dtype=torch.float32)
    da = torch.cos(torch.arange(4097, dtype=torch.float32))
    dz = torch.empty(4097, device="cuda")
    dz16 = torch.empty(4097, dtype=torch.bfloat16, device="cuda")
    fdp.op_gelu_bwd(z.cuda(), da.cuda(), dz, dz16)
    torch.cuda.synchronize()
    want = gelu_bwd(z.double(), da.double())
    assert float((dz.cpu().double() - want).abs().max()) < 2e-6
    assert torch.equal(dz16.cpu(), dz.cpu().to(torch.bfloat16))


def test_l1_pixel_backward_kernel():
    """fd_op_l1_pixel_bwd: the loss and dL/dF through the pixel shuffle against the oracle's
    l1_bwd and pixel_shuffle_bwd (the inverse permutation), on a 4-frame 480p-shaped chunk."""
    from oracle.backward import l1_bwd, pixel_shuffle_bwd
    from helpers import randn
    frames, gh, gw, C, rs = 4, 6, 7, 3, 16
    F = randn((frames * gh * gw, C * rs * rs), 5, 0.3)
    x = synth.make_target_pixels(synth.PRESETS["tiny"].replace(r_t=frames, latent_h=gh,
                                                               latent_w=gw, vae_spatial=rs),
                                 chunks=1, min_abs=0.3)[0]
    dF = torch.empty(F.shape, device="cuda")
    loss = torch.zeros(1, device="cuda")
    fdp.op_l1_pixel_bwd(torch.from_numpy(F).cuda(), torch.from_numpy(x).cuda(), frames, gh, gw,
                        C, rs, dF, loss)
    torch.cuda.synchronize()
    pix = oracle.pixel_shuffle(torch.from_numpy(F).double(), frames, gh, gw, C, rs)
    total = pix.numel()
    want_loss = float((pix - torch.from_numpy(x).double()).abs().sum() / total)
    want_dF = pixel_shuffle_bwd(l1_bwd(pix, x, total), frames, gh, gw, C, rs)
    assert abs(float(loss.item()) - want_loss) <= 1e-6 * want_loss
    assert float((dF.cpu().double() - want_dF).abs().max()) <= 1e-7 / total


@pytest.mark.parametrize("heads,Pc,Lp,L,N", [
    (2, 256, 128, 100, 384),   # padding query rows and padding keys, ragged 128-row tiles
    (4, 128, 128, 128, 256),   # no padding (the 480p backbone's heads of one group, shrunk)
    (1, 384, 384, 360, 1152),  # one head, three chunks of keys
])
def test_scores_backward_kernel(heads, Pc, Lp, L, N):
    """fd_op_scores_bwd (S and dP on the tensor cores, the softmax derivative in the epilogue)
    against oracle.attention_bwd: its dS, dS^T and P^T chained through fp64 products (dQ = dS K,
    dK = dS^T Q, dV = P^T dO) give the oracle's gradients of one KV group, with the log-sum-exp
    and delta of an fp64 forward. Padding query rows carry dO = 0, as in the step."""
    from helpers import bf16_values, randn
    M = heads * Pc
    rows = torch.arange(M)
    live = (rows % Pc % Lp) < L
    keys = (torch.arange(N) % Lp) < L
    q = torch.from_numpy(bf16_values(randn((M, 64), M + N, 1.0))).double()
    k = torch.from_numpy(bf16_values(randn((N, 64), M + N + 1, 1.0))).double()
    v = torch.from_numpy(bf16_values(randn((N, 64), M + N + 2, 1.0))).double()
    do = torch.from_numpy(bf16_values(randn((M, 64), M + N + 3, 1.0))).double()
    do[~live] = 0.0
    # the forward's log-sum-exp and delta = rowsum(dO o O), from their definitions in fp64
    s = (q @ k.T) / 8.0
    s[:, ~keys] = float("-inf")
    lse = torch.logsumexp(s, dim=1)
    o = torch.softmax(s, dim=1) @ v
    delta = (do * o).sum(dim=1)
    cu = lambda t: t.to(torch.bfloat16).cuda()
    dS = torch.empty(M, N, dtype=torch.bfloat16, device="cuda")
    dST = torch.empty(N, M, dtype=torch.bfloat16, device="cuda")
    PT = torch.empty(N, M, dtype=torch.bfloat16, device="cuda")
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    fdp.op_scores_bwd(cu(q), cu(do), cu(k), cu(v), lse.float().cuda(), delta.float().cuda(), Pc,
                      Lp, L, dS, dST, PT, err=err)
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    assert torch.equal(dST.cpu(), dS.cpu().T.contiguous())
    dS, PT = dS.cpu().double(), PT.cpu().double()
    assert float(dS[~live].abs().sum()) == 0.0 and float(PT[:, ~live].abs().sum()) == 0.0
    assert float(PT[~keys].abs().sum()) == 0.0  # padding rows and keys: P = dS = 0
    # the oracle's gradients of the group (its heads as query heads over one KV group)
    allowed = keys[None, :].expand(Pc, N)
    dq, dk, dv = oracle_bwd.attention_bwd(q.reshape(heads, Pc, 64), k[None], v[None],
                                          do.reshape(heads, Pc, 64), allowed)
    got = {"dq": (dS @ k).reshape(heads, Pc, 64), "dk": dS.T @ q, "dv": PT @ do}
    want = {"dq": dq, "dk": dk[0], "dv": dv[0]}
    for name in got:
        w = want[name].clone()
        if name == "dq":
            w[~live.reshape(heads, Pc)] = 0.0
        rel = float((got[name] - w).norm() / w.norm())
        assert rel < 1e-2, (name, rel)


def test_training_profile_counts_every_kind():
    """fd_train_profile_*: one profiled step brackets launches of every kernel kind; a second
    collect returns nothing (the events were released); the profiled step's gradients equal an
    unprofiled step's bits."""
    cfg = synth.PRESETS["tiny_rt"]
    w, z = synth.make_weights(cfg), synth.make_latents(cfg)
    x = synth.make_target_pixels(cfg, min_abs=0.3)
    W = fdp.Weights(cfg, fdp.pack_blob(cfg, w))
    tr = fdp.Trainer(cfg, W, len(z))
    lat = torch.from_numpy(np.ascontiguousarray(np.stack(z))).cuda()
    tgt = torch.from_numpy(np.ascontiguousarray(np.stack(x))).cuda()
    loss = torch.zeros(1, device="cuda")
    plain = torch.zeros(tr.grad_elems, device="cuda")
    tr.step(lat, tgt, loss, plain)
    grads = torch.zeros(tr.grad_elems, device="cuda")
    tr.profile(True)
    tr.step(lat, tgt, loss, grads)
    prof = tr.profile_collect()
    tr.profile(False)
    assert set(prof) == set(fdp.TRAIN_KINDS)
    for k, (n, ms) in prof.items():
        assert n > 0 and ms > 0, (k, n, ms)
    assert all(v == (0, 0.0) for v in tr.profile_collect().values())
    assert torch.equal(grads, plain)
    tr.close()
    W.close()


@pytest.mark.parametrize("lat_h,lat_w,chunks,window,r_t,heads,groups,qk", [
    (2, 2, 2, 2, 1, 2, 2, False),     # one token per frame (127 padding keys), one head per group
    (16, 16, 1, 1, 1, 2, 1, False),   # 64 tokens, a single chunk
    (16, 32, 3, 2, 1, 4, 1, True),    # 128 tokens: no padding rows; all heads on one group
    (6, 86, 3, 3, 2, 4, 2, False),    # 129 tokens: one token in the second tile; two refined frames
    (30, 34, 2, 4, 4, 2, 2, False),   # 255 tokens, window longer than the clip, four frames
])
def test_attention_backward_tiles(lat_h, lat_w, chunks, window, r_t, heads, groups, qk):
    """The step's fused attention backward at the edges of its 128-row query and key tiles, of
    its windows and of its head groups, through every parameter's gradient (the bars above)."""
    cfg = synth.FDConfig(latent_h=lat_h, latent_w=lat_w, patch=2, hidden=64 * heads, heads=heads,
                         kv_groups=groups, n_blocks=1, n_refine=1 if r_t > 1 else 0,
                         window=window, r_t=r_t, qk_norm=qk, chunks=chunks, name="tiles")
    w, z = synth.make_weights(cfg), synth.make_latents(cfg)
    x = synth.make_target_pixels(cfg, min_abs=0.3)
    loss_ref, g_ref = training_step_explicit(cfg, w, z, x)
    loss, flat = gpu_step(cfg, w, z, x)
    assert abs(loss - loss_ref) <= LOSS_REL * abs(loss_ref)
    for k, g in split(cfg, flat).items():
        ref = g_ref[k].reshape(g.shape)
        assert torch.isfinite(g).all(), k
        # the gradients of Q and K rows vanish where a query sees one key (P = 1): held against
        # the tensor's own scale plus fp32 noise of the whole step
        err, scale = float((g - ref).norm()), float(ref.norm())
        assert err <= GRAD_REL * scale + 1e-6, (k, err, scale)


def test_qkv_slots_past_one_block():
    """Heads and KV groups of more slots (12 + 2 x 12) than one block of the QKV kernels takes."""
    test_attention_backward_tiles(6, 10, 2, 2, 1, 12, 12, True)


@pytest.mark.parametrize("M,D,off", [
    (1, 64, 0), (17, 64, 0),           # fewer rows than the thread groups of a narrow D
    (5, 33, 0), (16, 1025, 0),         # D no multiple of 4
    (33, 100, 0), (33, 100, 1),        # a multiple; the same off 16 bytes
])
def test_rmsnorm_backward_widths_and_alignments(M, D, off):
    """fd_op_rmsnorm_bwd's vector and scalar columns (bound as in test_rmsnorm_backward_kernel)."""
    from oracle.backward import rms_norm_bwd
    from helpers import randn

    def place(a):  # `off` floats into a buffer
        t = torch.empty(a.size + off, device="cuda")[off:].view(a.shape)
        t.copy_(torch.from_numpy(a))
        return t
    x, g, dy = randn((M, D), M + D, 2.0), 1 + randn((D,), M + D + 1, 0.02), randn((M, D), M + D + 2)
    dx, dg = place(np.zeros((M, D), np.float32)), torch.empty(D, device="cuda")
    fdp.op_rmsnorm_bwd(place(x), torch.from_numpy(g).cuda(), place(dy), 1e-6, dx, dg)
    torch.cuda.synchronize()
    want = rms_norm_bwd(torch.from_numpy(x).double(), torch.from_numpy(g).double(), 1e-6,
                        torch.from_numpy(dy).double())
    for got, ref in zip((dx, dg), want):
        assert float((got.cpu().double() - ref).abs().max()) < 2e-5 * float(ref.abs().max())


@pytest.mark.parametrize("n,off", [(3, 0), (4096, 0), (4096, 1), (4098, 0)])
def test_gelu_backward_lengths_and_alignments(n, off):
    """fd_op_gelu_bwd's vector and scalar forms give the oracle's values (bounds as in
    test_gelu_backward_kernel)."""
    from oracle.backward import gelu_bwd
    z = torch.linspace(-9, 9, n, dtype=torch.float32)
    da = torch.cos(torch.arange(n, dtype=torch.float32))
    zd, dad, dz = (torch.zeros(n + off, device="cuda")[off:] for _ in range(3))
    dz16 = torch.zeros(n, dtype=torch.bfloat16, device="cuda")
    zd.copy_(z)
    dad.copy_(da)
    fdp.op_gelu_bwd(zd, dad, dz, dz16)
    torch.cuda.synchronize()
    assert float((dz.cpu().double() - gelu_bwd(z.double(), da.double())).abs().max()) < 2e-6
    assert torch.equal(dz16.cpu(), dz.cpu().to(torch.bfloat16))


@pytest.mark.parametrize("frames,gh,gw,C,rs", [(2, 3, 5, 3, 6), (1, 1, 1, 1, 4), (3, 5, 7, 3, 20)])
def test_l1_pixel_backward_pixel_rows(frames, gh, gw, C, rs):
    """fd_op_l1_pixel_bwd with pixel rows that are no multiple of 4 (element by element), with a
    single token, and with more than 1024 columns (two strips). Loss bound: fp32 terms summed in a
    tree and in fp64."""
    from oracle.backward import l1_bwd, pixel_shuffle_bwd
    from helpers import randn
    F = randn((frames * gh * gw, C * rs * rs), 5, 0.3)
    x = randn((C, frames, gh * rs, gw * rs), 6, 0.3)
    dF, loss = torch.empty(F.shape, device="cuda"), torch.zeros(1, device="cuda")
    fdp.op_l1_pixel_bwd(torch.from_numpy(F).cuda(), torch.from_numpy(x).cuda(), frames, gh, gw,
                        C, rs, dF, loss)
    torch.cuda.synchronize()
    pix = oracle.pixel_shuffle(torch.from_numpy(F).double(), frames, gh, gw, C, rs)
    want = float((pix - torch.from_numpy(x).double()).abs().mean())
    assert abs(float(loss.item()) - want) <= 1e-6 * want
    want_dF = pixel_shuffle_bwd(l1_bwd(pix, x, pix.numel()), frames, gh, gw, C, rs)
    assert float((dF.cpu().double() - want_dF).abs().max()) <= 1e-7 / pix.numel()


@pytest.mark.parametrize("T,N,G,W,frames,L,hs", [
    (2, 2, 2, 2, 1, 2, 1),      # two tokens per frame (126 padding rows), one head per group
    (3, 4, 1, 2, 1, 128, 4),    # no padding; every head of a chunk in one accumulator chain
    (3, 4, 2, 3, 2, 129, 2),    # one token in a frame's second tile; two frames per chunk
    (3, 4, 2, 3, 2, 129, 1),    # the same, each head its own chain
    (2, 2, 1, 4, 4, 255, 2),    # one padding row per frame; window longer than the clip
    (5, 6, 1, 2, 1, 100, 3),    # two chains per chunk and group
    (4, 8, 1, 4, 1, 200, 8),    # chains of more blocks than the load ring holds
])
def test_attention_backward_kernels(T, N, G, W, frames, L, hs):
    """fd_op_attention_bwd, the step's dQ and dK / dV launches, against oracle.attention_bwd in fp64,
    each tensor by itself. Bar: the kernels round P and dS to bf16 and do the rest in fp32, so
    1.5 times the movement that these two roundings alone cause in fp64, plus 1e-4 (64-term fp32
    sums, exponents below 8: a few 1e-6 per score). Padding rows get exact zeros."""
    from helpers import bf16_values, randn
    Lp = (L + 127) // 128 * 128
    Pc, hpg = frames * Lp, N // G
    M = T * Pc
    pos = torch.arange(M)
    live, chunk = pos % Lp < L, pos // Pc
    allowed = live[None] & (chunk[None] <= chunk[:, None]) & (chunk[None] > chunk[:, None] - W)
    t = lambda shape, i: torch.from_numpy(bf16_values(randn(shape, 1000 * T + 10 * L + i))).double()
    q, k, v, do = t((N, M, 64), 0), t((G, M, 64), 1), t((G, M, 64), 2), t((N, M, 64), 3)
    do[:, ~live] = 0.0
    kk, vv = k.repeat_interleave(hpg, 0), v.repeat_interleave(hpg, 0)
    s = (q @ kk.transpose(1, 2) / 8.0).masked_fill(~allowed, float("-inf"))
    lse = torch.logsumexp(s, -1)
    p = torch.softmax(s, -1)
    delta = (do * (p @ vv)).sum(-1)
    want = dict(zip(("dq", "dk", "dv"), oracle_bwd.attention_bwd(q, k, v, do, allowed)))
    # the movement of the bf16 P and dS
    bf = lambda x: x.to(torch.bfloat16).double()
    ds = bf(p * (do @ vv.transpose(1, 2) - delta[..., None]) / 8.0)
    group = lambda x: x.reshape(G, hpg, M, 64).sum(1)
    moved = {"dq": ds @ kk, "dk": group(ds.transpose(1, 2) @ q),
             "dv": group(bf(p).transpose(1, 2) @ do)}
    rows = lambda x: x.reshape(N, T, Pc, *x.shape[2:]).transpose(0, 1).contiguous().cuda()
    lse[:, ~live] = float("inf")
    got = {"dq": torch.full((T, N, Pc, 64), float("nan"), device="cuda"),
           "dk": torch.full((G, M, 64), float("nan"), device="cuda"),
           "dv": torch.full((G, M, 64), float("nan"), device="cuda")}
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    fdp.op_attention_bwd(rows(q.bfloat16()), rows(do.bfloat16()), k.bfloat16().cuda(),
                         v.bfloat16().cuda(), rows(lse.float()), rows(delta.float()), W, Lp, L, hs,
                         got["dq"], got["dk"], got["dv"], err=err)
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    got["dq"] = got["dq"].transpose(0, 1).reshape(N, M, 64)
    for name, x in got.items():
        x, ref = x.cpu().double(), want[name]
        assert float(x[:, ~live].abs().sum()) == 0.0, name
        bar = 1.5 * float((moved[name] - ref).norm()) + 1e-4 * float(ref.norm())
        assert float((x - ref).norm()) <= bar, (name, float((x - ref).norm()), bar)


@pytest.mark.parametrize("lat_h,lat_w,chunks,window,r_t,heads,groups,qk", [
    (16, 16, 1, 1, 1, 2, 1, False), (16, 32, 3, 2, 1, 4, 1, True), (6, 86, 3, 3, 2, 4, 2, False),
    (30, 34, 2, 4, 4, 2, 2, False), (20, 26, 5, 3, 4, 4, 2, False),
])
def test_query_key_and_value_gradients_each_by_itself(lat_h, lat_w, chunks, window, r_t, heads,
                                                      groups, qk):
    """The step's gradients that dQ, dK and dV reach, each held to its own norm: the Q, K and V rows
    of the QKV weight and bias (V's are several times larger than Q's and K's, and would hide them)
    and the gains. Bars: with every matrix operand of the step rounded to bf16 / fp16 (forward, and
    dY, dO, P, dS backward) the fp64 oracle moves these by at most 0.71 % on these clips, K's bias
    rows by 2.1 % (sums of a key's dS over all queries nearly cancel); 3 times that."""
    cfg = synth.FDConfig(latent_h=lat_h, latent_w=lat_w, patch=2, hidden=64 * heads, heads=heads,
                         kv_groups=groups, n_blocks=1, n_refine=1 if r_t > 1 else 0,
                         window=window, r_t=r_t, qk_norm=qk, chunks=chunks, name="qkv")
    w, z = synth.make_weights(cfg), synth.make_latents(cfg)
    x = synth.make_target_pixels(cfg, min_abs=0.3)
    _, g_ref = training_step_explicit(cfg, w, z, x)
    got = split(cfg, gpu_step(cfg, w, z, x)[1])
    nq, nk = 64 * heads, 64 * groups
    for name, ref in g_ref.items():
        if "qkv." not in name and not name.endswith("norm.g"):
            continue
        parts = {"": slice(None)} if "qkv." not in name else {
            "Q": slice(0, nq), "K": slice(nq, nq + nk), "V": slice(nq + nk, None)}
        for part, rows in parts.items():
            a, b = got[name][rows], ref.reshape(got[name].shape)[rows]
            bar = 6.3e-2 if name.endswith("qkv.b") and part == "K" else 2.1e-2
            assert float((a - b).norm()) <= bar * float(b.norm()), (name, part)
