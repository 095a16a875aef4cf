"""The work that a calibration or deployment program has this library do, as measurable cases.

Every case is a dict of plain values with a "kind":

  step       one linear's calibration step: (8-bit activations,) forward at a schedule point, the
             reconstruction loss against the teacher output, the backward into the activations and
             the three factors, and AdamW on the factors
  block      one step of a whole decoder block as the reconstruction window (all seven linears)
  moe        forward, loss and backward of the stacked experts of a mixture-of-experts layer
  decode     the deployed 2-bit layers of consecutive decoder blocks for a few token rows: one call
             per set of independent layers, or one staged call for the chain
  attention  causal grouped-query attention, forward and backward
  layers     what lies between a block's linears and its attention: norms with the residual, head
             norms, rotary embedding, SwiGLU and the block output with its loss, forward and backward
  weights    group statistics at the start of a layer's calibration and its hard pack at the end

Sizes are those of the decoder shapes in synthetic.py and generic odd ones around them.  Inputs come
from the seed alone: normal weights, activations that are normal with a few outlier channels or
Student-t distributed, factors a little off the identity.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2606_26650_gb300 import block as BK
from paper_2606_26650_gb300 import catq as C

BF, F32, F64 = torch.bfloat16, torch.float32, torch.float64

# hidden size, query columns, key/value columns, MLP width
SHAPES = {"1p7b": (2048, 2048, 1024, 6144), "8b": (4096, 4096, 1024, 14336), "14b": (5120, 5120, 1024, 17408)}

PHASES = {"soft": C.PHASE_SOFT, "hard": C.PHASE_HARD}


def listed():
    return [
        # The smallest calls: the single fp32 linear of 512 x 512 (8 sequences of 128 tokens,
        # channel-wise groups, TWN threshold), where launches and latency count.
        dict(name="step_fp32_512", kind="step", dtype="f32", M=1024, N=512, K=512, g=512, thr="twn07", phase="soft",
             s=30.0, recon=0, a8=False, fused=False, x="normal"),
        # A key/value projection on a ragged handful of sequences early in the soft stage (low
        # sharpness, two-term transition function).
        dict(name="step_kv_ragged", kind="step", dtype="bf16", M=300, N=1024, K=2048, g=128, thr="half",
             phase="soft", s=3.75, recon=0, a8=False, fused=False, x="outlier"),
        # A down projection of the 1.7B shape late in calibration (hard stage) in the
        # weight-and-activation setting (8-bit tokens), an odd number of rows.
        dict(name="step_down_a8_hard", kind="step", dtype="bf16", M=1999, N=2048, K=6144, g=128, thr="half",
             phase="hard", s=30.0, recon=0, a8=True, fused=False, x="outlier"),
        # The ordinary large step: gate_proj of the 8B shape on 4 x 2048 tokens.
        dict(name="step_gate_8b", kind="step", dtype="bf16", M=8192, N=14336, K=4096, g=128, thr="half",
             phase="soft", s=30.0, recon=0, a8=False, fused=False, x="student"),
        # The whole window of the 1.7B block with its query/key norms, 4 x 2048 tokens.
        dict(name="block_1p7b", kind="block", H=2048, nh=16, nkv=8, d=128, I=6144, B=4, S=2048, g=128, phase="soft",
             s=30.0, qk_norm=True),
        # The largest: 128 experts' gate projection, 8192 tokens routed to 8 experts each.
        dict(name="moe_gate_128", kind="moe", E=128, N=1536, K=4096, tokens=8192, top_k=8, zipf=1.1, g=128,
             phase="soft", s=30.0),
        # One token row through two 8B blocks, four launches a block.
        dict(name="decode_8b_b1", kind="decode", shape="8b", blocks=2, B=1, g=128, mu=False, staged=False),
        # A small batch through four 1.7B blocks as one staged call, scale and offset per 64 weights.
        dict(name="decode_1p7b_b6_staged", kind="decode", shape="1p7b", blocks=4, B=6, g=64, mu=True, staged=True),
        # The 8B block's attention.
        dict(name="attention_8b", kind="attention", B=4, S=2048, nh=32, nkv=8, d=128),
        # 64-wide heads and a sequence length that is no multiple of 128.
        dict(name="attention_d64", kind="attention", B=3, S=1088, nh=12, nkv=4, d=64),
        # The 8B block's memory-bound layers on 4 x 2048 tokens.
        dict(name="layers_8b", kind="layers", T=8192, S=2048, H=4096, I=14336, nh=32, d=128),
        # Statistics and pack of the 14B shape's down projection.
        dict(name="weights_down_14b", kind="weights", N=5120, K=17408, g=128, thr="half", recon=0),
    ]


THR = {"half": C.THR_HALF, "twn07": C.THR_TWN07, "absmean": C.THR_ABSMEAN, "twn": C.THR_TWN_STATIC}


# ------------------------------------------------------------------ drawn cases

def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _mult(v, m, lo):
    return max(lo, v // m * m)


def _draw_step(rng):
    if rng.random() < 0.15:
        g = rng.choice([16, 64, 128])
        return dict(kind="step", dtype="f32", M=_log(rng, 1, 2048), N=_log(rng, 16, 1024), K=g * rng.randint(1, 1024 // g),
                    g=g, thr=rng.choice(["half", "twn07"]), phase="soft", s=rng.choice([7.5, 30.0]), recon=rng.choice([0, 1]),
                    a8=False, fused=False, x="normal")
    g = rng.choice([64, 128, 128, 128, 256])
    N, K = _mult(_log(rng, 64, 14336), 8, 64), _mult(_log(rng, 256, 14336), g, g)
    M = _log(rng, 1, 8192)
    while M * N * K > 8192 * 14336 * 4096:
        M = max(1, M // 2 - 1)
    fused = rng.random() < 0.25
    return dict(kind="step", dtype="bf16", M=M, N=N, K=K, g=g, thr="half", phase=rng.choice(["soft", "soft", "hard"]),
                s=rng.choice([1.875, 7.5, 15.0, 30.0]), recon=int(rng.random() < 0.2), a8=(not fused and rng.random() < 0.2),
                fused=fused, x=rng.choice(["normal", "outlier", "student"]))


def _draw_block(rng):
    d, nkv = 128, rng.choice([2, 4, 8])
    nh = nkv * rng.choice([1, 2, 4])
    H = 128 * rng.randint(4, 20)
    B, S = rng.randint(1, 4), 64 * rng.randint(2, 32)
    while B * S > 4096:
        B = max(1, B - 1)
        S = _mult(S - 64, 64, 64) if B == 1 and S > 4096 else S
    return dict(kind="block", H=H, nh=nh, nkv=nkv, d=d, I=128 * rng.randint(8, 48), B=B, S=S, g=128,
                phase=rng.choice(["soft", "soft", "hard"]), s=30.0, qk_norm=rng.random() < 0.5)


def _draw_moe(rng):
    N, K = rng.choice([(1536, 4096), (4096, 1536), (768, 2048), (1024, 1408)])
    return dict(kind="moe", E=rng.randint(4, 64), N=N, K=K, tokens=_log(rng, 64, 8192), top_k=rng.randint(1, 4),
                zipf=rng.choice([0.0, 0.6, 1.1]), g=128, phase=rng.choice(["soft", "soft", "hard"]), s=30.0)


def _draw_decode(rng):
    staged = rng.random() < 0.35
    shape = rng.choice(["1p7b", "1p7b", "8b", "14b"])
    return dict(kind="decode", shape=shape, blocks=rng.randint(1, 4), B=rng.choice([1, 1, 1, 2, 3, 5, 8, 11]),
                g=rng.choice([64, 128, 128, 256]), mu=rng.random() < 0.3, staged=staged)


def _draw_attention(rng):
    d = rng.choice([64, 128, 128])
    nkv = rng.choice([1, 2, 4, 8])
    S = 64 * _log(rng, 1, 48)
    return dict(kind="attention", B=rng.randint(1, max(1, min(8, 8192 // S))), S=S, nh=nkv * rng.choice([1, 2, 4, 5]),
                nkv=nkv, d=d)


def _draw_layers(rng):
    nh, d = rng.choice([4, 8, 16, 20, 32, 40]), rng.choice([64, 128, 128])
    return dict(kind="layers", T=_log(rng, 1, 8192), S=rng.choice([64, 500, 1024, 2048]), H=8 * _log(rng, 16, 640),
                I=8 * _log(rng, 32, 2176), nh=nh, d=d)


def _draw_weights(rng):
    g = rng.choice([64, 128, 128, 128, 192, 256, 1024])
    return dict(kind="weights", N=_mult(_log(rng, 64, 17408), 8, 64), K=g * max(1, _log(rng, 256, 5120) // g), g=g,
                thr=rng.choice(["half", "half", "twn07", "absmean", "twn"]), recon=int(rng.random() < 0.3))


def draw(rng):
    return rng.choice([_draw_step, _draw_step, _draw_step, _draw_block, _draw_moe, _draw_decode, _draw_decode,
                       _draw_attention, _draw_attention, _draw_layers, _draw_layers, _draw_weights])(rng)


# ------------------------------------------------------------------ inputs

class _Inputs:
    """Seeded tensors on the current GPU."""

    def __init__(self, seed):
        self.dev = torch.device("cuda")
        self.gen = torch.Generator(device=self.dev).manual_seed(int(seed))

    def normal(self, *shape, std=1.0, dtype=BF):
        return torch.randn(*shape, generator=self.gen, device=self.dev, dtype=dtype).mul_(std)

    def uniform(self, n, lo, hi):
        return torch.rand(n, generator=self.gen, device=self.dev).mul_(hi - lo).add_(lo)

    def activations(self, M, K, how, dtype=BF):
        x = torch.randn(M, K, generator=self.gen, device=self.dev)
        if how == "student":  # four degrees of freedom
            v = torch.zeros(M, K, device=self.dev)
            for _ in range(4):
                v.add_(torch.randn(M, K, generator=self.gen, device=self.dev).square_())
            x.div_(v.div_(4).sqrt_())
        elif how == "outlier":  # 1 % of the channels x 30
            n = max(1, K // 100)
            x[:, torch.randperm(K, generator=self.gen, device=self.dev)[:n]] *= 30.0
        return x.to(dtype)

    def factors(self, G):
        return self.uniform(G, -0.1, 0.1), self.uniform(G, 0.8, 1.2), self.uniform(G, 0.8, 1.2)

    def empty(self, *shape, dtype=BF):
        return torch.empty(*shape, device=self.dev, dtype=dtype)


def _sched(case):
    return C.schedule(PHASES[case["phase"]], case["s"])


# ------------------------------------------------------------------ step

def _step_inputs(c, inp):
    dt = F32 if c["dtype"] == "f32" else BF
    N, K, g = c["N"], c["K"], c["g"]
    W = inp.normal(N, K, std=0.02, dtype=dt)
    X = inp.activations(c["M"], K, c["x"], dt)
    return W, X, X @ W.t(), inp.factors(N * K // g)


# The last hundred of the schedule's updates: a learning rate that moves the factors little.
_UPDATES = 60 * 171


def _prepare_step(c, seed):
    inp = _Inputs(seed)
    W, X, Yt, fac = _step_inputs(c, inp)
    layer = C.Layer.create(W, c["g"], *fac, recon=c["recon"])
    C.catq_group_stats(layer, THR[c["thr"]])
    M, G, dt = c["M"], layer.G, X.dtype
    st = dict(layer=layer, X=X, Yt=Yt, sched=_sched(c), hp=C.adamw(), t=0,
              lr=C.catq_linear_decay_lr(1e-3, _UPDATES - 100, _UPDATES),
              Y=torch.empty_like(Yt), dY=torch.empty_like(Yt), dX=torch.empty_like(X), loss=inp.empty(1, dtype=F32),
              grads=[inp.empty(G, dtype=F32) for _ in range(3)], moments=torch.zeros(6 * G, device=inp.dev),
              ws=C.workspace(C.catq_bwd_workspace_bytes(layer, M), inp.dev))
    if c["fused"]:
        st["loss_ws"] = C.workspace(C.catq_fwd_loss_workspace_bytes(layer, M), inp.dev)
    else:
        st["loss_ws"] = C.workspace(C.catq_recon_loss_workspace_bytes(Yt.numel()), inp.dev)
    if c["a8"]:
        st.update(codes=torch.empty_like(X), scale=inp.empty(M, dtype=F32), Xq=torch.empty_like(X), )
    return st


def _run_step(c, st):
    layer, sched, X = st["layer"], st["sched"], st["X"]
    out = {}
    if c["fused"]:
        C.catq_soft_ternary_linear_fwd_loss(layer, sched, X, st["Yt"], st["loss"], st["dY"], workspace=st["loss_ws"])
    else:
        if c["a8"]:
            C.catq_act_quant_a8(X, st["codes"], st["scale"], st["Xq"])
            C.catq_soft_ternary_linear_fwd_ex(layer, sched, st["codes"], st["Y"], x_row_scale=st["scale"])
            X = st["Xq"]
            out.update(codes=st["codes"], scale=st["scale"])
        else:
            C.catq_soft_ternary_linear_fwd(layer, sched, X, st["Y"])
        C.catq_recon_loss(st["Y"], st["Yt"], st["loss"], st["dY"], st["loss_ws"])
        out["Y"] = st["Y"]
    C.catq_soft_ternary_linear_bwd(layer, sched, X, st["dY"], st["dX"], *st["grads"], st["ws"])
    st["t"] += 1
    C.catq_factor_adamw_step(layer.d_mu, layer.d_alpha, layer.d_delta, *st["grads"], st["moments"], st["hp"], st["t"],
                             st["lr"])
    out.update(loss=st["loss"], dY=st["dY"], dX=st["dX"], grads=st["grads"],
               factors=[layer.d_mu, layer.d_alpha, layer.d_delta], moments=st["moments"])
    return out


def _stats64(W, g, thr):
    """mu0, alpha0, Delta0 of each group, [G, 1] in 64 bits."""
    w = W.double().reshape(-1, g)
    mag = w.abs().mean(1, keepdim=True)
    half = torch.full_like(mag, 0.5)
    if thr == "absmean":
        return torch.zeros_like(mag), mag, half
    if thr == "twn":
        over = (w.abs() > 0.7 * mag)
        a = (w.abs() * over).sum(1, keepdim=True) / over.sum(1, keepdim=True).clamp_min(1)
        return torch.zeros_like(mag), a, torch.where(a > 0, 0.7 * mag / a, half)
    mu = w.mean(1, keepdim=True)
    a = (w - mu).abs().mean(1, keepdim=True)
    return mu, a, torch.where(a > 0, 0.7 * mag / a, half) if thr == "twn07" else half


def _wq64(W, g, stats, fac, phase, s, recon=0):
    """The quantized weight in 64 bits, differentiable in the factors; the hard stage uses the
    hard codes forward and the soft transition's derivatives backward."""
    mu0, a0, D0 = stats
    dmu, dal, ddl = (f.reshape(-1, 1) for f in fac)
    mu, alpha, delta = mu0 + dmu * a0, dal * a0, ddl * D0
    what = (W.double().reshape(-1, g) - mu) / alpha
    T = (torch.tanh(s * (what - delta)) + torch.tanh(s * (what + delta))) / (2 * math.tanh(s))
    if phase == "hard":
        with torch.no_grad():
            gap = torch.sign(what) * (what.abs() > delta) - T
        T = T + gap
    wq = alpha * T + mu if recon else alpha * T
    return wq.reshape(W.shape)


def _linear_step64(c, W, X, Yt, fac, count):
    """Y, squared error, dY, dX and factor gradients of one linear with its rows, in 64 bits."""
    fac = [f.double().requires_grad_() for f in fac]
    wq = _wq64(W, c["g"], _stats64(W, c["g"], c.get("thr", "half")), fac, c["phase"], c["s"], c.get("recon", 0))
    with torch.no_grad():
        Y = X @ wq.t()
        d = Y - Yt.double()
        dY = d * (2.0 / count)
        dX = dY @ wq
        G = dY.t() @ X
    grads = torch.autograd.grad(wq, fac, G)
    return Y, d.square().sum(), dY, dX, grads


def _exact_step(c, seed):
    W, X, Yt, fac = _step_inputs(c, _Inputs(seed))
    out, x64 = {}, X.double()
    if c["a8"]:
        x32 = X.float()
        scale = x32.abs().amax(1, keepdim=True) / 127.0
        codes = torch.where(scale > 0, torch.round(x32 / scale).clamp(-127, 127), torch.zeros_like(x32))
        x64 = codes.double() * scale.double()
        out.update(codes=codes.double(), scale=scale.double().reshape(-1))
    Y, sq, dY, dX, grads = _linear_step64(c, W, x64, Yt, fac, Yt.numel())
    if not c["fused"]:
        out["Y"] = Y
    lr, new, m, v = 1e-3 * (1.0 - (_UPDATES - 100) / _UPDATES), [], [], []
    for i, (p, g) in enumerate(zip(fac, grads)):
        p = p.double() - lr * g / (g.abs() + 1e-8)
        new.append(p.clamp(-1 + 1e-4, 1 - 1e-4) if i == 0 else p.clamp_min(1e-4))
        m.append(0.1 * g)
        v.append(0.001 * g * g)
    out.update(loss=(sq / Yt.numel()).reshape(1), dY=dY, dX=dX, grads=list(grads), factors=new, moments=torch.cat(m + v))
    return out


def _work_step(c):
    e = 4 if c["dtype"] == "f32" else 2
    M, N, K = c["M"], c["N"], c["K"]
    G = N * K // c["g"]
    y_out = M * N * e * (1 if c["fused"] else 2)
    return {"bytes": e * (N * K + 2 * M * K + M * N) + y_out + (2 * M * K * e if c["a8"] else 0) + 4 * G * (3 + 12 + 12),
            "flops": 6.0 * M * N * K}


# ------------------------------------------------------------------ block

def _block_inputs(c, inp):
    shape = BK.BlockShape(H=c["H"], n_heads=c["nh"], n_kv_heads=c["nkv"], d=c["d"], I=c["I"], B=c["B"], S=c["S"],
                          base=1e6 if c["qk_norm"] else 5e5)
    W = {n: inp.normal(*nk, std=0.02) for n, nk in shape.linear_shapes().items()}
    fac = {n: inp.factors(w.numel() // c["g"]) for n, w in W.items()}
    x = inp.activations(shape.T, c["H"], "normal", F32)
    gammas = [inp.uniform(c["H"], 0.7, 1.3) for _ in range(2)]
    heads = [inp.uniform(c["d"], 0.7, 1.3) for _ in range(2)] if c["qk_norm"] else [None, None]
    return shape, W, fac, x, gammas, heads


def _norm(x, gamma, eps):
    return gamma * x * torch.rsqrt(x.square().mean(-1, keepdim=True) + eps)


def _rope(x, S, base, inverse=False):
    """x [T, heads, d], half-split pairs."""
    T, _, d = x.shape
    pos = (torch.arange(T, device=x.device) % S).double()
    ang = pos[:, None] * torch.pow(torch.tensor(base, device=x.device, dtype=F64),
                                   -2.0 * torch.arange(d // 2, device=x.device).double() / d)
    cs, sn = ang.cos().to(x.dtype)[:, None], ang.sin().to(x.dtype)[:, None]
    if inverse:
        sn = -sn
    a, b = x[..., : d // 2], x[..., d // 2:]
    return torch.cat([a * cs - b * sn, a * sn + b * cs], -1)


def _attend(q, k, v):
    """q [h, S, d] against k, v [h, S, d], causal; output and log-sum-exp."""
    S = q.shape[1]
    s = (q @ k.transpose(1, 2)) / math.sqrt(q.shape[2])
    s = s.masked_fill(torch.ones(S, S, dtype=torch.bool, device=q.device).triu(1), -math.inf)
    lse = torch.logsumexp(s, -1)
    return torch.exp(s - lse[..., None]) @ v, lse


def _plain_block(shape, W, x, gammas, heads):
    """The block's output with weights W in their own precision."""
    T, rep = shape.T, shape.n_heads // shape.n_kv_heads
    z = _norm(x, gammas[0], shape.eps)
    q = (z @ W["q_proj"].t()).view(T, shape.n_heads, shape.d)
    k = (z @ W["k_proj"].t()).view(T, shape.n_kv_heads, shape.d)
    v = (z @ W["v_proj"].t()).view(T, shape.n_kv_heads, shape.d)
    if heads[0] is not None:
        q, k = _norm(q, heads[0], shape.eps), _norm(k, heads[1], shape.eps)
    q, k = _rope(q, shape.S, shape.base), _rope(k, shape.S, shape.base)
    rows = []
    for b in range(shape.B):
        at = slice(b * shape.S, (b + 1) * shape.S)
        o, _ = _attend(q[at].transpose(0, 1), k[at].transpose(0, 1).repeat_interleave(rep, 0),
                       v[at].transpose(0, 1).repeat_interleave(rep, 0))
        rows.append(o.transpose(0, 1).reshape(shape.S, -1))
    h = x + torch.cat(rows) @ W["o_proj"].t()
    z = _norm(h, gammas[1], shape.eps)
    m = torch.nn.functional.silu(z @ W["gate_proj"].t()) * (z @ W["up_proj"].t())
    return h + m @ W["down_proj"].t()


def _prepare_block(c, seed):
    inp = _Inputs(seed)
    shape, W, fac, x, gammas, heads = _block_inputs(c, inp)
    blk = BK.Block(shape, W, *gammas, c["g"], factors=fac, q_norm=heads[0], k_norm=heads[1])
    with torch.no_grad():
        ref = _plain_block(shape, {n: w.float() for n, w in W.items()}, x, gammas, heads)
    grads = {n: [inp.empty(blk.layers[n].G, dtype=F32) for _ in range(3)] for n in BK.LINEARS}
    return dict(blk=blk, x=x, ref=ref, sched=_sched(c), loss=inp.empty(1, dtype=F32), grads=grads,
                out=torch.empty_like(x))


def _run_block(c, st):
    st["blk"].step(st["x"], st["ref"], st["sched"], st["loss"], st["grads"], out=st["out"])
    return dict(out=st["out"], loss=st["loss"], grads=st["grads"])


def _exact_block(c, seed):
    shape, W, fac, x, gammas, heads = _block_inputs(c, _Inputs(seed))
    with torch.no_grad():
        ref = _plain_block(shape, {n: w.float() for n, w in W.items()}, x, gammas, heads).double()
    fac = {n: [f.double().requires_grad_() for f in v] for n, v in fac.items()}
    wq = {n: _wq64(W[n], c["g"], _stats64(W[n], c["g"], "half"), fac[n], c["phase"], c["s"]) for n in BK.LINEARS}
    out = _plain_block(shape, wq, x.double(), [g.double() for g in gammas], [h if h is None else h.double() for h in heads])
    loss = (out - ref).square().mean()
    loss.backward()
    return dict(out=out.detach(), loss=loss.detach().reshape(1), grads={n: [f.grad for f in fac[n]] for n in BK.LINEARS})


def _work_block(c):
    shape = BK.BlockShape(H=c["H"], n_heads=c["nh"], n_kv_heads=c["nkv"], d=c["d"], I=c["I"], B=c["B"], S=c["S"])
    w = sum(n * k for n, k in shape.linear_shapes().values())
    return {"bytes": 2 * w + 24 * w // c["g"] + 12 * w // c["g"] + 12 * shape.T * c["H"],
            "flops": shape.linear_flops() + shape.attention_flops()}


# ------------------------------------------------------------------ mixture of experts

def _moe_inputs(c, seed, inp):
    E, N, K = c["E"], c["N"], c["K"]
    r = np.random.default_rng(int(seed))
    score = -c["zipf"] * np.log(np.arange(1, E + 1)) + r.gumbel(size=(c["tokens"], E))
    choice = np.argpartition(-score, min(c["top_k"], E) - 1, axis=1)[:, :c["top_k"]]
    off = [0] + [int(v) for v in np.cumsum(np.bincount(choice.reshape(-1), minlength=E))]
    W = inp.normal(E, N, K, std=0.02)
    X = inp.activations(off[-1], K, "normal")
    Yt = torch.empty(off[-1], N, device=inp.dev, dtype=BF)
    for e in range(E):
        Yt[off[e]:off[e + 1]] = X[off[e]:off[e + 1]] @ W[e].t()
    return off, W, X, Yt, inp.factors(E * N * K // c["g"])


def _prepare_moe(c, seed):
    inp = _Inputs(seed)
    off, W, X, Yt, fac = _moe_inputs(c, seed, inp)
    layer = C.GroupedLayer.create(W, c["g"], *fac)
    C.catq_group_stats(layer.dense)
    return dict(layer=layer, off=off, X=X, Yt=Yt, sched=_sched(c), Y=torch.empty_like(Yt), dY=torch.empty_like(Yt),
                dX=torch.empty_like(X), loss=inp.empty(1, dtype=F32),
                grads=[inp.empty(layer.dense.G, dtype=F32) for _ in range(3)],
                ws=C.workspace(C.catq_grouped_bwd_workspace_bytes(layer, off), inp.dev),
                loss_ws=C.workspace(C.catq_recon_loss_workspace_bytes(Yt.numel()), inp.dev))


def _run_moe(c, st):
    C.catq_grouped_soft_ternary_linear_fwd(st["layer"], st["sched"], st["X"], st["off"], st["Y"])
    C.catq_recon_loss(st["Y"], st["Yt"], st["loss"], st["dY"], st["loss_ws"])
    C.catq_grouped_soft_ternary_linear_bwd(st["layer"], st["sched"], st["X"], st["dY"], st["off"], st["dX"],
                                           *st["grads"], workspace=st["ws"])
    return dict(Y=st["Y"], loss=st["loss"], dY=st["dY"], dX=st["dX"], grads=st["grads"])


def _exact_moe(c, seed):
    off, W, X, Yt, fac = _moe_inputs(c, seed, _Inputs(seed))
    per, sq, parts = W[0].numel() // c["g"], 0.0, []
    for e in range(c["E"]):
        at = slice(off[e], off[e + 1])
        parts.append(_linear_step64(c, W[e], X[at].double(), Yt[at], [f[e * per:(e + 1) * per] for f in fac], Yt.numel()))
        sq = sq + parts[-1][1]
    cat = [torch.cat([p[i] for p in parts]) for i in (0, 2, 3)]
    return dict(Y=cat[0], loss=(sq / Yt.numel()).reshape(1), dY=cat[1], dX=cat[2],
                grads=[torch.cat([p[4][i] for p in parts]) for i in range(3)])


def _work_moe(c):
    R, E, N, K = c["tokens"] * min(c["top_k"], c["E"]), c["E"], c["N"], c["K"]
    return {"bytes": 2 * (E * N * K + 2 * R * K + 3 * R * N) + 36 * E * N * K // c["g"], "flops": 6.0 * R * N * K}


# ------------------------------------------------------------------ decode

def _decode_layers(c):
    """(name, N, K, source, stage in its block): the source is the layer whose output stands for
    what the block's attention or activation makes of it."""
    H, Q, KV, I = SHAPES[c["shape"]]
    return [("q", Q, H, "in", 0), ("k", KV, H, "in", 0), ("v", KV, H, "in", 0), ("o", H, Q, "q", 1),
            ("gate", I, H, "o", 2), ("up", I, H, "o", 2), ("down", H, I, "gate", 3)]


def _decode_inputs(c, inp):
    H, g = SHAPES[c["shape"]][0], c["g"]
    x = inp.activations(c["B"], H, "normal")
    layers = []
    for _ in range(c["blocks"]):
        for _, N, K, _, _ in _decode_layers(c):
            # codes as the thresholds of a normal weight give them: about 31 % zeros
            u = torch.rand(N * K, generator=inp.gen, device=inp.dev)
            code = (u > 0.345).to(torch.uint8) + (u > 0.655).to(torch.uint8)
            q = code.view(-1, 4)
            packed = q[:, 0] | (q[:, 1] << 2) | (q[:, 2] << 4) | (q[:, 3] << 6)
            a0 = 1.2 / math.sqrt(K)
            layers.append((packed, inp.uniform(N * K // g, 0.8 * a0, 1.2 * a0),
                           inp.uniform(N * K // g, -0.1 * a0, 0.1 * a0) if c["mu"] else None))
    return x, layers


def _prepare_decode(c, seed):
    inp = _Inputs(seed)
    x, weights = _decode_inputs(c, inp)
    calls, stages, chain, outs = [], [], [], []
    src = x
    for b in range(c["blocks"]):
        made = {"in": src}
        for i, (name, N, K, frm, stage) in enumerate(_decode_layers(c)):
            codes, alpha, mu = weights[7 * b + i]
            y = inp.empty(c["B"], N)
            made[name] = y
            outs.append(y)
            chain.append((codes, alpha, N, K, made[frm], y, mu))
            stages.append(4 * b + stage)
        src = made["down"]
    for s in range(4 * c["blocks"]):
        calls.append([layer for layer, at in zip(chain, stages) if at == s])
    sync = torch.zeros(C.catq_ternary_infer_sync_bytes(), dtype=torch.uint8, device=inp.dev)
    return dict(calls=calls, chain=chain, stages=stages, sync=sync, outs=outs)


def _run_decode(c, st):
    if c["staged"]:
        C.catq_ternary_infer_staged(st["chain"], st["stages"], c["g"], st["sync"])
    else:
        for layers in st["calls"]:
            C.catq_ternary_infer_batched(layers, c["g"])
    return st["outs"]


def _exact_decode(c, seed):
    x, weights = _decode_inputs(c, _Inputs(seed))
    src, outs, g = x.double(), [], c["g"]
    for b in range(c["blocks"]):
        made = {"in": src}
        for i, (name, N, K, frm, _) in enumerate(_decode_layers(c)):
            packed, alpha, mu = weights[7 * b + i]
            code = torch.stack([(packed >> s) & 3 for s in (0, 2, 4, 6)], 1)
            w = (code.double() - 1).view(-1, g) * alpha.double()[:, None]
            if mu is not None:
                w = w + mu.double()[:, None]
            made[name] = made[frm] @ w.view(N, K).t()
            outs.append(made[name])
        src = made["down"]
    return outs


def _work_decode(c):
    per = sum(N * K for _, N, K, _, _ in _decode_layers(c))
    io = sum(N + K for _, N, K, _, _ in _decode_layers(c))
    return {"bytes": c["blocks"] * (per / 4 + 4 * per / c["g"] * (2 if c["mu"] else 1) + 2 * c["B"] * io),
            "flops": 2.0 * c["B"] * per * c["blocks"]}


# ------------------------------------------------------------------ attention

def _attention_inputs(c, inp):
    T = c["B"] * c["S"]
    q, k, v = (inp.normal(T, n * c["d"]) for n in (c["nh"], c["nkv"], c["nkv"]))
    return q, k, v, inp.normal(T, c["nh"] * c["d"], std=1e-3)


def _prepare_attention(c, seed):
    inp = _Inputs(seed)
    q, k, v, do = _attention_inputs(c, inp)
    rows = c["B"] * c["nh"] * c["S"]
    return dict(q=q, k=k, v=v, do=do, o=torch.empty_like(q), lse=inp.empty(rows, dtype=F32),
                delta=inp.empty(rows, dtype=F32), dq=torch.empty_like(q), dk=torch.empty_like(k), dv=torch.empty_like(v))


def _run_attention(c, st):
    size = (c["B"], c["S"], c["nh"], c["nkv"], c["d"])
    C.catq_attention_fwd(st["q"], st["k"], st["v"], st["o"], st["lse"], *size)
    C.catq_attention_bwd(st["q"], st["k"], st["v"], st["o"], st["do"], st["lse"], st["delta"], st["dq"], st["dk"],
                         st["dv"], *size)
    return {n: st[n] for n in ("o", "lse", "dq", "dk", "dv")}


def _exact_attention(c, seed):
    q, k, v, do = (t.double().view(c["B"], c["S"], -1, c["d"]).transpose(1, 2) for t in _attention_inputs(c, _Inputs(seed)))
    rep, got = c["nh"] // c["nkv"], {n: [] for n in ("o", "lse", "dq", "dk", "dv")}
    for b in range(c["B"]):
        one = {n: [] for n in got}
        for h in range(c["nkv"]):
            qh, kh, vh = (t.detach().requires_grad_() for t in (q[b, h * rep:(h + 1) * rep], k[b, h:h + 1], v[b, h:h + 1]))
            o, lse = _attend(qh, kh, vh)
            o.backward(do[b, h * rep:(h + 1) * rep])
            for n, t in zip(("o", "lse", "dq", "dk", "dv"), (o, lse, qh.grad, kh.grad, vh.grad)):
                one[n].append(t.detach())
        for n, t in one.items():
            t = torch.cat(t)
            got[n].append(t.reshape(-1) if n == "lse" else t.transpose(0, 1).reshape(c["S"], -1))
    return {n: torch.cat(t) for n, t in got.items()}


def _work_attention(c):
    T, d = c["B"] * c["S"], c["d"]
    return {"bytes": 2 * T * d * (4 * c["nh"] + 4 * c["nkv"]) + 4 * T * c["nh"],
            "flops": 7.0 * c["B"] * c["nh"] * c["S"] * c["S"] * d}


# ------------------------------------------------------------------ the layers between

def _layers_inputs(c, inp):
    T, H, I, qd = c["T"], c["H"], c["I"], c["nh"] * c["d"]
    return dict(x=inp.normal(T, H, dtype=F32), branch=inp.normal(T, H, std=0.5), gamma=inp.uniform(H, 0.7, 1.3),
                hgamma=inp.uniform(c["d"], 0.7, 1.3), qp=inp.normal(T, qd), gate=inp.normal(T, I), up=inp.normal(T, I),
                mlp=inp.normal(T, H, std=0.5), ref=inp.normal(T, H, dtype=F32), dm=inp.normal(T, I, std=1e-3),
                dz=inp.normal(T, H, std=1e-3), dz2=inp.normal(T, H, std=1e-3), dres=inp.normal(T, H, std=1e-3),
                dq=inp.normal(T, qd, std=1e-3))


def _prepare_layers(c, seed):
    inp = _Inputs(seed)
    st = _layers_inputs(c, inp)
    T, H, I, qd = c["T"], c["H"], c["I"], c["nh"] * c["d"]
    for n, k in (("z", H), ("dh", H), ("d_out", H), ("q", qd), ("dqp", qd), ("m", I), ("dgate", I), ("dup", I)):
        st[n] = inp.empty(T, k)
    st.update(h=inp.empty(T, H, dtype=F32), out=inp.empty(T, H, dtype=F32), r=inp.empty(T, dtype=F32),
              rq=inp.empty(T * c["nh"], dtype=F32), loss=inp.empty(1, dtype=F32),
              ws=C.workspace(C.catq_recon_loss_workspace_bytes(T * H), inp.dev))
    return st


def _run_layers(c, st):
    d, nh, S = c["d"], c["nh"], c["S"]
    # forward: the head norm and rotary embedding of the queries, the second norm with the
    # attention branch's residual, the MLP's activation, the block output with its loss
    C.catq_rmsnorm_fwd(st["qp"].view(-1, d), st["hgamma"], st["q"].view(-1, d), st["rq"], 1e-6)
    C.catq_rope(st["q"], S, nh, d, 1e6)
    C.catq_rmsnorm_fwd(st["x"], st["gamma"], st["z"], st["r"], 1e-6, residual=st["branch"], h_out=st["h"])
    C.catq_swiglu_fwd(st["gate"], st["up"], st["m"])
    C.catq_block_output_loss(st["h"], st["mlp"], st["ref"], st["loss"], st["d_out"], st["out"], st["ws"])
    # backward, in its order; the query gradient is turned back in place
    C.catq_swiglu_bwd(st["gate"], st["up"], st["dm"], st["dgate"], st["dup"])
    C.catq_rmsnorm_bwd(st["h"], st["gamma"], st["r"], st["dz"], st["dh"], dZ2=st["dz2"], d_residual=st["dres"])
    C.catq_rope(st["dq"], S, nh, d, 1e6, inverse=True)
    C.catq_rmsnorm_bwd(st["qp"].view(-1, d), st["hgamma"], st["rq"], st["dq"].view(-1, d), st["dqp"].view(-1, d))
    return {n: st[n] for n in ("q", "rq", "z", "r", "h", "m", "loss", "d_out", "out", "dgate", "dup", "dh", "dq", "dqp")}


def _norm_back(x, gamma, dz, eps):
    x = x.detach().requires_grad_()
    _norm(x, gamma, eps).backward(dz)
    return x.grad


def _exact_layers(c, seed):
    t = {n: v.double() for n, v in _layers_inputs(c, _Inputs(seed)).items()}
    T, d = c["T"], c["d"]
    head = (T, c["nh"], d)
    h = t["x"] + t["branch"]
    out = h + t["mlp"]
    diff = out - t["ref"]
    gate, up = t["gate"].requires_grad_(), t["up"].requires_grad_()
    m = torch.nn.functional.silu(gate) * up
    dgate, dup = torch.autograd.grad(m, (gate, up), t["dm"])
    dq = _rope(t["dq"].view(head), c["S"], 1e6, inverse=True)
    qp = t["qp"].view(head)
    return dict(q=_rope(_norm(qp, t["hgamma"], 1e-6), c["S"], 1e6).reshape(T, -1),
                rq=torch.rsqrt(qp.square().mean(-1) + 1e-6).reshape(-1), z=_norm(h, t["gamma"], 1e-6),
                r=torch.rsqrt(h.square().mean(-1) + 1e-6), h=h, m=m.detach(), loss=diff.square().mean().reshape(1),
                d_out=diff * (2.0 / diff.numel()), out=out, dgate=dgate, dup=dup,
                dh=_norm_back(h, t["gamma"], t["dz"] + t["dz2"], 1e-6) + t["dres"], dq=dq.reshape(T, -1),
                dqp=_norm_back(qp, t["hgamma"], dq, 1e-6).reshape(T, -1))


def _work_layers(c):
    T, H, I, qd = c["T"], c["H"], c["I"], c["nh"] * c["d"]
    # per element: h 4+2 in, 4+2 out, norm backward 4+2+2+2 in, 2 out, output 4+2+4 in, 4+2 out;
    # SwiGLU 4 in, 2 out and 6 in, 4 out; head norm and rotation each 2 in, 2 out, both ways
    # (the norm's backward also reads its input)
    return {"bytes": T * H * 40 + T * I * 16 + T * qd * 18, "flops": 0.0}


# ------------------------------------------------------------------ weights

def _prepare_weights(c, seed):
    inp = _Inputs(seed)
    W = inp.normal(c["N"], c["K"], std=0.02)
    G = W.numel() // c["g"]
    layer = C.Layer.create(W, c["g"], *inp.factors(G), recon=c["recon"])
    return dict(layer=layer, codes=inp.empty(W.numel() // 4, dtype=torch.uint8), alpha=inp.empty(G, dtype=F32),
                mu=inp.empty(G, dtype=F32) if c["recon"] else None)


def _run_weights(c, st):
    layer = st["layer"]
    C.catq_group_stats(layer, THR[c["thr"]])
    C.catq_hard_ternarize_pack(layer, st["codes"], st["alpha"], st["mu"])
    out = dict(mu0=layer.mu0, alpha0=layer.alpha0, delta0=layer.delta0, codes=st["codes"], alpha=st["alpha"])
    if st["mu"] is not None:
        out["mu"] = st["mu"]
    return out


def _exact_weights(c, seed):
    inp = _Inputs(seed)
    W = inp.normal(c["N"], c["K"], std=0.02)
    dmu, dal, _ = (f.double() for f in inp.factors(W.numel() // c["g"]))
    mu0, a0, D0 = (v.reshape(-1) for v in _stats64(W, c["g"], c["thr"]))
    out = dict(mu0=mu0, alpha0=a0, delta0=D0, codes=None, alpha=dal * a0)
    if c["recon"]:
        out["mu"] = mu0 + dmu * a0
    return out


def _work_weights(c):
    n = c["N"] * c["K"]
    return {"bytes": 2 * n + n / 4 + n / c["g"] * (12 + 12 + (8 if c["recon"] else 4)), "flops": 0.0}


# ------------------------------------------------------------------ the interface

def prepare(case, seed):
    st = globals()["_prepare_" + case["kind"]](case, seed)
    st["case"] = case
    return st


def run(state):
    return globals()["_run_" + state["case"]["kind"]](state["case"], state)


def work(case):
    return globals()["_work_" + case["kind"]](case)


def exact(case, seed):
    return globals()["_exact_" + case["kind"]](case, seed)


def tolerance(case):
    # fp32 layers: sums of up to a thousand fp32 terms in another order, and the loss's difference
    # of nearly equal outputs.  Statistics: fp32 sums; a code may move where a weight meets its
    # threshold.  The rest is bf16: outputs rounded once, operands rounded once.
    if case["kind"] == "weights":
        return {"rel": 1e-6, "differ": 1e-6}
    if case["kind"] == "step" and case["dtype"] == "f32":
        return {"rel": 2e-5}
    return {"rel": 1e-2}
