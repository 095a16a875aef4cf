"""GPU vs oracle parity at the edges of the size rules by which a call picks its kernel: one small
test per kernel variant, at the sizes where its tiles, teams or splits begin and end."""
import numpy as np
import pytest

from oracle import catq_oracle as O
from paper_2606_26650_gb300 import synthetic as syn
from tests import gpu_util as U

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def device():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.device("cuda:0")


def _bf16(r, shape, scale=1.0):
    return syn.round_bf16((r.standard_normal(shape) * scale).astype(np.float32))


def _f64(t):
    return U.to_host(t).astype(np.float64)


# Row norms: teams of 1 to 32 lanes (H to 1024, with 1, 2 and 4 vectors a lane), a CTA per row above with 1, 2 or 4 a thread,
# and rows past the vectors a CTA keeps in registers (8192 elements).  bf16 outputs of fp32
# arithmetic round once: 2^-9 relative, so 4e-3 bounds the relative Frobenius error.
@pytest.mark.parametrize("H", [8, 24, 128, 136, 256, 264, 512, 520, 1024, 1032, 2048, 2056, 4096, 4104, 8192, 8200])
@pytest.mark.parametrize("gamma_offset", [0, 1])
def test_row_norm_edges(device, H, gamma_offset):
    import torch

    from paper_2606_26650_gb300 import catq as C
    T = 67
    r = syn.rng(300, f"rows/{H}")
    x = r.standard_normal((T, H)).astype(np.float32)
    res, dz = _bf16(r, (T, H), 0.5), _bf16(r, (T, H))
    gamma = r.uniform(0.5, 1.5, H).astype(np.float32)
    gbuf = torch.zeros(H + 4, dtype=torch.float32, device=device)
    gd = gbuf[gamma_offset:gamma_offset + H]  # offset 1: aligned to 4 bytes only
    gd.copy_(torch.from_numpy(gamma))
    xd, resd = torch.from_numpy(x).to(device), U.to_device(res, "bf16", device)
    Z = torch.empty(T, H, dtype=torch.bfloat16, device=device)
    h = torch.empty(T, H, dtype=torch.float32, device=device)
    rr = torch.empty(T, dtype=torch.float32, device=device)
    C.catq_rmsnorm_fwd(xd, gd, Z, rr, 1e-5, residual=resd, h_out=h)
    hx = x.astype(np.float64) + res
    z_ref, r_ref = O.rmsnorm(hx, gamma, 1e-5)
    assert U.max_rel(_f64(h), hx) <= 1e-7
    assert U.max_rel(_f64(rr), r_ref) <= 1e-6
    assert U.fro_rel(_f64(Z), z_ref) <= 4e-3
    # backward in place on its upstream gradient
    g = U.to_device(dz, "bf16", device)
    C.catq_rmsnorm_bwd(h, gd, rr, g, g, d_residual=resd)
    want = O.rmsnorm_bwd(_f64(h), gamma, _f64(rr), dz) + res
    assert U.fro_rel(_f64(g), want) <= 4e-3


# Weights 4, 8 and 12 bytes past a 16-byte boundary, in every kind of row: the arithmetic is the aligned one's,
# bit for bit.  And launches of one row a team in flight beside those of two or four (9000
# rows and more).
@pytest.mark.parametrize("H,T", [(8, 3), (24, 40000), (128, 9000), (136, 9000), (256, 67), (520, 67), (1024, 67), (1032, 67), (2056, 67), (8200, 19)])
def test_row_norm_weight_alignment(device, H, T):
    import torch

    from paper_2606_26650_gb300 import catq as C
    gen = torch.Generator(device=device).manual_seed(H)
    x = torch.randn(T, H, generator=gen, device=device)
    dz = torch.randn(T, H, generator=gen, device=device).bfloat16()
    buf = torch.rand(H + 4, generator=gen, device=device) + 0.5
    first = None
    for off in range(4):
        g = torch.zeros(H + 4, device=device)[off:off + H]
        g.copy_(buf[:H])
        out = []
        for a in (x, x.bfloat16()):
            z, r, dx = torch.empty_like(dz), torch.empty(T, device=device), torch.empty_like(dz)
            C.catq_rmsnorm_fwd(a, g, z, r, 1e-5)
            C.catq_rmsnorm_bwd(a, g, r, dz, dx)
            out += [z, r, dx]
        first = first or out
        assert all(torch.equal(a, b) for a, b in zip(first, out)), off
    want, _ = O.rmsnorm(_f64(x), _f64(buf[:H]), 1e-5)
    assert U.fro_rel(_f64(first[0]), want) <= 4e-3


# Rotary embedding: runs of 1, 2, 4 and 8 heads per thread (by the size of the launch: 1 in the first three
# cases), head counts that are no multiple of the run.
@pytest.mark.parametrize("T,S,nh,d", [(3, 2, 1, 16), (65, 64, 9, 64), (1024, 512, 33, 128), (8192, 2048, 13, 128),
                                       (8192, 2048, 21, 128), (8192, 2048, 37, 128)])
def test_rope_head_runs(device, T, S, nh, d):
    from paper_2606_26650_gb300 import catq as C
    r = syn.rng(301, f"rope/{T}/{nh}")
    x = _bf16(r, (T, nh * d))
    xd = U.to_device(x, "bf16", device)
    C.catq_rope(xd, S, nh, d, 500000.0)
    assert U.fro_rel(_f64(xd), O.rope(x, S, nh, d, 500000.0)) <= 4e-3


# The fused contraction's narrow form at odd sizes: one row, rows and columns past the matrix, the
# contraction cut into 1 to 8 shares (of unequal length where their number does not divide it), both soft
# forms and the hard one, the loss in its epilogue; and pairs of CTAs on fewer than 512 rows
# (400 x 2048 x 8192).  The bf16 bar.  (Every form by its columns and accumulators: test_gpu_linear_forms.py.)
@pytest.mark.parametrize("M,N,K,g,recon,phase,s,fused", [
    (1, 8, 64, 64, 0, O.PHASE_SOFT, 30.0, False), (3, 72, 1408, 128, 0, O.PHASE_SOFT, 3.75, True),
    (127, 328, 960, 192, 1, O.PHASE_SOFT, 30.0, True), (129, 136, 4032, 64, 0, O.PHASE_HARD, 30.0, False),
    (300, 1024, 2048, 2048, 0, O.PHASE_SOFT, 7.5, False), (513, 264, 1152, 384, 1, O.PHASE_HARD, 15.0, False),
    (1000, 520, 704, 64, 0, O.PHASE_SOFT, 30.0, True), (400, 8192, 2048, 128, 0, O.PHASE_SOFT, 30.0, False)])
def test_linear_narrow_forms(device, M, N, K, g, recon, phase, s, fused):
    r = syn.rng(302, f"narrow/{M}/{N}/{K}")
    W, X = _bf16(r, (N, K), 0.02), _bf16(r, (M, K))
    fac = syn.factors(N * K // g, 3, f"narrow/{N}/{K}", perturbed=True)
    got = U.gpu_step(W, X, g, fac, O.THR_HALF, phase, s, "bf16", device, recon=recon, fused=fused)
    ref = O.calibration_step(X, W, g, O.group_stats(W, g, O.THR_HALF), fac, phase, s, with_mu=bool(recon))
    errs = {k: U.fro_rel(got[k], ref[k]) for k in ("Y", "dY", "dX")}
    errs["loss"] = abs(got["loss"] - ref["loss"]) / ref["loss"]
    bad = {k: v for k, v in errs.items() if not v <= U.TOL_BF16}
    assert not bad, (bad, errs)


# Grouped launches in the narrow form: experts of 0, 1, 130 and 257 rows, and the same rows expert by
# expert as dense layers, cut otherwise, agree (the contraction's order alone differs, in fp32: 1e-2 in
# bf16).  Against the oracle: test_gpu_linear_forms.py.
def test_grouped_narrow_matches_dense(device):
    import torch

    from paper_2606_26650_gb300 import catq as C
    E, N, K, g, rows = 5, 192, 1024, 128, [130, 0, 1, 257, 40]
    off = [0] + [int(v) for v in np.cumsum(rows)]
    r = syn.rng(303, "grouped narrow")
    W = U.to_device(_bf16(r, (E * N, K), 0.02), "bf16", device).view(E, N, K)
    X = U.to_device(_bf16(r, (off[-1], K)), "bf16", device)
    dY = U.to_device(_bf16(r, (off[-1], N)), "bf16", device)
    fac = [torch.from_numpy(f).to(device) for f in syn.factors(E * N * K // g, 3, "grouped narrow", perturbed=True)]
    layer = C.GroupedLayer.create(W, g, *fac)
    C.catq_group_stats(layer.dense)
    sched = C.schedule(C.PHASE_SOFT, 30.0)
    Y, dX = torch.empty(off[-1], N, dtype=X.dtype, device=device), torch.empty_like(X)
    C.catq_grouped_soft_ternary_linear_fwd(layer, sched, X, off, Y)
    C.catq_grouped_soft_ternary_linear_bwd(layer, sched, X, dY, off, dX)
    per = N * K // g
    for e in range(E):
        a, b = off[e], off[e + 1]
        if a == b:
            continue
        one = C.Layer.create(W[e], g, *(f[e * per:(e + 1) * per].clone() for f in fac))
        C.catq_group_stats(one)
        y, dx = torch.empty(b - a, N, dtype=X.dtype, device=device), torch.empty(b - a, K, dtype=X.dtype, device=device)
        C.catq_soft_ternary_linear_fwd(one, sched, X[a:b], y)
        C.catq_soft_ternary_linear_bwd(one, sched, X[a:b], dY[a:b], dx)
        assert U.fro_rel(_f64(Y[a:b]), _f64(y)) <= 1e-2
        assert U.fro_rel(_f64(dX[a:b]), _f64(dx)) <= 1e-2


# Grouped dW: one CTA per tile and pairs, rows and columns short of a tile, groups of 64 (a partial sum per
# 64 columns), 128 and more, both phases and reconstructions, experts of no and of few rows (tiles
# whose weights follow each other closely; three runs, the same bits).  Against the oracle.
@pytest.mark.parametrize("N,K,g,recon,phase,s", [
    (120, 448, 64, 0, O.PHASE_SOFT, 30.0), (392, 640, 128, 1, O.PHASE_SOFT, 7.5), (768, 2048, 128, 0, O.PHASE_SOFT, 30.0),
    (264, 768, 384, 0, O.PHASE_HARD, 30.0), (512, 1024, 512, 0, O.PHASE_SOFT, 3.75)])
def test_grouped_dw(device, N, K, g, recon, phase, s):
    import torch

    from paper_2606_26650_gb300 import catq as C
    rows = [3, 0, 300, 1, 64, 17, 130, 5]
    E, per, off = len(rows), N * K // g, [0] + [int(v) for v in np.cumsum(rows)]
    r = syn.rng(307, f"grouped dw/{N}/{K}")
    W, X, dY = _bf16(r, (E, N, K), 0.02), _bf16(r, (off[-1], K)), _bf16(r, (off[-1], N))
    fac = syn.factors(E * per, 3, f"grouped dw/{N}/{K}", perturbed=True)
    layer = C.GroupedLayer.create(U.to_device(W.reshape(E * N, K), "bf16", device).view(E, N, K), g,
                                  *(torch.from_numpy(f).to(device) for f in fac), recon=recon)
    C.catq_group_stats(layer.dense)
    x, dy = U.to_device(X, "bf16", device), U.to_device(dY, "bf16", device)
    first, ws = None, C.workspace(C.catq_grouped_bwd_workspace_bytes(layer, off), device)
    for _ in range(3):
        got = [torch.full((E * per,), float("nan"), device=device) for _ in range(3)]
        C.catq_grouped_soft_ternary_linear_bwd(layer, C.schedule(phase, s), x, dy, off, torch.empty_like(x), *got,
                                               workspace=ws)
        assert C.catq_device_status() == 0
        first = first or got
        assert all(torch.equal(a, b) for a, b in zip(first, got))
    want = [np.zeros(E * per) for _ in range(3)]
    for e in range(E):
        at, grp = slice(off[e], off[e + 1]), slice(e * per, (e + 1) * per)
        ref = O.linear_bwd(X[at], dY[at], W[e], g, O.group_stats(W[e], g, O.THR_HALF), tuple(f[grp] for f in fac), phase, s,
                           with_mu=bool(recon))
        for dst, src in zip(want, ref[1:]):
            dst[grp] = src
    for name, a, b in zip(("g_dmu", "g_dalpha", "g_ddelta"), first, want):
        assert U.fro_rel(_f64(a), b) <= U.TOL_BF16, name


# The fp32 path: tiles of 32, 128 and 256 rows with remainders, an output width that is no multiple of
# 4, groups of 4 to 512, contractions shared by 1 to 8 CTAs, a single slice.  The fp32 bar.
@pytest.mark.parametrize("M,N,K,g,recon,phase,s", [
    (1, 17, 4, 4, 0, O.PHASE_SOFT, 30.0), (13, 342, 640, 64, 1, O.PHASE_SOFT, 7.5), (33, 36, 1024, 16, 0, O.PHASE_HARD, 30.0),
    (129, 130, 96, 32, 0, O.PHASE_SOFT, 3.75), (300, 64, 520, 8, 1, O.PHASE_SOFT, 30.0), (700, 511, 512, 512, 0, O.PHASE_SOFT, 30.0)])
def test_linear_fp32_tiles(device, M, N, K, g, recon, phase, s):
    r = syn.rng(304, f"fp32/{M}/{N}/{K}")
    W, X = (r.standard_normal((N, K)) * 0.02).astype(np.float32), r.standard_normal((M, K)).astype(np.float32)
    fac = syn.factors(N * K // g, 3, f"fp32/{N}/{K}", perturbed=True)
    got = U.gpu_step(W, X, g, fac, O.THR_HALF, phase, s, "f32", device, recon=recon)
    ref = O.calibration_step(X, W, g, O.group_stats(W, g, O.THR_HALF), fac, phase, s, with_mu=bool(recon))
    errs = {k: U.max_rel(got[k], ref[k]) for k in ("Y_ref", "Y", "dY", "dX", "g_dmu", "g_dalpha", "g_ddelta")}
    errs["loss"] = abs(got["loss"] - ref["loss"]) / ref["loss"]
    bad = {k: v for k, v in errs.items() if not v <= U.TOL_F32}
    assert not bad, (bad, errs)


# Attention tiles of 128 tokens with a last one of 64, for both head widths: one tile, a half tile alone,
# odd numbers of 64-token blocks, query heads in groups of 1, 2, 3 and 5; log-sum-exp and delta on
# 4-byte alignment.  Two sequences, so that what lies past the first one's end is the second.  bf16
# operands and probabilities: the bf16 bar.
@pytest.mark.parametrize("S,nh,nkv,d", [(64, 3, 1, 64), (192, 2, 2, 64), (320, 5, 1, 128), (64, 2, 1, 128),
                                        (448, 4, 2, 128), (128, 6, 2, 64), (832, 2, 1, 64)])
def test_attention_ragged_tiles(device, S, nh, nkv, d):
    import torch

    from paper_2606_26650_gb300 import catq as C
    B = 2
    r = syn.rng(305, f"attn/{S}/{nh}/{d}")
    q, k, v, do = (_bf16(r, (B * S, n * d)) for n in (nh, nkv, nkv, nh))
    qd, kd, vd, dod = (U.to_device(t, "bf16", device) for t in (q, k, v, do))
    o, dq, dk, dv = (torch.full_like(t, float("nan")) for t in (qd, qd, kd, vd))
    rows = B * nh * S
    lse = torch.zeros(rows + 1, dtype=torch.float32, device=device)[1:]
    delta = torch.zeros(rows + 1, dtype=torch.float32, device=device)[1:]
    C.catq_attention_fwd(qd, kd, vd, o, lse, B, S, nh, nkv, d)
    C.catq_attention_bwd(qd, kd, vd, o, dod, lse, delta, dq, dk, dv, B, S, nh, nkv, d)
    assert C.catq_device_status() == 0
    o_ref, p = O.attention(q, k, v, B, S, nh, nkv, d)
    dq_ref, dk_ref, dv_ref = (t.reshape(B * S, -1) for t in O.attention_bwd(q, k, v, p, do, B, S, nh, nkv, d))
    assert np.abs(_f64(lse).reshape(B, nh, S) - O.attention_logsumexp(q, k, B, S, nh, nkv, d)).max() <= 1e-4
    for name, got, want in (("o", o, o_ref.reshape(B * S, -1)), ("dq", dq, dq_ref), ("dk", dk, dk_ref), ("dv", dv, dv_ref)):
        assert U.fro_rel(_f64(got), want) <= U.TOL_BF16, name


# Inference on packed codes: one super-chunk for eight warps, groups longer and shorter than a slab, several
# slabs of equal and (16 x 20608, 23 x 20160, 9720 x 6720) unequal length, items of 16 rows and (9720) of 32
# with remainders, two token blocks, scales and activations at their least alignment (no 16-byte scale
# copies, no 32-byte activation loads).
@pytest.mark.parametrize("N,K,g,B,mu,shift", [
    (33, 64, 64, 1, False, 0), (40, 192, 192, 9, True, 1), (16, 20480, 256, 8, False, 0), (48, 24576, 24576, 3, True, 0),
    (9744, 256, 128, 2, False, 1), (9744, 640, 64, 8, True, 0), (31, 17408, 128, 5, False, 1),
    (9720, 256, 128, 2, False, 1), (9720, 6720, 64, 3, True, 0), (16, 20608, 128, 8, False, 0), (23, 20160, 192, 5, True, 1)])
def test_ternary_infer_slabs(device, N, K, g, B, mu, shift):
    import torch

    from paper_2606_26650_gb300 import catq as C
    r = syn.rng(306, f"infer/{N}/{K}/{g}")
    c = r.integers(0, 3, (N * K // 4, 4)).astype(np.uint8)
    packed = (c[:, 0] | c[:, 1] << 2 | c[:, 2] << 4 | c[:, 3] << 6).astype(np.uint8)
    G = N * K // g
    alpha = r.uniform(0.5, 1.5, G).astype(np.float32) / np.sqrt(K).astype(np.float32)
    off = r.uniform(-0.1, 0.1, G).astype(np.float32) / np.sqrt(K).astype(np.float32) if mu else None
    X = _bf16(r, (B, K))

    def at(a, dtype, skip):  # on the device, `skip` elements into its buffer
        buf = torch.zeros(a.size + skip, dtype=dtype, device=device)
        buf[skip:] = torch.from_numpy(np.ascontiguousarray(a).reshape(-1)).to(device).to(dtype)
        return buf[skip:].view(a.shape)

    codes, al = at(packed, torch.uint8, 0), at(alpha, torch.float32, shift)
    m = at(off, torch.float32, shift) if mu else None
    x, y = at(X, torch.bfloat16, 8 * shift), torch.full((B, N), float("nan"), dtype=torch.bfloat16, device=device)
    want = O.ternary_infer(packed, alpha, N, K, g, X, mu=off)
    for _ in range(2):
        C.catq_ternary_infer_batched([(codes, al, N, K, x, y, m)], g)
        assert C.catq_device_status() == 0
        assert U.fro_rel(_f64(y), want) <= U.TOL_BF16
    sync = torch.zeros(C.catq_ternary_infer_sync_bytes() // 4, dtype=torch.int32, device=device)
    y2 = torch.full_like(y, float("nan"))
    C.catq_ternary_infer_staged([(codes, al, N, K, x, y, m), (codes, al, N, K, x, y2, m)], [0, 1], g, sync)
    assert C.catq_device_status() == 0
    assert torch.equal(y, y2) and not sync.any()


# 8-bit activations: rows in a warp's registers (2 and 8 vectors a lane) and in a block's (2, 4 and 8 a thread),
# at both ends of each and past the last; a row of zeros, the largest element first and last.
# Scales and codes are the oracle's, bit for bit.
@pytest.mark.parametrize("dtype,V", [("bf16", 8), ("f32", 4)])
@pytest.mark.parametrize("nvec", [1, 64, 65, 256, 257, 512, 513, 1024, 1025, 2048, 2049])
def test_act_quant_rows(device, dtype, V, nvec):
    import torch

    from paper_2606_26650_gb300 import catq as C
    M, K = 19, nvec * V
    X = (syn.rng(308, f"a8/{nvec}").standard_normal((M, K)) * 3.0).astype(np.float32)
    X[7] = 0.0
    X[11, -1], X[12, 0] = 40.0, -50.0
    X = syn.round_bf16(X) if dtype == "bf16" else X
    x = U.to_device(X, dtype, device)
    codes, deq = torch.full_like(x, float("nan")), torch.full_like(x, float("nan"))
    scale = torch.full((M,), float("nan"), device=device)
    C.catq_act_quant_a8(x, codes, scale, deq)
    q, s = O.act_quant_a8(X)
    np.testing.assert_array_equal(U.to_host(scale), s)
    np.testing.assert_array_equal(_f64(codes), q)
    C.catq_act_quant_a8(x, codes, scale)
    np.testing.assert_array_equal(_f64(codes), q)
    assert U.err(_f64(deq), q * s.astype(np.float64)[:, None], dtype) <= (3e-3 if dtype == "bf16" else 1e-6)


# Scores of -inf, and of the type's lowest value, in the online softmax's two chains of key tiles: whole tiles
# of such keys first, second and last in their chain, and single ones; a query that sees one such
# key alone in a tile (128 in tile 1).  -inf keys weigh nothing; rows whose every key is lowest weigh
# them alike.  Outputs to the bf16 bar, log-sum-exp to 1e-5 of its value (fp32) or 1e-4.
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("S,keys,value", [
    (576, [(128, 256)], -np.inf), (576, [(128, 129), (300, 301), (575, 576)], -np.inf),
    (576, [(128, 384), (512, 576)], -np.inf), (576, [(0, 128)], -3.38e38), (576, [(128, 256), (384, 512)], -3.38e38),
    (320, [(0, 320)], -3.38e38), (192, [(1, 64), (128, 130)], -np.inf)])
def test_attention_masking_scores(device, S, keys, value, d):
    import torch

    from paper_2606_26650_gb300 import catq as C
    B, nh, nkv = 2, 3, 1
    r = syn.rng(309, f"mask/{S}/{d}/{len(keys)}")
    q, k, v = (_bf16(r, (B * S, n * d)) for n in (nh, nkv, nkv))
    q.reshape(B * S, nh, d)[:, :, 0] = 1.0  # the first column carries the mask
    for a, b in keys:
        k.reshape(B, S, nkv * d)[:, a:b, 0] = syn.round_bf16(np.array([value], np.float32))[0]
    qd, kd, vd = (U.to_device(t, "bf16", device) for t in (q, k, v))
    o, lse = torch.full_like(qd, float("nan")), torch.full((B * nh * S,), float("nan"), device=device)
    C.catq_attention_fwd(qd, kd, vd, o, lse, B, S, nh, nkv, d)
    assert C.catq_device_status() == 0
    want, _ = O.attention(q, k, v, B, S, nh, nkv, d)
    l_ref = O.attention_logsumexp(q, k, B, S, nh, nkv, d)
    assert np.isfinite(want).all() and np.isfinite(l_ref).all()
    assert U.fro_rel(_f64(o), want.reshape(B * S, -1)) <= U.TOL_BF16
    assert (np.abs(_f64(lse).reshape(B, nh, S) - l_ref) <= 1e-4 + 1e-5 * np.abs(l_ref)).all()


# A pack, or a copy into the codes, and the inference that reads them, one after the other on a stream with
# no synchronisation, the same buffers every time: each result is that of its own codes, bit for bit.
@pytest.mark.parametrize("N,K,g,B", [(64, 256, 64, 1), (1024, 4096, 128, 3), (9744, 2048, 128, 1)])
def test_inference_follows_its_pack(device, N, K, g, B):
    import torch

    from paper_2606_26650_gb300 import catq as C
    r = syn.rng(310, f"pack/{N}/{K}")
    layers = [C.Layer.create(U.to_device(_bf16(r, (N, K), 0.02), "bf16", device), g) for _ in range(3)]
    X = U.to_device(_bf16(r, (B, K)), "bf16", device)
    codes = torch.zeros(N * K // 4, dtype=torch.uint8, device=device)
    alpha = torch.zeros(N * K // g, device=device)
    want, kept = [], []
    for layer in layers:
        C.catq_group_stats(layer)
        C.catq_hard_ternarize_pack(layer, codes, alpha)
        torch.cuda.synchronize()
        y = torch.empty(B, N, dtype=X.dtype, device=device)
        C.catq_ternary_infer(codes, alpha, N, K, g, X, y)
        torch.cuda.synchronize()
        want.append(y)
        kept.append((codes.clone(), alpha.clone()))
    assert not torch.equal(want[0], want[1])
    got = torch.full((120, B, N), float("nan"), dtype=X.dtype, device=device)
    for i in range(120):
        if i % 2:
            C.catq_hard_ternarize_pack(layers[i % 3], codes, alpha)
        else:
            codes.copy_(kept[i % 3][0])
            alpha.copy_(kept[i % 3][1])
        C.catq_ternary_infer(codes, alpha, N, K, g, X, got[i])
    assert C.catq_device_status() == 0
    assert all(torch.equal(got[i], want[i % 3]) for i in range(120))


# Host threads, each with its own stream, layer and buffers, whose two shapes take ring depths of their own in
# one kernel: what one call asks for in shared memory must not depend on another's.  (Arguments are made
# beforehand: the calls themselves run side by side, without the interpreter's lock.)
@pytest.mark.parametrize("what", ["forward", "infer"])
def test_threads_with_different_shapes(device, what):
    import threading

    import torch

    from paper_2606_26650_gb300 import catq as C
    failed = []

    def work(N, K, g):
        with torch.cuda.stream(torch.cuda.Stream(device)):
            X, Y = (torch.ones(1, n, dtype=torch.bfloat16, device=device) for n in (K, N))
            layer = C.Layer.create(torch.randn(N, K, device=device).bfloat16(), g)
            C.catq_group_stats(layer)
            codes = torch.zeros(N * K // 4, dtype=torch.uint8, device=device)
            alpha = torch.ones(N * K // g, device=device)
            stream = torch.cuda.current_stream()
            stream.synchronize()
            if what == "forward":
                st = layer.struct()
                call, args = C.lib().catq_soft_ternary_linear_fwd, (
                    C.ctypes.byref(st), C.schedule(C.PHASE_HARD, 30.0), X.data_ptr(), 1, C.BF16, Y.data_ptr(),
                    stream.cuda_stream)
            else:
                call, args = C.lib().catq_ternary_infer, (codes.data_ptr(), alpha.data_ptr(), None, N, K, g,
                                                          X.data_ptr(), 1, C.BF16, Y.data_ptr(), stream.cuda_stream)
            for _ in range(5000):
                status = call(*args)
                if status != 0:
                    failed.append(C.STATUS.get(status, status))
                    break
            stream.synchronize()

    threads = [threading.Thread(target=work, args=a) for a in [(64, 64, 64), (64, 16384, 64)] * 2]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed and C.catq_device_status() == 0, failed
