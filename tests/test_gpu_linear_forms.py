"""GPU vs oracle parity of the fused forward and dX in every form that a call can take (pairs of CTAs, two
pairs sharing each weight tile, single CTAs, the narrow kernel by columns, accumulators and shares), with every
epilogue.  catq_linear_form gives the form of a call, and each case asserts the one it is here for."""
import numpy as np
import pytest

from oracle import catq_oracle as O
from paper_2606_26650_gb300 import synthetic as syn
from tests import gpu_util as U

pytestmark = pytest.mark.gpu

SOFT, HARD = O.PHASE_SOFT, O.PHASE_HARD


@pytest.fixture(scope="module")
def device():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.device("cuda:0")


def _form(device, N, K, g, sched, **kw):
    """Pairs per cluster, -1 for tiles of one CTA, or (columns, accumulators, shares) of the narrow kernel,
    on this device."""
    import torch

    from paper_2606_26650_gb300 import catq as C
    sm = torch.cuda.get_device_properties(device).multi_processor_count
    f = C.catq_linear_form(N, K, g, sched, sm_count=sm, **kw)
    return f[0] or f[1:4]


def _bf16(r, shape, scale=1.0):
    return syn.round_bf16((r.standard_normal(shape) * scale).astype(np.float32))


# One linear's step.  what: "plain", "a8" (8-bit activations: the row scale's epilogue), "fused" (loss in the
# epilogue; "f32": a teacher output in fp32, "sum": the sum reduction).  Ragged rows everywhere, ragged
# columns in all but the 72- to 1024-wide dX.  The bf16 bar.
@pytest.mark.parametrize("M,N,K,g,recon,phase,s,what,fwd,dx", [
    # pairs and pairs of pairs: every epilogue, both reconstructions
    (2100, 3080, 576, 192, 1, SOFT, 30.0, "fused", 1, None),
    (2100, 3080, 512, 64, 0, HARD, 30.0, "fused f32 sum", 1, None),
    (2100, 3080, 512, 64, 0, SOFT, 30.0, "a8", 1, None),
    (2100, 3080, 512, 64, 1, SOFT, 3.75, "plain", 1, None),
    (3100, 2056, 192, 192, 1, SOFT, 3.75, "fused", 2, None),
    (3100, 2056, 192, 192, 0, HARD, 30.0, "fused f32", 2, None),
    (3100, 2056, 192, 192, 1, SOFT, 30.0, "fused sum", 2, None),
    (4100, 2056, 64, 64, 0, SOFT, 30.0, "a8", 2, None),
    (3100, 2056, 192, 192, 1, SOFT, 30.0, "plain", 2, None),
    (4100, 136, 2048, 64, 1, SOFT, 30.0, "plain", None, 1),
    (4100, 136, 2048, 64, 0, HARD, 30.0, "plain", None, 1),
    (4100, 72, 2304, 192, 1, SOFT, 30.0, "plain", None, 2),
    (2100, 72, 4096, 64, 0, HARD, 30.0, "plain", None, 2),
    # the narrow forward: 64 and 128 columns, 1 to 4 accumulators, 1 to 8 shares
    (40, 72, 384, 192, 0, SOFT, 3.75, "fused f32", (64, 1, 4), None),
    (1500, 1544, 192, 192, 1, SOFT, 30.0, "fused sum", (64, 2, 1), None),
    (1999, 520, 2304, 192, 0, SOFT, 30.0, "a8", (64, 2, 2), None),
    (777, 1544, 2304, 192, 0, SOFT, 3.75, "fused sum", (64, 3, 2), None),
    (1300, 392, 4608, 192, 1, HARD, 30.0, "plain", (64, 3, 4), None),
    (5586, 8, 11072, 64, 0, SOFT, 30.0, "fused", (64, 4, 8), None),
    (257, 4104, 64, 64, 0, SOFT, 30.0, "a8", (128, 1, 1), None),
    (130, 3080, 2304, 192, 1, SOFT, 30.0, "fused", (128, 2, 4), None),
    (2600, 72, 4096, 64, 0, HARD, 30.0, "a8", (128, 2, 8), None),
    (1030, 4104, 192, 192, 0, HARD, 30.0, "fused f32", (128, 3, 1), None),
    (257, 4104, 2304, 192, 1, SOFT, 30.0, "plain", (128, 3, 4), None),
    (3100, 2056, 64, 64, 1, SOFT, 30.0, "fused", (128, 4, 1), None),
    # the narrow dX; groups of 192 that straddle a tile of 128 columns
    (513, 776, 2304, 192, 1, SOFT, 30.0, "plain", None, (64, 2, 1)),
    (1999, 2056, 576, 192, 0, HARD, 30.0, "plain", None, (64, 2, 2)),
    (4100, 392, 576, 192, 0, SOFT, 30.0, "plain", None, (64, 3, 1)),
    (513, 4104, 1152, 192, 1, SOFT, 30.0, "plain", None, (64, 3, 4)),
    (5641, 11232, 64, 64, 0, SOFT, 30.0, "plain", None, (64, 4, 8)),
    (513, 72, 2304, 192, 0, SOFT, 30.0, "plain", None, (128, 1, 1)),
    (4100, 72, 576, 192, 1, SOFT, 30.0, "plain", None, (128, 2, 1)),
    (130, 4104, 1536, 192, 0, SOFT, 30.0, "plain", None, (128, 2, 8)),
    (4100, 72, 1152, 192, 0, HARD, 30.0, "plain", None, (128, 3, 1)),
    (513, 2056, 2304, 192, 1, SOFT, 30.0, "plain", None, (128, 3, 4)),
    (2600, 4104, 256, 64, 0, SOFT, 30.0, "plain", None, (128, 3, 8)),
    (3100, 72, 2304, 192, 1, SOFT, 30.0, "plain", None, (128, 4, 1))])
def test_form(device, M, N, K, g, recon, phase, s, what, fwd, dx):
    from paper_2606_26650_gb300 import catq as C
    fused, a8 = "fused" in what, "a8" in what
    sched = C.schedule(phase, s)
    assert fwd is None or _form(device, N, K, g, sched, M=M, fused_loss=fused, recon=recon) == fwd
    assert dx is None or _form(device, N, K, g, sched, M=M, dx=True, recon=recon) == dx
    r = syn.rng(320, f"form/{M}/{N}/{K}/{g}")
    W, X = _bf16(r, (N, K), 0.02), _bf16(r, (M, K))
    fac = syn.factors(N * K // g, 320, f"form/{N}/{K}", perturbed=True)
    red = int("sum" in what)
    got = U.gpu_step(W, X, g, fac, O.THR_HALF, phase, s, "bf16", device, recon=recon, fused=fused, a8=a8,
                     teacher_f32="f32" in what, reduction=red)
    stats = O.group_stats(W, g, O.THR_HALF)
    if a8:
        ref = O.a8_calibration_step(X, W, g, stats, fac, phase, s)
    else:
        ref = O.calibration_step(X, W, g, stats, fac, phase, s, reduction=red, with_mu=bool(recon))
    errs = {k: U.fro_rel(got[k], ref[k]) for k in ("Y", "dY", "dX", "g_dmu", "g_dalpha", "g_ddelta")}
    errs["loss"] = abs(got["loss"] - ref["loss"]) / ref["loss"]
    bad = {k: v for k, v in errs.items() if not v <= U.TOL_BF16}
    assert not bad, (bad, errs)


# Grouped launches: experts of no, one, few and many rows, whose tiles end inside the next expert's rows.
# Forward, forward with the loss in its epilogue, and dX, expert by expert against the oracle.
@pytest.mark.parametrize("rows,N,K,g,recon,phase,s,fwd,dx", [
    ([130, 0, 1, 257, 40], 192, 1024, 64, 0, SOFT, 30.0, (128, 1, 8), (64, 1, 1)),
    ([300, 5, 0, 700], 1032, 1152, 192, 1, SOFT, 30.0, (64, 2, 1), (64, 2, 1)),
    ([300, 5, 0, 700], 2056, 1152, 192, 0, HARD, 30.0, (64, 3, 1), (128, 3, 4)),
    ([1100, 0, 900, 2100], 264, 1536, 192, 0, SOFT, 30.0, (128, 3, 4), (128, 3, 1)),
    ([2100, 600, 1030, 1], 2056, 1152, 192, 1, SOFT, 30.0, 1, 1),
    ([2100, 0, 1030, 1], 2056, 1152, 192, 1, SOFT, 30.0, -1, 1),
    ([520, 513, 300, 0, 700, 600], 2056, 576, 64, 0, HARD, 30.0, -1, (128, 2, 2)),
    ([2100, 0, 1030, 1], 1032, 2304, 192, 0, SOFT, 3.75, 1, -1),
    ([520, 513, 300, 0, 700, 600], 1032, 2304, 192, 1, SOFT, 30.0, (128, 2, 1), -1),
    ([1100, 0, 900, 2100], 1032, 1152, 192, 0, SOFT, 30.0, 2, 2),
    ([1100, 0, 900, 2100], 1032, 1152, 192, 1, HARD, 30.0, 2, 2)])
def test_grouped_form(device, rows, N, K, g, recon, phase, s, fwd, dx):
    import torch

    from paper_2606_26650_gb300 import catq as C
    sched = C.schedule(phase, s)
    off = [0] + [int(v) for v in np.cumsum(rows)]
    E, R, per = len(rows), off[-1], N * K // g
    for loss in (False, True):
        assert _form(device, N, K, g, sched, row_offsets=off, fused_loss=loss, recon=recon) == fwd
    assert _form(device, N, K, g, sched, row_offsets=off, dx=True, recon=recon) == dx
    r = syn.rng(321, f"grouped form/{R}/{N}/{K}")
    W, X, dY, Yr = _bf16(r, (E, N, K), 0.02), _bf16(r, (R, K)), _bf16(r, (R, N)), _bf16(r, (R, N))
    fac = syn.factors(E * per, 321, f"grouped form/{N}/{K}", perturbed=True)
    layer = C.GroupedLayer.create(U.to_device(W.reshape(E * N, K), "bf16", device).view(E, N, K), g,
                                  *(torch.from_numpy(f).to(device) for f in fac), recon=recon)
    C.catq_group_stats(layer.dense)
    x, dy, yr = (U.to_device(a, "bf16", device) for a in (X, dY, Yr))
    y, y2, dl = (torch.full_like(yr, float("nan")) for _ in range(3))
    dxd, loss = torch.full_like(x, float("nan")), torch.zeros(1, device=device)
    C.catq_grouped_soft_ternary_linear_fwd(layer, sched, x, off, y)
    ws = C.workspace(C.catq_grouped_fwd_loss_workspace_bytes(layer, off), device)
    C.catq_grouped_soft_ternary_linear_fwd_loss(layer, sched, x, off, yr, loss, dl, Y=y2, workspace=ws)
    C.catq_grouped_soft_ternary_linear_bwd(layer, sched, x, dy, off, dxd)
    assert C.catq_device_status() == 0
    yh, y2h, dxh = (U.to_host(t) for t in (y, y2, dxd))
    want = np.zeros((R, N))
    for e in range(E):
        a, b = off[e], off[e + 1]
        if a == b:
            continue
        fe = tuple(f[e * per:(e + 1) * per] for f in fac)
        Wq = O.ternary_weight(W[e], g, O.group_stats(W[e], g, O.THR_HALF), fe, phase, s, with_mu=bool(recon))[0]
        want[a:b] = X[a:b].astype(np.float64) @ Wq.T
        assert U.fro_rel(yh[a:b], want[a:b]) <= U.TOL_BF16, e
        assert U.fro_rel(y2h[a:b], want[a:b]) <= U.TOL_BF16, e
        assert U.fro_rel(dxh[a:b], dY[a:b].astype(np.float64) @ Wq) <= U.TOL_BF16, e
    ref_loss, ref_dY = O.recon_loss(want, Yr.astype(np.float64))
    assert abs(loss.item() - ref_loss) <= U.TOL_BF16 * ref_loss
    assert U.fro_rel(U.to_host(dl), ref_dY) <= U.TOL_BF16
