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


# Rotary embedding: runs of 1, 2, 4 and 8 heads per thread (by the size of the launch), head counts
# that are no multiple of the run.
@pytest.mark.parametrize("T,S,nh,d", [(3, 2, 1, 16), (65, 64, 9, 64), (1024, 512, 33, 128), (8192, 2048, 21, 128)])
def test_rope_head_runs(device, T, S, nh, d):
    from paper_2606_26650_gb300 import catq as C
    r = syn.rng(301, f"rope/{T}/{nh}")
    x = _bf16(r, (T, nh * d))
    xd = U.to_device(x, "bf16", device)
    C.catq_rope(xd, S, nh, d, 500000.0)
    assert U.fro_rel(_f64(xd), O.rope(x, S, nh, d, 500000.0)) <= 4e-3
