"""How the fused forward and dX are cut, on the CPU: the plan's rings and constants' table fit, and the
choice between the narrow kernel and CTA pairs at sizes measured on both sides."""
import ctypes
import random

import pytest

from paper_2606_26650_gb300 import catq as C

SMEM = 227 * 1024 - 128  # of a CTA, less the kernel's static part
SOFT = C.schedule(C.PHASE_SOFT, 30.0)


def _ceil(a, b):
    return -(-a // b)


def _table_pairs(bn, dx, N, K, g, kb0, kb1, col0):
    """(weight row, group) pairs that one CTA's share meets: blocks kb0 .. kb1 - 1 of the contraction and
    the tile's columns from col0, rows past N counted like the others."""
    if dx:  # the share's rows x the groups of the tile's columns
        last = min(col0 + bn, K) - 1
        return (kb1 - kb0) * 64 * (last // g - col0 // g + 1)
    last = min(kb1 * 64, K) - 1
    return bn * (last // g - kb0 * 64 // g + 1)


def test_narrow_tables_and_rings_fit():
    r = random.Random(7)
    seen = set()
    for _ in range(4000):
        g = 64 * r.choice([1, 1, 2, 3, 4, 5, 6, 8, 16])
        K = g * max(1, int(2 ** r.uniform(6, 14.2)) // g)
        N, M = 8 * int(2 ** r.uniform(0, 11)), int(2 ** r.uniform(0, 12.5))
        dx, recon = r.random() < 0.5, r.choice([0, 1])
        pairs, bn, nacc, splits, sa, sw, entries = C.catq_linear_form(N, K, g, SOFT, M, dx=dx, recon=recon)
        if pairs:
            assert (bn, nacc, splits, sa, sw, entries) == (0,) * 6
            continue
        seen.add((bn, nacc, splits, dx, g % bn != 0 and bn % g != 0))
        T, cols = _ceil(N if dx else K, 64), K if dx else N
        for rank in range(splits):
            kb0, kb1 = T * rank // splits, T * (rank + 1) // splits
            assert kb0 < kb1
            for col0 in {0, bn * (cols // bn // 2), bn * ((cols - 1) // bn)}:
                assert _table_pairs(bn, dx, N, K, g, kb0, kb1, col0) <= entries
        assert 2 <= sa <= 8 and sw in (2, 4, 6, 8) and bn * nacc <= 512
        rings = sa * nacc * 16384 + sw * bn * 128
        assert rings >= 128 * bn * 4  # the partial sums meet in them
        assert rings + entries * (20 if recon else 16) + 344 + 16 + 1024 <= SMEM
    assert {s[:2] for s in seen} >= {(b, n) for b in (64, 128) for n in (1, 2, 3)} | {(128, 4)}
    assert {s[2] for s in seen} == {1, 2, 4, 8}
    assert any(s[0] == 128 and s[3] and s[4] for s in seen)  # groups that straddle a tile's columns


# Sizes where the narrow kernel's two-slot rings, or two tanh a weight in dX, ran 1.1 to 2 times longer than
# CTA pairs (one GB300, both measured).
@pytest.mark.parametrize("M,N,K,g,dx,recon,phase,s", [
    (654, 4096, 14336, 128, False, 0, C.PHASE_SOFT, 30.0), (520, 4096, 14336, 128, False, 0, C.PHASE_HARD, 30.0),
    (520, 4096, 4096, 128, True, 0, C.PHASE_SOFT, 1.875), (191, 7496, 9216, 128, True, 0, C.PHASE_HARD, 30.0),
    (284, 5120, 5120, 64, False, 0, C.PHASE_SOFT, 30.0), (968, 5664, 3072, 64, True, 1, C.PHASE_SOFT, 30.0),
    (2369, 1024, 5120, 64, False, 0, C.PHASE_SOFT, 30.0), (1494, 14536, 2176, 128, True, 0, C.PHASE_SOFT, 30.0),
    (1484, 2048, 2048, 64, True, 0, C.PHASE_SOFT, 1.875), (1039, 1088, 3328, 64, True, 0, C.PHASE_SOFT, 1.875)])
def test_pairs_where_the_narrow_kernel_is_slower(M, N, K, g, dx, recon, phase, s):
    assert C.catq_linear_form(N, K, g, C.schedule(phase, s), M, dx=dx, recon=recon)[0] > 0


# And where it is the faster one, by 1.1 to 5 times.
@pytest.mark.parametrize("M,N,K,g,dx,recon", [
    (8, 1024, 2048, 128, False, 0), (300, 1024, 2048, 128, False, 0), (300, 1024, 2048, 128, True, 0),
    (1000, 2048, 2048, 128, False, 0), (674, 6144, 2048, 64, True, 1), (312, 14336, 4096, 128, True, 0)])
def test_narrow_where_it_is_faster(M, N, K, g, dx, recon):
    assert C.catq_linear_form(N, K, g, SOFT, M, dx=dx, recon=recon)[0] == 0


# Grouped launches of few rows an expert, where pairs leave most of a tile's rows empty: forms that measured 1.1
# to 1.3 times faster than pairs.
@pytest.mark.parametrize("E,rows,N,K,dx,form", [
    (62, 6, 4096, 1536, False, (-1, 0, 0, 0)), (62, 6, 4096, 1536, True, (-1, 0, 0, 0)),
    (61, 10, 1536, 4096, True, (-1, 0, 0, 0)), (40, 11, 1536, 4096, False, (-1, 0, 0, 0)),
    (64, 10, 768, 2048, False, (0, 128, 1, 1)), (64, 10, 768, 2048, True, (-1, 0, 0, 0)),
    (128, 512, 1536, 4096, False, (1, 0, 0, 0))])
def test_grouped_form_for_few_rows(E, rows, N, K, dx, form):
    assert C.catq_linear_form(N, K, 128, SOFT, row_offsets=[rows * e for e in range(E + 1)], dx=dx)[:4] == form


def test_grouped_and_argument_checks():
    off = [0, 130, 130, 131, 388]
    assert C.catq_linear_form(192, 1024, 128, SOFT, row_offsets=off)[0] == 0
    assert C.catq_linear_form(1536, 4096, 128, SOFT, row_offsets=[0, 4096, 8192])[0] == 2
    lib, form = C.lib(), (ctypes.c_int32 * 7)()

    def status(N=64, K=256, g=128, recon=0, sched=SOFT, M=4, E=0, off=None, dx=0, loss=0, sm=152, out=form):
        return lib.catq_linear_form(N, K, g, recon, sched, M, E, off, dx, loss, sm, out)

    assert status() == 0
    assert status(N=60) == 2 and status(K=250) == 2 and status(g=32) == 2 and status(g=0) == 2
    assert status(M=0) == 1 and status(sm=0) == 1 and status(recon=2) == 1 and status(out=None) == 1
    assert status(dx=1, loss=1) == 1 and status(sched=C.schedule(C.PHASE_SOFT, 0.0)) == 1
    assert status(E=129, off=C._offsets([0] * 130)) == 1 and status(E=2, off=C._offsets([0, 3, 2])) == 1
    assert status(E=2, off=C._offsets([0, 0, 0])) == 1
