"""Pair tables formed by a warp per slot and by a thread per slot: the same
arithmetic, so the same blocks bit for bit on both sides of the rule, and the
oracle's."""
import numpy as np
import pytest

import paper_2506_12501_gb300 as eri
import synth
from gpu_helpers import assert_close, oracle_blocks, to_device

pytestmark = pytest.mark.gpu


# limit: the last number of bra pairs that take warps, 640 sqrt(terms) slots for 33 and 1920 terms
@pytest.mark.parametrize("cls,K,limit", [((1, 1, 0, 0), 1, 3676), ((1, 1, 1, 0), 3, 3676 // 9), ((3, 3, 0, 0), 1, 28043)])
def test_warp_and_thread_tables_agree(cls, K, limit):
    basis, pools = synth.class_sweep_pools(seed=11, lmax=max(cls), pool=40, K=K, cube=3.0)
    bra, ket, _ = synth.class_sweep_batch(pools, cls, seed=12, npairs=37, nq=1)
    db = eri.DeviceBasis(basis)
    q = np.stack([np.arange(37), np.arange(37) % len(ket)], 1).astype(np.int64)
    ref = oracle_blocks(cls, basis, bra, ket, q)
    eri.eri_set_forms(1)
    try:
        got = []
        for n in (37, limit, limit + 1):  # the last one past the rule; the 37 pairs at the end of the list
            rows = np.concatenate([np.tile(bra, (n // 37 + 1, 1))[:n - 37], bra]).astype(np.int32)
            b, k, qq = to_device(rows, ket, q + np.array([n - 37, 0]))
            got.append(eri.eri_batch(cls, db, b, k, qq).cpu().numpy().reshape(-1, 37).T)
    finally:
        eri.eri_set_forms(0)
    assert_close(got[0], ref, what=f"{cls} K={K}")
    for g in got[1:]:
        np.testing.assert_array_equal(g, got[0])
