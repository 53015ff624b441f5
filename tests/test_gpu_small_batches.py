"""Tile shapes of batches too small to be timed, against the oracle: one
quartet, about one per SM, several per SM, and the last size below the timing."""
import numpy as np
import pytest

import paper_2506_12501_gb300 as eri
import synth
from gpu_helpers import assert_close, oracle_blocks, to_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nq", [1, 153, 1217, 16383])
@pytest.mark.parametrize("cls,K", [((0, 0, 0, 0), 3), ((1, 0, 1, 0), 3), ((1, 1, 1, 1), 1), ((2, 2, 2, 2), 2), ((3, 3, 1, 1), 1)])
def test_small_batch_tiles(cls, K, nq):
    basis, pools = synth.class_sweep_pools(seed=21, lmax=max(cls), pool=30, K=K, cube=3.0)
    bra, ket, q = synth.class_sweep_batch(pools, cls, seed=22, npairs=40, nq=nq)
    b, k, qq = to_device(bra, ket, q)
    db = eri.DeviceBasis(basis)
    pick = np.unique(np.r_[0:min(nq, 6), max(nq - 6, 0):nq])
    ref = oracle_blocks(cls, basis, bra, ket, q[pick])
    for form in (0, 1, 2, 4, 8):
        eri.eri_set_forms(form)
        try:
            out = eri.eri_batch(cls, db, b, k, qq).cpu().numpy().reshape(-1, nq).T
        finally:
            eri.eri_set_forms(0)
        assert_close(out[pick], ref, what=f"{cls} K={K} nq={nq} form {form}")
