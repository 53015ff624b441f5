"""The fixed-point tile of eri_batch where its scales are tight: one-centre
quartets whose scale bound is attained, at powers of two."""
import numpy as np
import pytest

import paper_2506_12501_gb300 as eri
import synth
from gpu_helpers import assert_close, oracle_blocks, to_device

pytestmark = pytest.mark.gpu


def _shells(atoms, l, exps, rng):
    return [(a, l, list(z), list(rng.uniform(0.5, 1.0, len(z)) * synth.norm_coef(np.asarray(z), l)))
            for a, z in zip(atoms, exps)]


@pytest.mark.parametrize("N,cls", [(0, (1, 0, 1, 0)), (6, (2, 1, 2, 1)), (8, (2, 2, 2, 2))])
def test_one_centre_bounds_at_powers_of_two(N, cls):
    """One-centre quartets whose order-N integral at the largest exponents, (N-1)!!/(N+1) sqrt(rho) in units of
    s = 1.1 sqrt(2 rho), attains the scale's bound at a power of two, to the rounding of a float on either side."""
    rng = np.random.default_rng(N)
    c = np.prod(np.arange(1, N, 2)) / (N + 1) / (1.1 * 1.00001) ** N
    nq = 10240
    bra, ket, q = np.array([[0, 1]], np.int32), np.array([[2, 3]], np.int32), np.zeros((nq, 2), np.int64)
    b, k, qq = to_device(bra, ket, q)
    eri.eri_set_forms(1)
    try:
        for _ in range(100):
            rho = (2.0 ** rng.integers(-2, 3) / c) ** 2 * (1 + rng.uniform(0, 2.5e-7))
            zb = rho * (1 + 10 ** rng.uniform(-1, 1))
            zk = 1 / (1 / rho - 1 / zb)
            exps = [(0.5 * z, 0.4 * z) for z in (zb, zb, zk, zk)]
            basis = synth.basis_from_shells(rng.uniform(-1, 1, (1, 3)), sum((_shells([0], l, [e], rng)
                                                                            for l, e in zip(cls, exps)), []))
            out = eri.eri_batch(cls, eri.DeviceBasis(basis), b, k, qq).cpu().numpy().reshape(-1, nq).T
            ref = oracle_blocks(cls, basis, bra, ket, q[:1])
            assert_close(out[:1], ref, atol=1e-12 * np.abs(ref).max(), what=f"zeta {zb!r} {zk!r}")
            np.testing.assert_array_equal(out[1:], out[:-1])
    finally:
        eri.eri_set_forms(0)
