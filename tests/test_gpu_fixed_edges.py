"""The fixed-point tile of eri_batch where its scales are tight: one-centre
quartets whose scale bound is attained at powers of two, tight pairs against
diffuse ones, multipoles at a distance, and its error beside the FP64 tile's."""
import numpy as np
import pytest

import oracle
import paper_2506_12501_gb300 as eri
import synth
from gpu_helpers import THREADS, assert_close, oracle_blocks, to_device

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _wherever_it_can():
    """The fixed-point tile wherever its precision allows, whatever would be faster."""
    eri.eri_set_fixed(eri.ERI_FIXED_ALWAYS)
    yield
    eri.eri_set_fixed(eri.ERI_FIXED_RULE)


def _shells(atoms, l, exps, rng):
    return [(a, l, list(z), list(rng.uniform(0.5, 1.0, len(z)) * synth.norm_coef(np.asarray(z), l)))
            for a, z in zip(atoms, exps)]


@pytest.mark.parametrize("N,cls", [(0, (1, 0, 1, 0)), (6, (2, 1, 2, 1))])
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


def _column_errors(got, ref):
    """Relative 2-norm error of every component quadruple over the quartets, where it is not zero by symmetry."""
    top = np.sqrt((ref ** 2).sum(axis=0))
    on = top > 1e-40
    return (np.sqrt(((got - ref) ** 2).sum(axis=0))[on] / top[on]).astype(float)


def _reference(cls, basis, bra, ket, q):
    """The long double oracle's blocks, in long double."""
    ref = oracle.eri_quartets(basis, synth.quartet_shells(bra, ket, q), prec="ld", threads=THREADS)
    return ref.reshape(len(q), -1)


def _both_tiles(cls, basis, bra, ket, q, n):
    """The first n quartets' integrals from the fixed-point and the FP64 tile, and the oracle's."""
    b, k, qq = to_device(bra, ket, q)
    db = eri.DeviceBasis(basis)
    out = []
    for mode, arithmetic in ((eri.ERI_FIXED_ALWAYS, eri.ERI_ARITH_FIXED), (eri.ERI_FIXED_NEVER, eri.ERI_ARITH_FP64)):
        eri.eri_set_fixed(mode)
        out.append(eri.eri_batch(cls, db, b, k, qq).cpu().numpy().reshape(-1, len(q)).T[:n])
        assert eri.eri_last_arithmetic() == arithmetic
    eri.eri_set_fixed(eri.ERI_FIXED_ALWAYS)
    return out[0], out[1], _reference(cls, basis, bra, ket, q[:n])


@pytest.mark.parametrize("tight", [30.0, 2e3, 1e5])
@pytest.mark.parametrize("cls", [(1, 0, 1, 0), (2, 1, 1, 0), (1, 1, 1, 1), (2, 2, 1, 0)])
def test_tight_one_centre_pairs_against_diffuse_ones(cls, tight):
    """A one-centre pair's columns may start at any Hermite order: each component is as close as from the FP64 tile,
    however far the pair's exponents lie above the other side's.  (Tight pairs at the origin: elsewhere the rounding
    of their centre, 1e-16 of the coordinate, bounds both tiles.)"""
    rng = np.random.default_rng(31)
    n, m, nq = 8, 40, 10240
    centres = np.concatenate([np.zeros((1, 3)), rng.uniform(-3, 3, (m, 3))])
    diffuse = 0.2 * np.array([1.0, 2.0])
    shells = sum((_shells([0] * n, l, [tight * (1 + i / n) * diffuse for i in range(n)], rng) for l in cls[:2]), [])
    shells += sum((_shells(range(1, m + 1), l, [diffuse] * m, rng) for l in cls[2:]), [])
    basis = synth.basis_from_shells(centres, shells)
    i, j = np.arange(n), np.arange(m)
    core = np.stack([i, n + i], 1).astype(np.int32)
    val = np.stack([2 * n + j, 2 * n + m + (j + j % 3) % m], 1).astype(np.int32)  # one- and two-centre pairs
    q = np.stack([np.arange(nq) % n, np.arange(nq) // n % m], 1).astype(np.int64)
    for sides, forms in ((0, 1), (1, 2)):  # the tight pair on the kernel's bra, from either place in the call
        eri.eri_set_forms(forms)
        try:
            if sides == 0:
                fixed, fp64, ref = _both_tiles(cls, basis, core, val, q, n * m)
            else:
                fixed, fp64, ref = _both_tiles(cls[2:] + cls[:2], basis, val, core, q[:, ::-1].copy(), n * m)
        finally:
            eri.eri_set_forms(0)
        # a component: one rounding of each product and sum, twice that for sums of a few hundred terms
        assert _column_errors(fixed, ref).max() < max(2e-14, 2 * _column_errors(fp64, ref).max())


@pytest.mark.parametrize("r", [4.0, 25.0, 90.0])
@pytest.mark.parametrize("cls", [(1, 1, 1, 1), (2, 1, 1, 1), (2, 2, 2, 0)])
def test_one_centre_pairs_at_a_distance(cls, r):
    """Quartets of one-centre pairs, whose integrals are multipoles of any order: each component is as close as from
    the FP64 tile at every distance.  (One side at the origin, the other at coordinates whose weighted means are exact:
    elsewhere the rounding of a centre, 1e-16 of the coordinate, bounds both tiles.)"""
    rng = np.random.default_rng(41)
    n, m, nq = 6, 40, 10240
    u = rng.normal(size=(m, 3))
    far = np.round(8 * r * rng.uniform(1, 1.3, (m, 1)) * u / np.linalg.norm(u, axis=1, keepdims=True)) / 8
    shells = sum((_shells([0] * n, l, [0.3 * np.array([1.0, 2.5]) * (1 + i / n) for i in range(n)], rng)
                  for l in cls[:2]), [])
    shells += sum((_shells(range(1, m + 1), l, [np.array([0.5, 0.5])] * m, rng) for l in cls[2:]), [])
    basis = synth.basis_from_shells(np.concatenate([np.zeros((1, 3)), far]), shells)
    i, j = np.arange(n), np.arange(m)
    bra = np.stack([i, n + i], 1).astype(np.int32)
    ket = np.stack([2 * n + j, 2 * n + m + j], 1).astype(np.int32)
    q = np.stack([np.arange(nq) % n, np.arange(nq) // n % m], 1).astype(np.int64)
    for forms in (1, 2):
        eri.eri_set_forms(forms)
        try:
            fixed, fp64, ref = _both_tiles(cls, basis, bra, ket, q, n * m)
        finally:
            eri.eri_set_forms(0)
        assert _column_errors(fixed, ref).max() < max(2e-14, 2 * _column_errors(fp64, ref).max())


@pytest.mark.parametrize("one_centre", [False, True])
@pytest.mark.parametrize("cls,K", [((1, 0, 1, 0), 3), ((1, 1, 1, 1), 2), ((1, 1, 1, 1), 3), ((2, 1, 1, 1), 2),
                                   ((2, 2, 1, 1), 2), ((2, 1, 2, 1), 2)])
def test_error_no_larger_than_the_fp64_tile(cls, K, one_centre):
    """Relative 2-norm error over a batch against the long double oracle, both tiles in the plain form.  The bound is
    a tenth over 1 for the sample: the means of a few thousand roundings."""
    rng = np.random.default_rng(51)
    m, nq = 24, 10240
    z = 0.2 * 3.0 ** np.arange(K)
    shells = sum((_shells(range(m), l, [z] * m, rng) for l in cls), [])
    basis = synth.basis_from_shells(rng.uniform(0, 4.0, (m, 3)), shells)
    i, j = rng.integers(0, m, (2, 60)), rng.integers(0, m, (2, 60))
    if one_centre:
        i[1], j[1] = i[0], j[0]
    bra, ket = (i.T + [0, m]).astype(np.int32), (j.T + [2 * m, 3 * m]).astype(np.int32)
    q = rng.integers(0, 60, (nq, 2)).astype(np.int64)
    eri.eri_set_forms(1)
    try:
        fixed, fp64, ref = _both_tiles(cls, basis, bra, ket, q, 400)
    finally:
        eri.eri_set_forms(0)
    error = [float(np.sqrt(((x - ref) ** 2).sum())) for x in (fixed, fp64)]
    assert error[0] <= 1.1 * error[1], error
