"""The fixed-point tile of eri_batch (contracted 4-centre classes in large
batches) against the oracle: ket primitive counts on both sides of the folds
and pairs of its sums, mixed contraction degrees, every order of the auxiliary
integrals it takes, both list forms and the solid-harmonic output."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

import paper_2506_12501_gb300 as eri
import synth
from gpu_helpers import assert_close, nc, oracle_blocks, to_device

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _wherever_it_can():
    """The fixed-point tile wherever its precision allows, whatever would be faster."""
    eri.eri_set_fixed(eri.ERI_FIXED_ALWAYS)
    yield
    eri.eri_set_fixed(eri.ERI_FIXED_RULE)

# class, primitives per shell: K_ket = 4 (even), 9 (odd), 16 (past one fold), 25 and 36 for s shells (several
# folds); L = 1..6 in fixed point, 7 and 8 in FP64; a component-pair list of one column, pairs and single columns
CASES = [((1, 0, 0, 0), 2), ((0, 1, 1, 0), 3), ((1, 1, 1, 0), 4), ((1, 1, 1, 1), 3), ((2, 1, 1, 1), 3),
         ((2, 1, 2, 1), 2), ((2, 2, 2, 1), 2), ((2, 2, 2, 2), 2), ((1, 0, 1, 0), 5), ((0, 0, 1, 0), 6), ((3, 1, 2, 0), 2)]


def _sample_error(got, ref):
    """Relative 2-norm error; the oracle's double build and the FP64 tile agree to a few 1e-15, times the
    recursion forms' magnification (below 10 on these pairs)."""
    return np.linalg.norm(got - ref) / np.linalg.norm(ref)


@pytest.mark.parametrize("cls,K", CASES)
def test_fixed_tile_against_oracle(cls, K):
    nq = max(2003, 150000 // K ** 4 + 7)  # odd: the last tile is ragged
    basis, pools = synth.class_sweep_pools(seed=3, lmax=max(cls), pool=64, K=K, cube=4.0)
    bra, ket, q = synth.class_sweep_batch(pools, cls, seed=4, npairs=50, nq=nq)
    b, k, qq = to_device(bra, ket, q)
    db = eri.DeviceBasis(basis)
    for form in (0, 1, 2, 3):
        eri.eri_set_forms(1 << form)
        try:
            out = eri.eri_batch(cls, db, b, k, qq).cpu().numpy().reshape(-1, nq).T
            assert eri.eri_last_arithmetic() == (eri.ERI_ARITH_FIXED if sum(cls) <= 6 else eri.ERI_ARITH_FP64)
        finally:
            eri.eri_set_forms(0)
        pick = np.r_[0:12, nq - 12:nq]
        ref = oracle_blocks(cls, basis, bra, ket, q[pick])
        assert_close(out[pick], ref, what=f"{cls} K={K} form {form}")
        assert _sample_error(out[pick], ref) < 2e-14


def test_fixed_tile_mixed_degrees_product_form_and_sph():
    cls = (1, 0, 1, 1)
    rng = np.random.default_rng(5)
    shells, centres = [], rng.uniform(0, 3.0, (90, 3))
    for i in range(90):
        l, K = (1, 0)[i % 2], (1, 2, 3, 5)[i % 4]
        z = 0.3 * 2.0 ** np.arange(K)
        shells.append((i, l, list(z), list(rng.uniform(0.5, 1, K) * synth.norm_coef(z, l))))
    basis = synth.basis_from_shells(centres, shells)
    p, s = np.arange(0, 90, 2), np.arange(1, 90, 2)
    bra = np.stack([rng.choice(p, 61), rng.choice(s, 61)], 1).astype(np.int32)
    ket = np.stack([rng.choice(p, 53), rng.choice(p, 53)], 1).astype(np.int32)
    b, k, _ = to_device(bra, ket)
    db = eri.DeviceBasis(basis)
    nab, ncd = 3, 9
    out = eri.eri_batch(cls, db, b, k).cpu().numpy().reshape(53, ncd, nab, 61)
    assert eri.eri_last_arithmetic() == eri.ERI_ARITH_FIXED
    q = np.array([(i, j) for i in range(0, 61, 7) for j in range(0, 53, 6)])
    ref = oracle_blocks(cls, basis, bra, ket, q).reshape(len(q), nab, ncd)
    got = np.stack([out[j, :, :, i].T for i, j in q])
    assert_close(got, ref, what="product form, mixed degrees")
    sph = eri.eri_batch_sph(cls, db, b, k).cpu().numpy().reshape(53, ncd, nab, 61)
    assert eri.eri_last_arithmetic() == eri.ERI_ARITH_FIXED
    # p functions in solid harmonics: m = -1, 0, 1 are y, z, x
    order = np.array([1, 2, 0])
    cd = (order[:, None] * 3 + order[None, :]).reshape(-1)
    assert_close(np.stack([sph[j, :, :, i].T for i, j in q]), ref[:, order][:, :, cd], what="solid harmonics")


def test_fixed_tile_far_and_coincident_centres():
    """Boys arguments of every range: coincident centres (T = 0) to far apart (T of thousands)."""
    cls, K, nq = (1, 1, 1, 0), 3, 4000
    rng = np.random.default_rng(6)
    centres = np.concatenate([np.zeros((20, 3)), rng.uniform(-1, 1, (20, 3)), rng.uniform(-60, 60, (20, 3))])
    shells = []
    for l in (0, 1):
        for i in range(60):
            z = 0.2 * 3.0 ** np.arange(K)
            shells.append((i, l, list(z), list(rng.uniform(0.5, 1, K) * synth.norm_coef(z, l))))
    basis = synth.basis_from_shells(centres, shells)
    near = np.array([(60 + i, 60 + j) for i in range(60) for j in (i, (i + 1) % 20)], np.int32)
    ket = np.array([(60 + i, j) for i in range(60) for j in (i, (i + 3) % 20)], np.int32)
    q = np.stack([rng.integers(0, len(near), nq), rng.integers(0, len(ket), nq)], 1)
    b, k, qq = to_device(near, ket, q)
    out = eri.eri_batch(cls, eri.DeviceBasis(basis), b, k, qq).cpu().numpy().reshape(-1, nq).T
    assert eri.eri_last_arithmetic() == eri.ERI_ARITH_FIXED
    ref = oracle_blocks(cls, basis, near, ket, q[:400])
    assert_close(out[:400], ref, what="centres of every distance")


def test_wide_exponents_and_non_finite_primitives_keep_the_fp64_tile():
    """Pairs whose exponents spread too far, and primitives out of the fixed-point range, give what they gave."""
    cls, nq = (1, 1, 1, 1), 4000
    basis, pools = synth.class_sweep_pools(seed=8, lmax=1, pool=32, K=2, cube=3.0,
                                           exps_fn=lambda rng, K: np.array([0.05, 900.0]))
    bra, ket, q = synth.class_sweep_batch(pools, cls, seed=9, npairs=40, nq=nq)
    b, k, qq = to_device(bra, ket, q)
    out = eri.eri_batch(cls, eri.DeviceBasis(basis), b, k, qq).cpu().numpy().reshape(-1, nq).T
    assert eri.eri_last_arithmetic() == eri.ERI_ARITH_FP64
    assert_close(out[:60], oracle_blocks(cls, basis, bra, ket, q[:60]), what="wide exponents")
    basis, pools = synth.class_sweep_pools(seed=8, lmax=1, pool=32, K=3, cube=3.0)
    basis.coefs[basis.shell_off[bra[0, 0]]] = np.nan
    out = eri.eri_batch(cls, eri.DeviceBasis(basis), b, k, qq).cpu().numpy().reshape(-1, nq).T
    assert eri.eri_last_arithmetic() == eri.ERI_ARITH_FP64
    bad = np.any(bra[q[:, 0]] == bra[0, 0], axis=1) | np.any(ket[q[:, 1]] == bra[0, 0], axis=1)
    assert bad.any() and np.isnan(out[bad]).all() and np.isfinite(out[~bad]).all()


@pytest.mark.parametrize("cls,ratio,fixed", [((2, 2, 2, 1), 3.0, True), ((2, 2, 2, 2), 3.0, True), ((3, 2, 1, 1), 3.0, True),
                                             ((1, 1, 1, 1), 60.0, True), ((3, 2, 2, 2), 3.0, False),
                                             ((1, 1, 1, 1), 70.0, False)])
def test_wide_pairs_admit_order_eight_and_six_bits(cls, ratio, fixed):
    """Pairs of centres up to 20 bohr apart: the tile takes order 8 and 6 bits of spread, where its error over the
    batch is no larger than the FP64 tile's in the form that runs (to 1.3 for the samples of 120 blocks)."""
    nq = 16384
    basis, pools = synth.class_sweep_pools(seed=25, lmax=max(cls), pool=64, K=2, cube=12.0,
                                           exps_fn=lambda rng, K: 0.2 * np.array([1.0, ratio]))
    bra, ket, q = synth.class_sweep_batch(pools, cls, seed=26, npairs=60, nq=nq)
    b, k, qq = to_device(bra, ket, q)
    db = eri.DeviceBasis(basis)
    ref = oracle_blocks(cls, basis, bra, ket, q[:120], prec="ld")
    error = []
    for mode in (eri.ERI_FIXED_ALWAYS, eri.ERI_FIXED_NEVER):
        eri.eri_set_fixed(mode)
        out = eri.eri_batch(cls, db, b, k, qq).cpu().numpy().reshape(-1, nq).T
        assert eri.eri_last_arithmetic() == (eri.ERI_ARITH_FIXED if fixed and not error else eri.ERI_ARITH_FP64)
        error.append(_sample_error(out[:120], ref))
    assert error[0] <= 1.3 * error[1], error


@pytest.mark.parametrize("ratio,fixed", [(30.0, True), (34.0, False), (60.0, False)])
def test_spread_beyond_five_bits_keeps_the_fp64_tile(ratio, fixed):
    """(pp|pp), K = 2: a pair's exponents spread by log2(ratio) = 4.9, 5.1 and 5.9 bits, in a small cube, where spread
    costs most (at 5.9 bits the fixed-point tile's error was four times the FP64 tile's 5e-16)."""
    cls, nq = (1, 1, 1, 1), 10240
    basis, pools = synth.class_sweep_pools(seed=23, lmax=1, pool=32, K=2, cube=1.5,
                                           exps_fn=lambda rng, K: 0.2 * np.array([1.0, ratio]))
    bra, ket, q = synth.class_sweep_batch(pools, cls, seed=24, npairs=60, nq=nq)
    b, k, qq = to_device(bra, ket, q)
    eri.eri_set_forms(1)
    try:
        out = eri.eri_batch(cls, eri.DeviceBasis(basis), b, k, qq).cpu().numpy().reshape(-1, nq).T
    finally:
        eri.eri_set_forms(0)
    assert eri.eri_last_arithmetic() == (eri.ERI_ARITH_FIXED if fixed else eri.ERI_ARITH_FP64)
    assert _sample_error(out[:240], oracle_blocks(cls, basis, bra, ket, q[:240], prec="ld")) < 1e-15


@pytest.mark.parametrize("cls", [(3, 2, 1, 1), (2, 2, 2, 1), (3, 3, 1, 1), (3, 2, 2, 2), (3, 2, 3, 2)])
def test_orders_above_six_keep_the_fp64_tile(cls):
    """Contracted classes of order 7 to 10, centres within 7 bohr: FP64 tile, whose error in the plain form stays near
    1e-15 on these pairs (in fixed point it was up to 3.4 times that at order 7 and 8, 1e-14 above)."""
    nq = 9382
    basis, pools = synth.class_sweep_pools(seed=3, lmax=3, pool=64, K=2, cube=4.0)
    bra, ket, q = synth.class_sweep_batch(pools, cls, seed=4, npairs=50, nq=nq)
    b, k, qq = to_device(bra, ket, q)
    eri.eri_set_forms(1)
    try:
        out = eri.eri_batch(cls, eri.DeviceBasis(basis), b, k, qq).cpu().numpy().reshape(-1, nq).T
    finally:
        eri.eri_set_forms(0)
    assert eri.eri_last_arithmetic() == eri.ERI_ARITH_FP64
    assert _sample_error(out[:24], oracle_blocks(cls, basis, bra, ket, q[:24], prec="ld")) < 5e-15


@pytest.mark.parametrize("cls,K,nq", [((1, 1, 1, 0), 3, 20011), ((2, 1, 1, 1), 3, 16384), ((2, 2, 1, 1), 2, 16385)])
def test_timed_tiles_and_form_against_oracle(cls, K, nq):
    """Batches long enough to be timed: the tile shape and the form come from the timing; the second call, which
    uses what the first remembered, gives the same bits."""
    basis, pools = synth.class_sweep_pools(seed=13, lmax=max(cls), pool=64, K=K, cube=4.0)
    bra, ket, q = synth.class_sweep_batch(pools, cls, seed=14, npairs=50, nq=nq)
    b, k, qq = to_device(bra, ket, q)
    db = eri.DeviceBasis(basis)
    out = []
    for _ in range(2):
        out.append(eri.eri_batch(cls, db, b, k, qq).cpu().numpy().reshape(-1, nq).T)
        assert eri.eri_last_arithmetic() == eri.ERI_ARITH_FIXED
    pick = np.r_[0:12, nq // 2:nq // 2 + 12, nq - 12:nq]
    assert_close(out[0][pick], oracle_blocks(cls, basis, bra, ket, q[pick]), what=f"{cls} K={K}")
    np.testing.assert_array_equal(out[0], out[1])


def test_callers_choice_of_the_fp64_tile():
    """ERI_FIXED_NEVER keeps this thread's batches on the FP64 tile; both agree to round-off."""
    cls, nq = (1, 1, 1, 0), 4001
    basis, pools = synth.class_sweep_pools(seed=15, lmax=1, pool=32, K=3, cube=4.0)
    bra, ket, q = synth.class_sweep_batch(pools, cls, seed=16, npairs=40, nq=nq)
    b, k, qq = to_device(bra, ket, q)
    db = eri.DeviceBasis(basis)
    fixed = eri.eri_batch(cls, db, b, k, qq).cpu().numpy()
    assert eri.eri_last_arithmetic() == eri.ERI_ARITH_FIXED
    assert eri.eri_set_fixed(eri.ERI_FIXED_NEVER) == eri.ERI_FIXED_ALWAYS
    fp64 = eri.eri_batch(cls, db, b, k, qq).cpu().numpy()
    assert eri.eri_last_arithmetic() == eri.ERI_ARITH_FP64
    assert_close(fixed, fp64, what="fixed point against FP64")
    assert not np.array_equal(fixed, fp64)


@pytest.mark.parametrize("cls,K,ratio,nq,fixed", [
    ((1, 1, 1, 0), 2, 3.0, 16383, False), ((2, 1, 2, 1), 2, 3.0, 9400, False),  # few primitive quartets, not timed
    ((2, 2, 0, 0), 3, 2.0, 2000, False), ((1, 0, 0, 0), 3, 2.0, 4000, False),  # the models
    ((1, 1, 1, 1), 3, 2.0, 8000, True), ((2, 1, 1, 1), 4, 1.5, 4000, True),
    ((3, 3, 0, 0), 2, 3.0, 20000, False),  # timed against the FP64 tile
    ((1, 1, 1, 0), 3, 2.0, 20000, True)])
def test_rule_takes_the_faster_tile(cls, K, ratio, nq, fixed):
    """Batches on which the two tiles' times differ by a tenth and more: the rule, and the timing, pick the faster."""
    eri.eri_set_fixed(eri.ERI_FIXED_RULE)
    basis, pools = synth.class_sweep_pools(seed=3, lmax=max(cls), pool=256, K=K,
                                           exps_fn=lambda rng, k: 0.2 * ratio ** np.arange(k))
    bra, ket, q = synth.class_sweep_batch(pools, cls, seed=4, npairs=1024, nq=nq)
    b, k, qq = to_device(bra, ket, q)
    db = eri.DeviceBasis(basis)
    for _ in range(2):
        out = eri.eri_batch(cls, db, b, k, qq)
        assert eri.eri_last_arithmetic() == (eri.ERI_ARITH_FIXED if fixed else eri.ERI_ARITH_FP64)
    pick = np.r_[0:6, nq - 6:nq]
    got = out.cpu().numpy().reshape(-1, nq).T[pick]
    assert_close(got, oracle_blocks(cls, basis, bra, ket, q[pick]), what=f"{cls} K={K}")


# in a process of its own: the library keeps its tables and workspace
_MEMORY = """
import sys
import numpy as np
import torch
import paper_2506_12501_gb300 as eri
import synth
from gpu_helpers import assert_close, nc, oracle_blocks, to_device

npairs, leave = int(sys.argv[1]), int(sys.argv[2])
cls, K, nq = (2, 1, 1, 0), 3, 10240
basis, pools = synth.class_sweep_pools(seed=17, lmax=2, pool=32, K=K, cube=4.0,
                                       exps_fn=lambda rng, K: 0.3 * 1.5 ** np.arange(K))
bra, ket, q = synth.class_sweep_batch(pools, cls, seed=18, npairs=64, nq=nq)
b, k, qq = to_device(np.tile(bra, (npairs // 64, 1)), ket, q)
db = eri.DeviceBasis(basis)
out = torch.empty(nq * nc(2) * nc(1) * nc(1), dtype=torch.float64, device="cuda")
eri.eri_set_forms(1)
if leave < 1 << 30:  # the FP64 tile's tables are there already
    eri.eri_set_fixed(eri.ERI_FIXED_NEVER)
    eri.eri_batch(cls, db, b, k, qq, out=out)
eri.eri_set_fixed(eri.ERI_FIXED_ALWAYS)
torch.cuda.synchronize()
held = torch.empty(torch.cuda.mem_get_info()[0] - leave, dtype=torch.uint8, device="cuda")
eri.eri_batch(cls, db, b, k, qq, out=out)
assert eri.eri_last_arithmetic() == eri.ERI_ARITH_FP64
del held
torch.cuda.empty_cache()
got = out.cpu().numpy().reshape(-1, nq).T
eri.eri_batch(cls, db, b, k, qq, out=out)
assert eri.eri_last_arithmetic() == eri.ERI_ARITH_FIXED
assert_close(out.cpu().numpy().reshape(-1, nq).T, got)
assert_close(got[:16], oracle_blocks(cls, basis, bra, ket, q[:16]))
print("memory: ok")
"""


@pytest.mark.parametrize("what,npairs,leave", [("Boys rows", 64, 6 << 20), ("pair tables", 260_032, 4 << 30)])
def test_memory_for_the_fp64_tile_is_enough(what, npairs, leave):
    """Where the fixed-point tile's tables find no memory, the batch runs on the FP64 tile, which needs less."""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    env = dict(os.environ, PYTHONPATH=os.pathsep.join([root, os.path.join(root, "tests")]))
    r = subprocess.run([sys.executable, "-c", _MEMORY, str(npairs), str(leave)], cwd=root, env=env,
                       capture_output=True, text=True, timeout=300)
    assert "memory: ok" in r.stdout, what + r.stderr[-2000:]
