"""Accuracy of the block fixed-point kernels away from links and fields of order one."""

import numpy as np
import pytest

from oracle import dirac, evenodd, force as oforce, md as omd
from oracle.dirac import PLANES, dagger, sigma
from oracle.lattice import parity
from paper_0910_0262_gb300 import synth
from gpu_util import require_gpu, to_dev, to_np, rel_l2, rand_eo

pytestmark = pytest.mark.gpu
KAPPA, CSW = 0.12, 1.0
LONG = np.clongdouble


def _context(dims, eps=0.2, seed=3):
    from paper_0910_0262_gb300.qcd import CloverWilson
    U = synth.make_problem(dims, eps, seed)[0]
    op = CloverWilson(dims, -1.0)
    op.load_gauge(to_dev(U))
    op.clover_build(KAPPA, CSW)
    return U, op


def chiral_errors(dims=(6, 4, 4, 6), ratio=2.0 ** -20, small=1, n=3):
    """Relative 2-norm errors of (A x, A^-1 x) per chiral block where one block of x is `ratio` times the other."""
    U, op = _context(dims)
    ref = evenodd.SchurOperator(U, KAPPA, CSW, -1.0)
    x = rand_eo(n, ref.A_ee.shape[0], np.random.default_rng(5))
    x[:, :, 2 * small:2 * small + 2] *= ratio
    out = []
    for o, A in ((4, ref.A_ee), (5, ref.A_oo_inv)):
        got = to_np(op.dslash(to_dev(x), o, precision=64))
        want = np.stack([ref.site(A, v) for v in x])
        out += [rel_l2(got[:, :, 2 * b:2 * b + 2], want[:, :, 2 * b:2 * b + 2]) for b in range(2)]
    op.close()
    return out


@pytest.mark.parametrize("small", [0, 1])
@pytest.mark.parametrize("bits", [20, 70])
def test_chiral_blocks_of_very_different_size(bits, small):
    """A and A^-1 do not mix the two chiral blocks of a site: each block of the result is right to its own size
    (a row sums 6 products, as test_operators states for blocks of like size: 1e-15)."""
    require_gpu()
    assert max(chiral_errors(ratio=2.0 ** -bits, small=small)) < 1e-15


@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_non_finite_block_leaves_the_other(value):
    """A and A^-1 of a site with a non-finite component: its chiral block is non-finite, the other as without it."""
    require_gpu()
    U, op = _context((4, 4, 2, 6))
    x = rand_eo(1, U.size // 72, np.random.default_rng(7))
    for o in (4, 5):
        clean = to_np(op.dslash(to_dev(x), o, precision=64))[0]
        y = x.copy()
        y[0, 9, 1, 2] = value
        got = to_np(op.dslash(to_dev(y), o, precision=64))[0]
        assert not np.isfinite(got[9, :2]).any() and np.array_equal(got[9, 2:], clean[9, 2:])
        assert np.array_equal(np.delete(got, 9, 0), np.delete(clean, 9, 0))
    op.close()


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (4, 4, 4, 6)], ids=["8", "192"])
def test_conversion_to_fp32(dims):
    """Canonical fields to FP32 as the hardware rounds them (to nearest even), at every end of the range: with c_sw = 0
    the clover operator is one.  8 and 192 sites: part of a block of 128, and one and a half."""
    require_gpu()
    from paper_0910_0262_gb300.qcd import CloverWilson
    U = synth.make_problem(dims, 0.2, 3)[0]
    op = CloverWilson(dims, -1.0)
    op.load_gauge(to_dev(U))
    op.clover_build(KAPPA, 0.0)
    vh = int(np.prod(dims)) // 2
    rng = np.random.default_rng(2)
    f = np.float32
    ends = [0.0, -0.0, 1.0, 1 + 2.0 ** -24, 1 + 3 * 2.0 ** -24, 2.0 ** -126, 2.0 ** -126 * (1 - 2.0 ** -25), 2.0 ** -149, 2.0 ** -150,
            1e-40, 1e-300, 5e-324, float(np.finfo(f).max), 2.0 ** 127, np.nextafter(2.0 ** 128 * (1 - 2.0 ** -25), 0)]
    x = rng.choice(ends, (1, vh, 4, 3)) * rng.choice([1, -1], (1, vh, 4, 3)) + 1j * rng.standard_normal((1, vh, 4, 3)) * 2.0 ** rng.integers(-30, 30, (1, vh, 4, 3))
    got = to_np(op.dslash(to_dev(x), 4, precision=32))
    with np.errstate(over="ignore"):
        want = x.real.astype(f) + 1j * x.imag.astype(f).astype(float)
    assert np.array_equal(got.real, want.real.astype(float)) and np.array_equal(got.imag, want.imag)
    for v in (1e39, -1e300, np.inf, np.nan):  # not in the range
        y = x.copy()
        y[0, 1, 0, 0] = v
        got = to_np(op.dslash(to_dev(y), 4, precision=32))
        assert not np.isfinite(got[0, 1, 0, 0]) and np.array_equal(np.delete(got, 1, 1), np.delete(want, 1, 1))
    op.close()


def hop_bias(dims=(6, 10, 2, 18), n=8):
    """(mean signed error of D_eo x over all components, 2^-57 times the mean of a site's bound 2^e)."""
    U, op = _context(dims)
    ref = evenodd.SchurOperator(U, KAPPA, CSW, -1.0)
    x = rand_eo(n, ref.A_ee.shape[0], np.random.default_rng(21))
    err = to_np(op.dslash(to_dev(x), 0, precision=64)) - np.stack([ref.D_eo(v) for v in x])
    op.close()
    bound = 2.0 ** np.ceil(np.log2(np.maximum(np.abs(x.real), np.abs(x.imag)).max(axis=(2, 3)))).mean()
    return max(abs(err.real.mean()), abs(err.imag.mean())), bound * 2.0 ** -57


def test_hops_are_rounded_without_bias():
    """Values cut off instead of rounded would move every component down by up to 2^-54 of a site's bound."""
    require_gpu()
    got, most = hop_bias()
    assert got < most


def rel(got, want):
    d = (got - want).reshape(-1)
    return float(np.sqrt((np.abs(d) ** 2).sum() / (np.abs(want.reshape(-1)) ** 2).sum()))


def many_rhs_error(n, dims=(4, 2, 2, 4)):
    """Relative 2-norm error of the force of n solutions."""
    U, op = _context(dims)
    ref = evenodd.SchurOperator(U, KAPPA, CSW, -1.0)
    x = rand_eo(n, ref.A_ee.shape[0], np.random.default_rng(31))
    want = np.zeros(U.shape, dtype=LONG)
    for v in x:
        want += oforce.gradient(ref, v)
    want = oforce.lie_force(U.astype(LONG), want)
    got = to_np(op.fermion_force(to_dev(x), input_is_solution=True)[0])
    op.close()
    return rel(got, want)


@pytest.mark.parametrize("n", [1, 8, 64, 200])
def test_force_of_many_right_hand_sides(n):
    """The error of a sum over right-hand sides does not grow with their number: 1e-15, a few times the 2^-53 of
    the results' last rounding and the oracle's own (the FP64 kernels: 5.2e-16 for one, 3.1e-16 for 200)."""
    require_gpu()
    assert many_rhs_error(n) < 1e-15


def _inverse(A):
    X = np.linalg.inv(A.astype(complex)).astype(LONG)
    one = np.eye(A.shape[-1], dtype=LONG)
    for _ in range(3):
        X = X @ (2 * one - A @ X)
    return X


def det_force(U):
    """The force of S_det = -2 sum_{x odd} log det A(x) (oracle.cloverdet) in long double."""
    U = U.astype(LONG)
    lat = U.shape[:4]
    A = np.zeros(lat + (4, 3, 4, 3), dtype=LONG)
    A += np.einsum('st,ab->satb', np.eye(4), np.eye(3))
    for mu, nu in PLANES:
        A -= LONG(KAPPA) * CSW * np.einsum('st,...ab->...satb', sigma(mu, nu), dirac.field_strength(U, mu, nu))
    inv = _inverse(A.reshape(lat + (12, 12))).reshape(lat + (4, 3, 4, 3))
    dims = (lat[3], lat[2], lat[1], lat[0])
    odd = (parity(dims) == 1)[..., None, None]
    G = np.zeros(U.shape, dtype=LONG)
    for mu, nu in PLANES:
        B = np.einsum('...satb,ts->...ab', inv, sigma(mu, nu))
        B = B - np.trace(B, axis1=-2, axis2=-1)[..., None, None] * np.eye(3) / LONG(3)
        C = odd * (-1j * (LONG(KAPPA) * CSW / 4) * (B + dagger(B)))
        for path in dirac.leaf_paths(mu, nu):
            oforce.insert(G, U, path, C)
    return oforce.lie_force(U, G)


def gauge_force(U, beta):
    U = U.astype(LONG)
    G = np.zeros(U.shape, dtype=LONG)
    C = np.broadcast_to(-LONG(beta) / 3 * np.eye(3, dtype=LONG), U.shape[:4] + (3, 3))
    for mu, nu in PLANES:
        oforce.insert(G, U, omd.plaquette_paths(mu, nu), C)
    return oforce.lie_force(U, G)


def weak_errors(eps, dims=(4, 4, 2, 6)):
    """Relative 2-norm errors on links exp(i eps H) of the gauge force and of the determinant force's off-diagonal
    colours (its diagonal holds differences of the diagonal of A^-1, close to one, in FP64 kernels too)."""
    U, op = _context(dims, eps)
    g = rel(to_np(op.gauge_force(5.6)), gauge_force(U, 5.6))
    off = 1 - np.eye(3)
    d = rel(off * to_np(op.fermion_force(None, clover_det=True)[0]), off * det_force(U))
    op.close()
    return g, d


@pytest.mark.parametrize("eps", [1.0, 0.2, 0.1, 0.05, 1e-2, 1e-3, 1e-6])
def test_forces_on_weak_fields(eps):
    """The forces depend on what links differ from one by, which FP64 products keep to their own size: the
    errors, relative to the force, do not grow as the field gets weak.  (The FP64 kernels give 1.3e-16 and
    1.0 to 1.2e-15 at every eps, the latter from A^-1.)"""
    require_gpu()
    g, d = weak_errors(eps)
    assert g < 2e-16 and d < 2e-15


def test_forces_where_weak_and_strong_links_meet():
    """One half of the lattice at eps 1e-3, the other at 0.3: each half's force is right to its own size (the
    links two sites into it, which no strong link reaches)."""
    require_gpu()
    dims = (2, 4, 2, 12)
    U = synth.make_problem(dims, 1e-3, 3)[0]
    U[6:] = synth.make_problem(dims, 0.3, 4)[0][6:]
    _, op = _context(dims)
    op.load_gauge(to_dev(U))
    op.clover_build(KAPPA, CSW)
    got = to_np(op.gauge_force(5.6)), to_np(op.fermion_force(None, clover_det=True)[0])
    op.close()
    want = gauge_force(U, 5.6), det_force(U)
    off = 1 - np.eye(3)
    for part in (slice(2, 4), slice(8, 10)):
        assert rel(got[0][part], want[0][part]) < 1e-15
        assert rel(off * got[1][part], off * want[1][part]) < 4e-15
