"""Accuracy of the block fixed-point kernels away from links and fields of order one."""

import numpy as np
import pytest

from oracle import evenodd, force as oforce
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
