"""The FP64 operators on block fixed-point integers (near-unitary links) and the FP64 kernels they stand
beside (other links), against the oracle.

Sizes at the edges of the kernels' blocks of 32 sites: 8 and 24 sites per parity (part of one block), 32
and 96 (whole blocks), 40, 72, 120 and 1080 (a ragged last block), with 1, 2, 3, 4 and 5 right-hand sides
(batches 2 + 1 and 4 + 1), where blocks times right-hand sides are no more than the GPU's SMs and the kernel
with a direction per pair of warps runs; and larger ones (test_operators_of_many_blocks) for the kernel with
1, 2 or 4 right-hand sides a block.  Tolerances: a row of an operator sums at most
8 x 6 products of a link and 11 of a clover block, each rounded to 2^-53 in FP64, so 1e-15 in the norm; of
one hopping term, site by site, 16 x 2^-53 of the neighbours' largest values.
"""

import numpy as np
import pytest

from oracle import evenodd
from oracle.lattice import join_eo, split_eo
from paper_0910_0262_gb300 import synth
from gpu_util import require_gpu, to_dev, to_np, rel_l2, rand_eo

gpu = pytest.mark.gpu
DIMS = [(2, 2, 2, 2), (2, 2, 6, 2), (6, 2, 10, 2), (4, 4, 2, 2), (4, 4, 2, 6), (10, 2, 2, 2), (18, 2, 2, 2), (6, 10, 2, 18)]
KAPPA, CSW = 0.12, 1.0


def test_fixed_point_arithmetic():
    """Conversions, limbs and sums of products against exact integers (host evaluation)."""
    from paper_0910_0262_gb300 import build, qcd
    build.build()
    assert qcd.qcd_selftest_fixed() == 0


def _context(dims, t_bc=-1.0, scale=1.0, seed=3, clover=True):
    from paper_0910_0262_gb300.qcd import CloverWilson
    U = synth.make_problem(dims, 0.2, seed)[0] * scale
    op = CloverWilson(dims, t_bc)
    op.load_gauge(to_dev(U))
    if clover:
        op.clover_build(KAPPA, CSW)
    return U, op


@gpu
@pytest.mark.parametrize("t_bc", [-1.0, 1.0])
@pytest.mark.parametrize("dims", DIMS, ids=["x".join(map(str, d)) for d in DIMS])
@pytest.mark.parametrize("scale", [1.0, 1.0 - 4e-6, 1.25], ids=["su3", "near", "far"])
def test_operators(dims, t_bc, scale):
    """scale 1 and 1 - 4e-6: fixed point (links unitary to 1e-5); 1.25: the FP64 kernels."""
    require_gpu()
    U, op = _context(dims, t_bc, scale)
    ref = evenodd.SchurOperator(U, KAPPA, CSW, t_bc)
    rng = np.random.default_rng(11)
    vh = ref.A_ee.shape[0]
    table = {(0, 0): ref.D_eo, (0, 1): ref.D_oe_dag, (1, 0): ref.D_oe, (1, 1): ref.D_eo_dag, (2, 0): ref.Mhat,
             (2, 1): ref.Mhat_dag, (3, 0): ref.MdagM, (4, 0): lambda v: ref.site(ref.A_ee, v),
             (5, 0): lambda v: ref.site(ref.A_oo_inv, v)}
    for n in (1, 2, 3, 4, 5):
        x = rand_eo(n, vh, rng)
        for (o, dag), f in table.items():
            got = to_np(op.dslash(to_dev(x), o, dagger=bool(dag), precision=64))
            assert rel_l2(got, np.stack([f(v) for v in x])) < 1e-15, (n, o, dag)
    op.close()


@gpu
@pytest.mark.parametrize("dims,n", [((6, 10, 2, 18), 8), ((10, 10, 10, 10), 1), ((10, 10, 10, 10), 2), ((10, 10, 10, 10), 4)],
                         ids=["1080_rhs8", "5000_rhs1", "5000_rhs2", "5000_rhs4"])
def test_operators_of_many_blocks(dims, n):
    """34 blocks x 8 right-hand sides (two turns of four, which reuse the block's shared memory) and 157 blocks x 1, 2
    and 4: more than any GPU's SMs this library runs on (152), each with a ragged last block."""
    require_gpu()
    U, op = _context(dims)
    ref = evenodd.SchurOperator(U, KAPPA, CSW, -1.0)
    vh = ref.A_ee.shape[0]
    x = rand_eo(n, vh, np.random.default_rng(23))
    for o, dag, f in ((0, False, ref.D_eo), (0, True, ref.D_oe_dag), (1, False, ref.D_oe), (2, False, ref.Mhat),
                      (2, True, ref.Mhat_dag), (3, False, ref.MdagM)):
        got = to_np(op.dslash(to_dev(x), o, dagger=dag, precision=64))
        for k in range(n):
            assert rel_l2(got[k], f(x[k])) < 1e-15, (o, dag, k)
    for prec in (64, 32):
        sol, stats, ok = op.cg_solve(to_dev(x), tol=1e-10, inner_prec=prec)
        assert ok
        for k, v in enumerate(to_np(sol)):
            rel = np.linalg.norm(ref.MdagM(v) - x[k]) / np.linalg.norm(x[k])
            assert rel < 1.001e-10 and abs(rel - stats[k]["true_rel_resid"]) < 1e-13
    op.close()


@gpu
def test_sums_in_two_steps():
    """488 blocks of 32 sites (the last one half full) are eight groups of 64, the last one of 40: sums of at least
    eight groups are formed group by group.  The residuals that the solves report against numpy's sums over the
    same operator's result (1e-13 of |b| in their rounding: 1e-5 of a residual of 1e-8), the plaquette against the
    oracle's; every call twice, as the groups' counters have to be left at zero."""
    require_gpu()
    from oracle import md as omd
    dims = (10, 10, 12, 26)
    U, op = _context(dims)
    b = rand_eo(4, int(np.prod(dims)) // 2, np.random.default_rng(29))
    iters = {}
    for n in (1, 4):
        for prec in (64, 32, 16):
            for turn in range(2):
                x, stats, ok = op.cg_solve(to_dev(b[:n]), tol=1e-8, inner_prec=prec)
                assert ok
                r = b[:n] - to_np(op.dslash(x, 3, precision=64))
                for k in range(n):
                    rel = np.linalg.norm(r[k]) / np.linalg.norm(b[k])
                    assert abs(rel - stats[k]["true_rel_resid"]) < 1e-13
                    iters[n, prec, turn, k] = stats[k]["iters"]
    for n in (1, 4):  # a wrong alpha or beta would not converge like exact ones
        for prec in (64, 32, 16):
            for k in range(n):
                assert iters[n, prec, 0, k] == iters[n, prec, 1, k]
                assert iters[n, 32, 0, k] <= iters[n, 64, 0, k] + 3
    want = omd.mean_plaquette(U)
    for turn in range(2):
        assert abs(op.plaquette() - want) < 4e-15
    op.close()


@gpu
def test_sites_of_very_different_size():
    """Each site keeps its own exponent: sites 2^-300 .. 2^300 apart, zero sites, subnormal ones."""
    require_gpu()
    dims = (6, 4, 4, 6)
    U, op = _context(dims, clover=False)
    ref = evenodd.SchurOperator(U, KAPPA, CSW, -1.0)
    rng = np.random.default_rng(7)
    vh = ref.A_ee.shape[0]
    x = rand_eo(1, vh, rng)
    x *= (2.0 ** rng.integers(-300, 300, vh))[None, :, None, None]
    x[0, ::7] = 0.0
    x[0, 3] = 5e-324
    x[0, 5] *= 1e-290 / np.abs(x[0, 5]).max()
    got = to_np(op.dslash(to_dev(x), 0, precision=64))[0]
    want = ref.D_eo(x[0])
    big = np.abs(x[0]).max(axis=(1, 2))  # per odd site
    full = join_eo(None, np.broadcast_to(big[:, None, None], (vh, 4, 3)).astype(complex), dims)
    near = sum(np.roll(full, s, ax) for ax in range(4) for s in (1, -1))
    near = split_eo(near, dims)[0].real[:, 0, 0]
    err = np.abs(got - want).max(axis=(1, 2))
    assert np.all(err <= 16 * 2.0 ** -53 * np.sqrt(6) * near + 5e-324)
    # a field of zeros gives zeros
    assert not np.any(to_np(op.dslash(to_dev(0 * x), 0, precision=64)))
    op.close()


@gpu
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_non_finite_sites_reach_their_neighbours_only(value):
    require_gpu()
    dims = (6, 4, 4, 6)
    U, op = _context(dims)
    x = rand_eo(1, U.size // 72, np.random.default_rng(9))
    clean = to_np(op.dslash(to_dev(x), 2, precision=64))[0]
    mark = np.zeros_like(x[0])
    mark[17] = 1.0
    around = lambda f: sum(np.roll(f, s, ax) for ax in range(4) for s in (1, -1))
    full = join_eo(mark, None, dims)
    reach = split_eo(full + around(around(full)), dims)[0].real[:, 0, 0] > 0  # two hops, and the site itself
    x[0, 17, 2, 1] = value
    got = to_np(op.dslash(to_dev(x), 2, precision=64))[0]
    finite = np.isfinite(got).all(axis=(1, 2))
    assert np.array_equal(finite[~reach], np.ones((~reach).sum(), bool)) and not finite[17]
    assert np.array_equal(got[~reach], clean[~reach])
    op.close()


@gpu
@pytest.mark.parametrize("nrhs", [1, 2, 3, 8])
def test_fp64_solve(nrhs):
    """Plain FP64 conjugate gradients with the search direction in fixed point, and a second kappa on the
    same context (whose recorded iterations must not be those of the first)."""
    require_gpu()
    dims = (6, 4, 4, 6)
    U, op = _context(dims)
    vh = U.size // 72
    b = rand_eo(nrhs, vh, np.random.default_rng(13))
    for kappa in (KAPPA, 0.11):
        op.clover_build(kappa, CSW)
        ref = evenodd.SchurOperator(U, kappa, CSW, -1.0)
        for prec in (64, 32, 16):
            x, st, ok = op.cg_solve(to_dev(b), tol=1e-11, inner_prec=prec)
            assert ok
            r = np.stack([ref.MdagM(v) for v in to_np(x)]) - b
            for k in range(nrhs):
                rel = np.linalg.norm(r[k]) / np.linalg.norm(b[k])
                assert rel < 1.01e-11 and abs(rel - st[k]["true_rel_resid"]) < 1e-13
    op.close()


@gpu
@pytest.mark.parametrize("prec", [64, 32, 16])
@pytest.mark.parametrize("nrhs", [1, 2, 5])
@pytest.mark.parametrize("dims", [(2, 2, 10, 2), (6, 10, 2, 18), (10, 8, 8, 10)], ids=["40", "1080", "3200"])
def test_solves_on_ragged_blocks(dims, nrhs, prec):
    """40 and 1080 sites per parity: a ragged last block of 32; 3200: 100 blocks.  The true residual, formed by the
    FP64 operator, differs between two evaluations by its rounding, below 1e-13."""
    require_gpu()
    U, op = _context(dims)
    b = rand_eo(nrhs, int(np.prod(dims)) // 2, np.random.default_rng(19))
    x, stats, ok = op.cg_solve(to_dev(b), tol=1e-10, inner_prec=prec)
    assert ok
    r = b - to_np(op.dslash(x, 3, precision=64))
    for i in range(nrhs):
        assert np.linalg.norm(r[i]) <= (1e-10 + 1e-13) * np.linalg.norm(b[i])
    op.close()


@gpu
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (4, 4, 2, 2), (4, 2, 6, 4), (6, 10, 2, 4)], ids=lambda d: "x".join(map(str, d)))
@pytest.mark.parametrize("scale,t_bc", [(1.0, -1.0), (1.0, 1.0), (1.25, -1.0)], ids=["su3", "su3_periodic", "far"])
def test_matrix_fields(dims, scale, t_bc):
    """Clover blocks and log det, fermion and determinant force, gauge force and plaquette on partial, whole
    and ragged blocks of sites, with 0, 1, 2 and 5 right-hand sides (sums over several exponents).  Sums of
    at most 12 triple products of matrices per link beside the fields' own 1e-15."""
    require_gpu()
    from oracle import cloverdet, force as oforce, md as omd
    U, op = _context(dims, t_bc, scale)
    ref = evenodd.SchurOperator(U, KAPPA, CSW, t_bc)
    vh = ref.A_ee.shape[0]
    rng = np.random.default_rng(19)
    for p, A in enumerate((ref.A_ee, ref.A_oo)):
        want = np.linalg.slogdet(A)[1].sum()
        assert abs(op.clover_logdet()[p] - want) < 1e-13 * vh
    if t_bc == -1.0:  # (the oracle's gradient helpers take the antiperiodic operator)
        Gdet = cloverdet.gradient(ref)
        for n in (1, 2, 5):
            x = rand_eo(n, vh, rng) * np.array([1.0, 2.0 ** -20, 3.0, 0.0, 2.0 ** 9])[:n, None, None, None]
            G = oforce.gradient(ref, x)
            for det in (False, True):
                want = G + Gdet if det else G
                got, _ = op.fermion_force(to_dev(x), input_is_solution=True, gradient=True, clover_det=det)
                assert rel_l2(to_np(got), want) < 2e-15
                got, _ = op.fermion_force(to_dev(x), input_is_solution=True, clover_det=det)
                assert rel_l2(to_np(got), oforce.lie_force(U, want)) < 4e-15
        got, _ = op.fermion_force(None, clover_det=True)
        assert rel_l2(to_np(got), oforce.lie_force(U, Gdet)) < 1e-14  # (small beside the blocks it comes from)
    want = omd.gauge_force(U, 5.6)
    F = op.gauge_force(5.6)
    assert rel_l2(to_np(F), want) < 4e-15
    op.gauge_force(5.6, out=F)
    assert rel_l2(to_np(F), 2 * want) < 4e-15
    assert rel_l2(to_np(op.gauge_force(5.6, gradient=True)), omd.gauge_gradient(U, 5.6)) < 2e-15
    assert abs(op.plaquette() - omd.mean_plaquette(U)) < 4e-15 * scale ** 4
    op.close()


@gpu
def test_force_of_fields_with_marked_and_empty_sites():
    """A non-finite solution gives non-finite links around it; one that meets zeros elsewhere stays marked."""
    require_gpu()
    dims = (4, 4, 4, 6)
    U, op = _context(dims)
    x = np.zeros((1, U.size // 72, 4, 3), complex)
    x[0, 40, 1, 1] = np.nan
    F, _ = op.fermion_force(to_dev(x), input_is_solution=True)
    bad = ~np.isfinite(to_np(F)).all(axis=(-1, -2, -3))
    full = join_eo(np.isnan(x[0]).astype(complex), None, dims)
    assert bad[np.abs(full).max(axis=(-1, -2)) > 0].all()  # the site itself
    x[:] = 0
    F, _ = op.fermion_force(to_dev(x), input_is_solution=True)
    assert not np.any(to_np(F))
    op.close()
