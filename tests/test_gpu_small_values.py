"""Loads in small (or huge) units and homogeneous problems run down to nothing:
the coarse CG squares its vectors, so from norms of about 1e-143 on its sums
would be subnormal numbers, whose reciprocals overflow.  Every launch form
solves them as it solves the same load in ordinary units."""

import numpy as np
import pytest

import hhg_inputs as I
import oracle as O
from parity import assert_close

pytestmark = pytest.mark.gpu

SHEAR = np.array([[1.0, 0.3, -0.2], [0.1, 0.9, 0.25], [-0.15, 0.2, 1.1]])


@pytest.fixture(scope="module")
def hhg():
    from paper_1506_06185_gb300.build import build
    from paper_1506_06185_gb300 import hhg as H
    build()
    return H


def _coeff(sub):
    return 10.0 ** np.random.default_rng(5).uniform(-1.0, 1.0, 6 * int(np.prod(sub)))


# (sub-cubes, refinement, coarsest, affine map, coefficients): 27 and 147
# coarse unknowns (one CTA), 343 (8 CTAs), 3375 (16), 12167 (several blocks per
# warp), 29791 (vectors in the work array); 15 points; preconditioned
FORMS = [((1, 1, 1), 3, 2, None, False), ((1, 2, 2), 3, 2, SHEAR, False), ((2, 2, 2), 3, 2, None, False),
         ((2, 2, 2), 3, 2, None, True), ((2, 2, 2), 4, 3, None, False), ((2, 2, 2), 4, 3, SHEAR, True),
         ((3, 3, 3), 4, 3, None, False), ((2, 2, 2), 5, 4, None, False)]


# The same load times a power of two, which no rounding changes (2^-900 leaves
# room for the smallest entries): the same bits, in every form.
@pytest.mark.parametrize("exponent", [-480, -500, -560, -900, 530])
@pytest.mark.parametrize("sub,R,r0,affine,var", FORMS)
def test_load_in_small_units(hhg, sub, R, r0, affine, var, exponent):
    f, u0 = I.random_load(sub, R, seed=4), np.zeros(tuple((s << R) + 1 for s in reversed(sub)))
    kw = dict(coarsest=r0, affine=affine, coeff=_coeff(sub) if var else None)
    A, B, T = hhg.Mesh(sub, R, **kw), hhg.Mesh(sub, R, **kw), hhg.Mesh((1, 1, 1), 3)
    T.set_problem(np.zeros(T.shape), np.zeros(T.shape))
    A.set_problem(f, u0)
    A.vcycle()
    ref = A.get_solution()
    small = np.ldexp(f, exponent)

    def check(M, what):
        assert np.array_equal(np.ldexp(M.get_solution(), -exponent), ref), what

    A.set_problem(small, u0)
    A.vcycle()
    check(A, "cycle")
    batch = hhg.Batch([(T, [0], 1)], B, 1)
    B.set_problem(small, u0)
    batch.launch_persistent()
    check(B, "persistent executor")
    if r0 < 4:
        B.set_problem(small, u0)
        hhg.hhg_vcycle_noalloc(B.h)
        check(B, "allocation-free")
    if r0 == 2 and affine is None:
        m = O.Mesh(sub, R, coeff=kw["coeff"])
        uo, fo = O.pad(u0.copy()), O.pad(f)
        O.vcycle(m, m.global_problem, len(m.levels) - 1, uo, fo)
        assert_close(np.ldexp(A.get_solution(), -exponent), O.interior(uo))
    batch.close()
    for M in (A, B, T):
        M.close()


@pytest.mark.parametrize("sub,R,var", [((1, 1, 1), 3, False), ((2, 2, 2), 3, False), ((2, 2, 2), 3, True)])
def test_homogeneous_problem_dies_out(hhg, sub, R, var):
    """f = 0: every cycle reduces the iterate, down to the smallest numbers."""
    M = hhg.Mesh(sub, R, coeff=_coeff(sub) if var else None)
    f = np.zeros(M.shape)
    u = np.zeros(M.shape)
    u[1:-1, 1:-1, 1:-1] = np.random.default_rng(9).uniform(-1, 1, tuple(n - 2 for n in M.shape))
    M.set_problem(f, u)
    last = 1.0
    for _ in range(20):
        for _ in range(20):
            M.vcycle()
        now = np.abs(M.get_solution()).max()
        assert np.isfinite(now) and (now < 1e-3 * last or now < 1e-300), (now, last)
        last = now
    assert last < 1e-150
    M.close()
