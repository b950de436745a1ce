"""The coarse CG's launch forms (one CTA, clusters of 8 and 16 CTAs, vectors in
registers or in the work array, the persistent executor's one CTA) follow one
summation order: the same iterate bit for bit, at the edges of their ranges."""

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


# coarse unknowns: 27, 147 (one CTA), 343 (8 CTAs), 1331, 3375 (16), 12167
# (several blocks per warp), 29791 (vectors in the work array, 128-row blocks)
@pytest.mark.parametrize("sub,R,r0,affine", [((1, 1, 1), 3, 2, None), ((1, 2, 2), 3, 2, SHEAR), ((2, 2, 2), 3, 2, None),
                                             ((3, 3, 3), 3, 2, SHEAR), ((2, 2, 2), 4, 3, None), ((2, 2, 2), 4, 3, SHEAR),
                                             ((3, 3, 3), 4, 3, SHEAR), ((2, 2, 2), 5, 4, None)])
def test_cluster_equals_persistent_executor(hhg, sub, R, r0, affine):
    f = I.random_load(sub, R, seed=11)
    u0 = I.initial_guess(sub, R, I.harmonic_boundary(sub, R))
    A, B, T = hhg.Mesh(sub, R, coarsest=r0, affine=affine), hhg.Mesh(sub, R, coarsest=r0, affine=affine), hhg.Mesh((1, 1, 1), 3)
    T.set_problem(np.zeros(T.shape), np.zeros(T.shape))
    A.set_problem(f, u0)
    r = A.vcycle()
    batch = hhg.Batch([(T, [0], 1)], B, 1)
    B.set_problem(f, u0)
    batch.launch_persistent()
    assert np.array_equal(A.get_solution(), B.get_solution())
    B.set_problem(f, u0)
    hhg.hhg_vcycle_noalloc(B.h) if r0 < 4 else B.vcycle()
    assert np.array_equal(A.get_solution(), B.get_solution())
    # the coarse solve is converged: a further cycle reduces the residual at
    # the method's rate (0.12 on the cube, 0.35 sheared)
    assert A.vcycle() < 0.4 * r
    batch.close()
    for M in (A, B, T):
        M.close()


@pytest.mark.parametrize("sub,R,r0", [((1, 1, 1), 3, 2), ((2, 2, 2), 3, 2), ((3, 3, 3), 3, 2), ((3, 3, 3), 4, 3)])
def test_preconditioned_forms(hhg, sub, R, r0):
    """Coefficients over three decades: Jacobi-preconditioned, all forms alike,
    and the solution is that of the oracle's plain CG."""
    k = 10.0 ** np.random.default_rng(5).uniform(-1.5, 1.5, 6 * int(np.prod(sub)))
    f, u0 = I.random_load(sub, R, seed=12), I.initial_guess(sub, R)
    A, B, T = hhg.Mesh(sub, R, coarsest=r0, coeff=k), hhg.Mesh(sub, R, coarsest=r0), hhg.Mesh((1, 1, 1), 3)
    B.set_coefficients(k)
    T.set_problem(np.zeros(T.shape), np.zeros(T.shape))
    A.set_problem(f, u0)
    A.vcycle()
    batch = hhg.Batch([(T, [0], 1)], B, 1)
    B.set_problem(f, u0)
    batch.launch_persistent()
    assert np.array_equal(A.get_solution(), B.get_solution())
    if r0 == 2:
        m = O.Mesh(sub, R, coeff=k)
        uo, fo = O.pad(u0.copy()), O.pad(f)
        O.vcycle(m, m.global_problem, len(m.levels) - 1, uo, fo)
        assert_close(A.get_solution(), O.interior(uo))
    batch.close()
    for M in (A, B, T):
        M.close()


@pytest.mark.parametrize("maxit,rtol", [(1, 0.0), (3, 0.0), (1000, 1e-2), (1000, 2.0)])
def test_caps_and_loose_tolerances(hhg, maxit, rtol):
    """The caller's cap and tolerance end the iteration where the oracle's CG ends."""
    sub, R = (2, 2, 1), 3
    f, u0 = I.random_load(sub, R, seed=2), I.initial_guess(sub, R)
    M = hhg.Mesh(sub, R)
    M.set_problem(f, u0)
    M.solve(rtol=1e-30, max_cycles=2, coarse_maxit=maxit, coarse_rtol=rtol, allow_not_converged=True)
    m = O.Mesh(sub, R)
    uo, fo = O.pad(u0.copy()), O.pad(f)
    for _ in range(2):
        O.vcycle(m, m.global_problem, len(m.levels) - 1, uo, fo, cg_rtol=rtol or 1e-12, cg_maxit=maxit)
    assert_close(M.get_solution(), O.interior(uo))
    M.close()
