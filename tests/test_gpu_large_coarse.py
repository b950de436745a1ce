"""A coarse problem beyond the cluster form of the CG (377055 unknowns): the
one-CTA kernel and the persistent executor give the same bits, also for the
load in small units, and the coarse solve is converged."""

import numpy as np
import pytest

import hhg_inputs as I

pytestmark = pytest.mark.gpu


def test_one_cta_cg():
    from paper_1506_06185_gb300.build import build
    from paper_1506_06185_gb300 import hhg
    build()
    sub, R, r0 = (3, 2, 2), 6, 5
    f, u0 = I.random_load(sub, R, seed=7), np.zeros(tuple((s << R) + 1 for s in reversed(sub)))
    A, T = hhg.Mesh(sub, R, coarsest=r0), hhg.Mesh((1, 1, 1), 3)
    T.set_problem(np.zeros(T.shape), np.zeros(T.shape))
    A.set_problem(f, u0)
    r = A.vcycle()
    u = A.get_solution()
    assert A.vcycle() < 0.2 * r                          # the method's rate on the cube: 0.12
    A.set_problem(np.ldexp(f, -500), u0)
    A.vcycle()
    assert np.array_equal(np.ldexp(A.get_solution(), 500), u)
    batch = hhg.Batch([(T, [0], 1)], A, 1)
    A.set_problem(f, u0)
    batch.launch_persistent()
    assert np.array_equal(A.get_solution(), u)
    batch.close()
    for M in (A, T):
        M.close()
