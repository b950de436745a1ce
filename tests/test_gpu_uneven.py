"""Cubes whose sub-cube counts do not divide evenly (spacings 1/3, 1/5, 1/7):
the eight vanishing stencil weights are found to be zero, so these meshes run
the 7-point kernels, and the cycles match the oracle."""

import numpy as np
import pytest

import hhg_inputs as I
import oracle as O
from parity import assert_close

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hhg():
    from paper_1506_06185_gb300.build import build
    from paper_1506_06185_gb300 import hhg as H
    build()
    return H


@pytest.mark.parametrize("sub,R", [((3, 3, 3), 4), ((1, 3, 5), 4), ((7, 1, 1), 3)])
def test_uneven_cube_is_seven_point(hhg, sub, R):
    f = I.random_load(sub, R, seed=3)
    u0 = I.initial_guess(sub, R, I.harmonic_boundary(sub, R))
    M = hhg.Mesh(sub, R)
    assert hhg.hhg_profile_info(M.h)[1]
    M.set_problem(f, u0)
    m = O.Mesh(sub, R)
    uo, fo = O.pad(u0.copy()), O.pad(f)
    for _ in range(3):
        M.vcycle()
        O.vcycle(m, m.global_problem, len(m.levels) - 1, uo, fo)
    assert_close(M.get_solution(), O.interior(uo))
    M.close()


def test_sheared_mesh_keeps_fifteen_points(hhg):
    M = hhg.Mesh((3, 1, 1), 3, affine=np.array([[1, 1e-6, 0], [0, 1, 0], [0, 0, 1.0]]))
    assert not hhg.hhg_profile_info(M.h)[1]
    M.close()
