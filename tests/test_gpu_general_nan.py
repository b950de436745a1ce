"""A Gauss-Seidel update does not use a node's old value: an infinity or NaN in
the initial guess at an interior macro vertex, whose neighbours all come later
in the sweep, is gone after it, also through the padded interface tables."""

import itertools

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hhg():
    from paper_1506_06185_gb300.build import build
    from paper_1506_06185_gb300 import hhg as H
    build()
    return H


def _cube_of_tets():
    """2x2x2 sub-cubes of six tetrahedra, corners moved a little; vertex 13 is
    inside, the others on the boundary."""
    z, y, x = np.meshgrid(*(np.arange(3),) * 3, indexing="ij")
    pos = np.stack([x, y, z], -1).reshape(-1, 3) / 2 + np.random.default_rng(1).uniform(-0.05, 0.05, (27, 3))
    tets = []
    for c in itertools.product(range(2), repeat=3):
        for p in itertools.permutations(range(3)):
            v, t = list(c), []
            for ax in (None, *p):
                if ax is not None:
                    v[ax] += 1
                t.append((v[2] * 3 + v[1]) * 3 + v[0])
            tets.append(t)
    return pos, np.array(tets, dtype=np.int32)


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_old_value_of_a_vertex_is_not_used(hhg, value):
    pos, tets = _cube_of_tets()
    out = []
    for v in (0.0, value):
        G = hhg.Mesh.general(pos, tets, 4)
        f = np.random.default_rng(2).uniform(-1, 1, G.n_nodes)
        u = np.zeros(G.n_nodes)
        u[13] = v                                        # vertices come first, in their own order
        G.set_problem(f, u)
        G.vcycle()
        out.append(G.get_solution())
        G.close()
    assert np.isfinite(out[0]).all() and np.array_equal(*out)
