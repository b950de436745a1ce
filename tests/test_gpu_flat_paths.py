"""The flat kernels and both walks of the tile kernels (grid stride and dynamic)
give the same iterates bit for bit, with the path each mesh takes asserted, so
that a changed default cannot leave a kernel compared with itself: a new mesh
runs flat, a launch limit selects the tile kernels, with the grid-stride walk
under a large one."""

import numpy as np
import pytest

import hhg_inputs as I

pytestmark = pytest.mark.gpu

SHEAR = np.array([[1.0, 0.3, -0.2], [0.1, 0.9, 0.25], [-0.15, 0.2, 1.1]])
STRIDE = 1 << 20      # more CTAs than the GPU holds


@pytest.fixture(scope="module")
def hhg():
    from paper_1506_06185_gb300.build import build
    from paper_1506_06185_gb300 import hhg as H
    build()
    return H


def _run(hhg, sub, R, limit, mesh_kw, call):
    """(solution, call's result) with the path checked; limit 0: flat."""
    M = hhg.Mesh(sub, R, **mesh_kw)
    hhg.hhg_set_launch_limit(M.h, limit)
    flat = hhg.hhg_flat_levels(M.h, R - 1)
    assert all(flat) if limit == 0 else not any(flat)
    M.set_problem(I.random_load(sub, R, seed=21), I.initial_guess(sub, R, I.harmonic_boundary(sub, R)))
    out = call(M)
    u, walks = M.get_solution(), hhg.hhg_walk_counts(M.h)
    assert (walks[0] > 0) == (0 < limit < STRIDE), walks
    M.close()
    return u, out


def _cycles(M):
    return [M.vcycle() for _ in range(3)]


def _solve(**kw):
    return lambda M: list(M.solve(rtol=1e-9, max_cycles=40, fault_cycle=3, n_global=2, eta=2.0, **kw)[0])


CASES = [((2, 2, 1), 5, {}, _cycles), ((2, 1, 2), 5, dict(affine=SHEAR), _cycles),
         ((2, 2, 2), 5, {}, _solve(fault_ids=list(range(6)), recovery=2)),
         ((2, 2, 2), 5, dict(precision=32), _solve(fault_ids=list(range(6)), recovery=2, mixed_precision=True)),
         ((3, 2, 2), 4, dict(affine=SHEAR), _solve(fault_ids=[13, 14, 30, 31], recovery=3))]


@pytest.mark.parametrize("sub,R,mesh_kw,call", CASES)
def test_flat_and_tile_kernels_alike(hhg, sub, R, mesh_kw, call):
    uf, hf = _run(hhg, sub, R, 0, mesh_kw, call)
    for limit in (STRIDE, 3):
        ut, ht = _run(hhg, sub, R, limit, mesh_kw, call)
        assert np.array_equal(uf, ut), limit
        # the norms' partial sums follow each launch's grid: equal up to rounding
        assert len(hf) == len(ht) and np.abs(np.array(hf) - ht).max() <= 1e-12 * hf[0], limit


@pytest.mark.parametrize("sub,R,mesh_kw", [((2, 2, 1), 5, {}), ((2, 1, 2), 5, dict(affine=SHEAR))])
def test_launch_limit_on_a_tuned_mesh(hhg, sub, R, mesh_kw):
    M = hhg.Mesh(sub, R, **mesh_kw)
    f, u0 = I.random_load(sub, R, seed=22), I.initial_guess(sub, R)
    M.set_problem(f, u0)
    M.vcycle()
    u = M.get_solution()
    hhg.hhg_autotune(M.h, R - 1)
    tuned = hhg.hhg_flat_levels(M.h, R - 1)
    hhg.hhg_set_launch_limit(M.h, 2)
    assert not any(hhg.hhg_flat_levels(M.h, R - 1))
    before = hhg.hhg_walk_counts(M.h)[0]
    M.set_problem(f, u0)
    M.vcycle()
    assert np.array_equal(M.get_solution(), u) and hhg.hhg_walk_counts(M.h)[0] >= before + 24
    hhg.hhg_set_launch_limit(M.h, 0)
    assert hhg.hhg_flat_levels(M.h, R - 1) == tuned
    M.close()


def test_switch_off_and_on(hhg):
    M = hhg.Mesh((2, 1, 1), 4)
    hhg.hhg_set_flat_gs(M.h, False)
    assert not any(hhg.hhg_flat_levels(M.h, 3))
    hhg.hhg_set_flat_gs(M.h, True)                       # asked for: a limit does not change it
    hhg.hhg_set_launch_limit(M.h, 5)
    assert all(hhg.hhg_flat_levels(M.h, 3))
    M.close()
