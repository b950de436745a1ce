"""Set-up followed at once by work on another, non-blocking stream: new
coefficients, fault sets, Dirichlet-Neumann set-up, flat and tile tables and
batches give the same bits as on the default stream."""

import numpy as np
import pytest

import hhg_inputs as I

pytestmark = pytest.mark.gpu

SHEAR = np.array([[1.0, 0.3, -0.2], [0.1, 0.9, 0.25], [-0.15, 0.2, 1.1]])


def _program(hhg, sub, R, kw):
    import torch
    n = 6 * int(np.prod(sub))
    M = hhg.Mesh(sub, R, **kw)
    f, u0 = I.random_load(sub, R, seed=31), I.initial_guess(sub, R)
    M.set_problem(torch.from_numpy(f).cuda(), torch.from_numpy(u0).cuda())
    out = []
    for k in range(4):
        M.set_coefficients(np.exp(0.3 * np.random.default_rng(k).standard_normal(n)))
        M.vcycle()
        out.append(M.get_solution())
        M.inject_fault([k, k + 5])
        M.recover_local([k, k + 5], 2, 1)
        out.append(M.get_solution())
        M.inject_fault([k + 2])
        M.recover_dn([k + 2], 2, 2.0)
        out.append(M.get_solution())
        hhg.hhg_set_launch_limit(M.h, 2 if k % 2 else 0)
        if "affine" not in kw:
            hhg.hhg_set_flat_gs(M.h, k % 2 == 0)
        M.vcycle()
        out.append(M.get_solution())
    hhg.hhg_autotune(M.h, R - 1, reps=1)
    M.set_problem(f, u0)
    M.vcycle()
    out.append(M.get_solution())
    T = hhg.Mesh(sub, R, **kw)
    T.set_problem(f, u0)
    batch = hhg.Batch([(T, [1], 2)])
    batch.launch_persistent()
    out.append(T.get_solution())
    batch.close()
    M.close()
    T.close()
    return out


@pytest.mark.parametrize("sub,R,kw", [((2, 2, 1), 4, {}), ((2, 1, 2), 3, dict(affine=SHEAR))])
def test_set_up_is_done_before_another_stream_uses_it(sub, R, kw):
    import torch
    from paper_1506_06185_gb300.build import build
    from paper_1506_06185_gb300 import hhg
    build()
    ref = _program(hhg, sub, R, kw)
    with torch.cuda.stream(torch.cuda.Stream()):
        got = _program(hhg, sub, R, kw)
    for k, (a, b) in enumerate(zip(ref, got)):
        assert np.isfinite(a).all() and np.array_equal(a, b), k
