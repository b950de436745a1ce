"""Meshes and the batch that holds their buffers may be destroyed in either
order; a batch whose mesh is gone refuses to launch."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hhg():
    from paper_1506_06185_gb300.build import build
    from paper_1506_06185_gb300 import hhg as H
    build()
    return H


def test_meshes_first(hhg):
    for _ in range(4):
        meshes = [hhg.Mesh((1, 1, 1), 3) for _ in range(6)]
        for M in meshes:
            M.set_problem(np.zeros(M.shape), np.zeros(M.shape))
        batch = hhg.Batch([(M, [0], 1) for M in meshes])
        batch.launch_persistent()
        meshes[0].close()
        for call in (batch.launch, batch.launch_persistent, batch.set_priority):
            with pytest.raises(hhg.HHGError) as e:
                call()
            assert e.value.code == hhg.HHG_ERR_STATE
        for M in meshes:
            M.close()
        batch.close()
