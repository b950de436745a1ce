"""Interface stencil tables of general meshes, row by row against the
sub-stencils of the nodes' copies (host program, no GPU)."""

import os
import shutil
import subprocess

import numpy as np
import pytest

import hhg_inputs as I

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def prog(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    cuda_inc = "/usr/local/cuda/include"
    if not cxx or not os.path.isdir(cuda_inc):
        pytest.skip("needs a C++ compiler and the CUDA headers")
    out = tmp_path_factory.mktemp("generaltables") / "general_tables"
    subprocess.check_call([cxx, "-O1", "-std=c++17", "-I" + cuda_inc, "-o", str(out),
                           os.path.join(ROOT, "tests", "host", "general_tables.cpp"),
                           os.path.join(ROOT, "paper_1506_06185_gb300", "csrc", "mesh.cpp")])
    return str(out)


@pytest.mark.parametrize("mesh", ["five-moved", "kuhn"])
@pytest.mark.parametrize("kind,faulty", [(0, []), (1, [0, 1, 2, 3, 4, 5]), (2, [3]), (3, [3]), (3, [0, 1, 7])])
def test_rows(prog, tmp_path, mesh, kind, faulty):
    v, t = I.kuhn_macro_mesh((2, 1, 2)) if mesh == "kuhn" else I.five_tet_macro_mesh((2, 2, 1), seed=3, amp=0.12)
    np.ascontiguousarray(v, dtype=np.float64).tofile(tmp_path / "verts.bin")
    np.ascontiguousarray(t, dtype=np.int32).tofile(tmp_path / "tets.bin")
    r = subprocess.run([prog, str(len(v)), str(len(t)), "4", str(tmp_path), str(kind), *map(str, faulty)],
                       capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.startswith("ok"), r.stdout + r.stderr
