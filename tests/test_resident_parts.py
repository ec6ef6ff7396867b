"""The resident kernel's parts (host side, mesh_build.cpp): a partition of the
cells whose records fill every face slot once, for every cell order and for
part counts from one to one cell per part. Compiles
tests/resident_parts_check.cpp against the library's mesh builder."""
import os
import shutil
import subprocess

import pytest

from paper_1807_00672_gb300 import inputs

from test_record_order import write_mesh

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("g++ not available")
    out = tmp_path_factory.mktemp("parts") / "resident_parts_check"
    subprocess.run([cxx, "-O2", "-std=c++17", "-pthread", "-o", str(out),
                    os.path.join(HERE, "resident_parts_check.cpp"),
                    os.path.join(ROOT, "paper_1807_00672_gb300", "csrc", "mesh_build.cpp"),
                    "-I", os.path.join(ROOT, "include")], check=True)
    return str(out)


@pytest.mark.parametrize("order", [0, 1, 2])
@pytest.mark.parametrize("parts", [1, 2, 7, 152, "cells"])
def test_parts_cover_the_mesh(checker, tmp_path, order, parts):
    for i, mesh in enumerate([inputs.random_flow_case(nx=37, ny=23, seed=41).mesh,
                              inputs.stoker_case().mesh,
                              inputs.jittered_grid(9, 31, 90.0, 310.0, jitter=0.3,
                                                   diagonal="shorter", seed=3)]):
        path = tmp_path / f"m{i}.bin"
        write_mesh(path, mesh)
        n = mesh.n_tris if parts == "cells" else parts
        r = subprocess.run([checker, str(path), str(order), str(n)], capture_output=True, text=True)
        assert r.returncode == 0, r.stdout + r.stderr
        assert r.stdout.startswith(f"ok {n} "), r.stdout
