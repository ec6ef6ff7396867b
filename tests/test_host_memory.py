"""Host memory that runs out while a mesh is built, on whichever host thread:
the process goes on, the optional stages leave their work out."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("g++ not available")
    out = tmp_path_factory.mktemp("memory") / "host_memory_check"
    subprocess.run([cxx, "-O2", "-std=c++17", "-pthread", "-o", str(out),
                    os.path.join(HERE, "host_memory_check.cpp"),
                    os.path.join(ROOT, "paper_1807_00672_gb300", "csrc", "mesh_build.cpp"),
                    "-I", os.path.join(ROOT, "include")], check=True)
    return str(out)


def test_parts_are_left_out(checker):
    r = subprocess.run([checker, "parts"], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.startswith("ok "), (r.returncode, r.stdout, r.stderr)
    assert int(r.stdout.split()[1]) > 30


def test_records_keep_their_order(checker):
    r = subprocess.run([checker, "banks"], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.startswith("ok "), (r.returncode, r.stdout, r.stderr)
    assert int(r.stdout.split()[1]) > 3
