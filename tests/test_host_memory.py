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



def test_a_handle_under_construction_goes_with_the_exception(checker):
    r = subprocess.run([checker, "guard"], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "ok 1", (r.returncode, r.stdout, r.stderr)


def test_a_batch_without_memory_is_an_error(tmp_path):
    """swe_mesh_create_batch, whose scenarios are built on several threads
    (tests/batch_memory_check.cpp), in a process without a GPU."""
    from paper_1807_00672_gb300 import build
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("g++ not available")
    lib = build.build()
    out = str(tmp_path / "batch_memory_check")
    subprocess.run([cxx, "-O2", "-std=c++17", "-pthread", "-o", out,
                    os.path.join(HERE, "batch_memory_check.cpp"), lib,
                    f"-Wl,-rpath,{os.path.dirname(lib)}", "-I", os.path.join(ROOT, "include")], check=True)
    r = subprocess.run([out], capture_output=True, text=True, env=dict(os.environ, CUDA_VISIBLE_DEVICES=""))
    assert r.returncode == 0 and r.stdout.startswith("ok "), (r.returncode, r.stdout, r.stderr)
    assert int(r.stdout.split()[1]) > 10
