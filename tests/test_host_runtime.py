"""The library's host code on a CUDA runtime without a GPU (fake_cudart.cpp):
no host memory is freed while a queued copy has still to read it, through mesh
creation, products, solves, sweeps, fields and gradients; and a handle of one
device is usable while another device is current.  Linked from the objects of
the build (built again where they are missing)."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2312_00005_gb300 import build, inputs

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    objs = [os.path.join(build.BUILD_DIR, os.path.splitext(f)[0] + ".o") for f in build.SOURCES]
    build.build(force=not all(os.path.exists(o) for o in objs))
    d = tmp_path_factory.mktemp("host")
    exe = str(d / "host")
    r = subprocess.run([cxx, "-O1", "-std=c++17", "-I/usr/local/cuda/include", os.path.join(ROOT, "tests", "fake_cudart.cpp")] +
                       objs + ["-lpthread", "-ldl", "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    files = {}
    for nu in (4, 16):                            # 16: the leaf-size tuner runs (4096 elements and more)
        nodes, tris = inputs.geodesic_sphere(nu)
        files[nu] = (str(d / ("nodes%d" % nu)), str(d / ("tris%d" % nu)))
        np.ascontiguousarray(0.1 * nodes, np.float64).tofile(files[nu][0])
        np.ascontiguousarray(tris, np.int32).tofile(files[nu][1])
    return exe, files


@pytest.mark.parametrize("nu", [4, 16])
def test_host_memory_outlives_its_copies(program, nu):
    exe, files = program
    r = subprocess.run([exe, "uploads", *files[nu]], capture_output=True, text=True, timeout=300)
    print(r.stdout)
    assert r.returncode == 0 and "errors 0, freed in flight 0" in r.stdout, (r.returncode, r.stdout, r.stderr[-1000:])

def test_handle_of_another_device_than_the_current(program):
    exe, files = program
    r = subprocess.run([exe, "devices", *files[4]], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "errors 0" in r.stdout, (r.returncode, r.stdout, r.stderr[-1000:])
