"""What the library does when device memory runs out, on the host: its host objects
on a fake CUDA runtime with a byte budget (tests/device_memory_check.cpp)."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import synth
from paper_2405_03456_gb300 import build as hbuild

HOST = ["trees.cpp", "linalg.cpp", "build.cpp", "codec.cpp", "program.cpp", "matrix.cpp"]


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("needs g++")
    hbuild.build()
    tmp = tmp_path_factory.mktemp("device_memory")
    exe = str(tmp / "device_memory_check")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "device_memory_check.cpp")
    objs = [os.path.join(hbuild.OUT, f + ".o") for f in HOST]
    subprocess.run(["g++", "-std=c++17", "-O1", "-fopenmp", "-I", hbuild.CSRC, "-I",
                    os.path.join(hbuild.HERE, "..", "include"), "-I", os.path.join(hbuild.CUDA, "include"), src] + objs +
                   ["-o", exe], check=True)
    return exe, tmp


@pytest.mark.parametrize("n,eps,codec,leaf,fmt", [(1500, "1e-8", 1, 32, 0), (400, "1e-4", 0, 64, 0),
                                                  (1500, "1e-6", 1, 32, 0), (300, "1e-6", 2, 128, 0),
                                                  (1200, "1e-6", 1, 64, 2), (700, "1e-6", 1, 32, 3)])
def test_optional_buffers_never_cost_a_matrix(checker, n, eps, codec, leaf, fmt):
    exe, tmp = checker
    path = tmp / f"sphere_{n}.bin"
    path.write_bytes(np.ascontiguousarray(synth.sphere_points(n)).tobytes())
    r = subprocess.run([exe, str(path), str(n), eps, str(codec), str(leaf), str(fmt)], stdout=subprocess.PIPE,
                       stderr=subprocess.STDOUT, text=True, timeout=600)
    assert r.returncode == 0 and r.stdout.rstrip().endswith("ok"), r.stdout[-2000:]
