"""Parts of the row chunks that several ranges of a panel launch share, walked on the
host as the tensor-core kernel walks them (tests/panel_parts_check.cpp)."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import synth
from paper_2405_03456_gb300 import build as hbuild

HOST = ["trees.cpp", "linalg.cpp", "build.cpp", "codec.cpp", "program.cpp"]


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("needs g++")
    hbuild.build()
    tmp = tmp_path_factory.mktemp("panel_parts")
    exe = str(tmp / "panel_parts_check")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "panel_parts_check.cpp")
    objs = [os.path.join(hbuild.OUT, f + ".o") for f in HOST]
    subprocess.run(["g++", "-std=c++17", "-O1", "-fopenmp", "-I", hbuild.CSRC, "-I",
                    os.path.join(hbuild.HERE, "..", "include"), src] + objs + ["-o", exe], check=True)
    return exe, tmp


@pytest.mark.parametrize("n,fmt,eps,codec,leaf,adm", [
    (1, 0, "1e-6", 1, 32, 0), (300, 0, "1e-6", 0, 128, 0), (2000, 0, "1e-6", 1, 128, 0), (2000, 1, "1e-6", 1, 64, 0),
    (2500, 2, "1e-4", 2, 64, 0), (1500, 3, "1e-6", 1, 33, 0), (4000, 0, "1e-6", 1, 7, 1), (1100, 0, "1e-4", 0, 128, 2),
])
def test_parts_by_cta(checker, n, fmt, eps, codec, leaf, adm):
    exe, tmp = checker
    path = tmp / f"sphere_{n}.bin"
    path.write_bytes(np.ascontiguousarray(synth.sphere_points(n)).tobytes())
    r = subprocess.run([exe, str(path), str(n), str(fmt), eps, str(codec), str(leaf), str(adm)], stdout=subprocess.PIPE,
                       stderr=subprocess.STDOUT, text=True, timeout=600)
    assert r.returncode == 0 and r.stdout.rstrip().endswith("ok"), r.stdout[-2000:]
