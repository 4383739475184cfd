"""Waits of the H-LU column items, piece by piece, on the host (tests/lu_pieces_check.cpp)."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import synth
from paper_2405_03456_gb300 import build as hbuild

HOST = ["trees.cpp", "linalg.cpp", "build.cpp", "codec.cpp", "program.cpp", "lu_factor.cpp"]


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("needs g++")
    hbuild.build()
    tmp = tmp_path_factory.mktemp("lu_pieces")
    exe = str(tmp / "lu_pieces_check")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "lu_pieces_check.cpp")
    objs = [os.path.join(hbuild.OUT, f + ".o") for f in HOST]
    subprocess.run(["g++", "-std=c++17", "-O2", "-fopenmp", "-I", hbuild.CSRC, "-I",
                    os.path.join(hbuild.HERE, "..", "include"), src] + objs + ["-o", exe], check=True)
    return exe, tmp


@pytest.mark.parametrize("n,leaf,codec", [(1, 32, 1), (300, 128, 2), (700, 24, 1), (1000, 33, 0), (1500, 100, 1)])
def test_every_piece_waits_for_its_rows(checker, n, leaf, codec):
    exe, tmp = checker
    path = tmp / f"cube_{n}.bin"
    path.write_bytes(np.ascontiguousarray(synth.cube_points(n)).tobytes())
    r = subprocess.run([exe, str(path), str(n), "1e-6", str(codec), str(leaf)], stdout=subprocess.PIPE,
                       stderr=subprocess.STDOUT, text=True, timeout=600)
    assert r.returncode == 0 and r.stdout.rstrip().endswith("ok"), r.stdout[-2000:]
