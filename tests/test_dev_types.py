"""Host check of the arithmetic that host and device code share (csrc/dev_types.h)."""
import os
import shutil
import subprocess

import pytest

from paper_2405_03456_gb300 import build as hbuild


def test_dev_types(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("needs g++")
    exe = str(tmp_path / "dev_types_check")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "dev_types_check.cpp")
    subprocess.run(["g++", "-std=c++17", "-O1", "-fsanitize=undefined", "-I", hbuild.CSRC, src, "-o", exe], check=True)
    r = subprocess.run([exe], stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.rstrip() == "ok", r.stdout
