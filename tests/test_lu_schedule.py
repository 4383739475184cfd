"""The device schedule of the H-LU triangular solves: replayed on the host
(tests/lu_schedule_check.cpp), and on the GPU at the sizes where its shapes
change -- one row, one leaf, leaves of 1 .. 128 rows, more right-hand sides than
one launch takes."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import synth
from oracle import kernels
from paper_2405_03456_gb300 import build as hbuild

HOST = ["trees.cpp", "linalg.cpp", "build.cpp", "codec.cpp", "program.cpp", "lu_factor.cpp"]


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("needs g++")
    hbuild.build()
    tmp = tmp_path_factory.mktemp("lu_schedule")
    exe = str(tmp / "lu_schedule_check")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "lu_schedule_check.cpp")
    objs = [os.path.join(hbuild.OUT, f + ".o") for f in HOST]
    subprocess.run(["g++", "-std=c++17", "-O2", "-fopenmp", "-ffp-contract=off", "-I", hbuild.CSRC, "-I",
                    os.path.join(hbuild.HERE, "..", "include"), src] + objs + ["-o", exe], check=True)
    return exe, tmp


@pytest.mark.parametrize("n,leaf,codec", [(1, 32, 1), (40, 1, 0), (300, 128, 2), (700, 24, 1), (1000, 32, 2)])
def test_lu_schedule_replay(checker, n, leaf, codec):
    exe, tmp = checker
    path = tmp / f"cube_{n}.bin"
    path.write_bytes(np.ascontiguousarray(synth.cube_points(n)).tobytes() +
                     np.ascontiguousarray(synth.rhs(n)[:, 0]).tobytes())
    r = subprocess.run([exe, str(path), str(n), "1", "1e-6", str(codec), str(leaf)], stdout=subprocess.PIPE,
                       stderr=subprocess.STDOUT, text=True, timeout=600)
    assert r.returncode == 0 and r.stdout.rstrip().endswith("ok"), r.stdout[-2000:]


@pytest.mark.gpu
@pytest.mark.parametrize("n,leaf,nrhs,codec", [(1, 32, 1, "aflp"), (40, 1, 2, "none"), (129, 128, 5, "fpx"),
                                               (700, 100, 4, "aflp"), (1000, 33, 9, "aflp"), (2048, 64, 3, "fpx")])
def test_lu_solve_shapes(n, leaf, nrhs, codec):
    """Residual below eps (norm-wise, as the larger solve test) and every column
    equal to its own single solve bit for bit."""
    torch = pytest.importorskip("torch")
    from paper_2405_03456_gb300 import hm
    hbuild.build()
    eps = 1e-6
    pts = synth.cube_points(n)
    a = kernels.entries("matern", pts, np.arange(n), np.arange(n), kernels.default_param("matern", n))
    b = synth.rhs(n, nrhs, seed=41)
    F = hm.HLU(pts, "matern", leaf, 2.0, eps)
    try:
        F.compress(eps, codec, True)
        bd = torch.from_numpy(np.ascontiguousarray(b.T)).cuda().t()
        xd = torch.zeros((nrhs, n), dtype=torch.float64, device="cuda").t()
        F.solve(bd, xd)
        assert F.sync_status() == 0
        x = xd.cpu().numpy()
        for k in range(nrhs):
            res = np.linalg.norm(a @ x[:, k] - b[:, k]) / (np.linalg.norm(a) * np.linalg.norm(x[:, k]))
            assert res <= eps, (k, res)
            xk = torch.zeros(n, dtype=torch.float64, device="cuda")
            F.solve(bd[:, k].contiguous(), xk)
            assert np.array_equal(xk.cpu().numpy().view(np.uint64), x[:, k].copy().view(np.uint64)), k
    finally:
        F.close()
