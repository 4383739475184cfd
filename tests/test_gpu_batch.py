"""Batches of a few right-hand sides (csrc/batch.cu) against single products.

Inside a piece a batch runs the single product's operations in the same order;
only the float-float order of a chunk's pieces may differ (about 2^-44), and a
coefficient whose float-float value moves by that much rounds to another FP32
multiplier with probability about 2^-20 (then by 2^-24 of one coefficient): every
column must equal its single product to 1e-9."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


@pytest.fixture(scope="module")
def hm():
    from paper_2405_03456_gb300 import build, hm as _hm
    build.build()
    _hm.load()
    return _hm


@pytest.mark.parametrize("fmt,leaf,n,eps,codec,counts", [
    ("h", 64, 3001, 1e-6, "aflp", (2, 3, 5, 8)),
    ("h", 7, 700, 1e-4, "fpx", (4, 7)),
    ("h", 128, 1024, 1e-6, "aflp", (8, 34)),
    ("uh", 33, 1500, 1e-6, "fpx", (2, 6)),
    ("h2", 32, 2048, 1e-6, "aflp", (3, 8)),
    ("uh_sep", 64, 1300, 1e-6, "aflp", (5,)),
    ("h", 64, 1, 1e-6, "aflp", (2, 8)),
    ("h", 64, 3001, 1e-8, "aflp", (2, 3, 9)),
    ("h", 50, 900, 1e-8, "fpx", (4, 64)),
    ("uh", 32, 1500, 1e-6, "none", (3,)),
    ("h2", 128, 2048, 1e-8, "aflp", (2, 5)),
])
def test_batch_equals_single_products(hm, fmt, leaf, n, eps, codec, counts):
    M = hm.HMatrix(synth.sphere_points(n), "laplace", leaf, 2.0, fmt, eps)
    try:
        M.compress(eps, codec)
        for r in counts:
            ld = n + 3
            x = torch.from_numpy(synth.rhs(ld, r, seed=r).T.copy()).cuda().t()[:n]
            y0 = torch.from_numpy(synth.rhs(ld, r, seed=50 + r).T.copy()).cuda().t()[:n]
            outs = []
            for _ in range(2):
                y = y0.t().contiguous().t()
                M.matvec(0.75, x, -0.5, y)
                outs.append(y.cpu().numpy())
            assert M.sync_status() == 0
            assert np.array_equal(outs[0], outs[1])
            for k in range(r):
                if eps > 1e-7 and codec != "none" and r >= 9 and k < 32:
                    continue   # those columns run as a panel
                ys = y0[:, k].contiguous()
                M.matvec(0.75, x[:, k].contiguous(), -0.5, ys)
                ys = ys.cpu().numpy()
                assert np.linalg.norm(outs[0][:, k] - ys) <= 1e-9 * np.linalg.norm(ys), (r, k)
    finally:
        M.close()
