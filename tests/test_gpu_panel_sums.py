"""Gather and segment sums of a panel (csrc/mrhs.cu) take one or four right-hand
sides per thread, by the entries of the launch and the partials of a sum: matrices
on both sides of each line, full and ragged panels, every column against its own
single product.  Both sum FP32 partials in float-float; the panel rounds its
coefficients to FP32 (2^-24) where the single product keeps float-float pairs, far
below the 1e-6 asked for."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


@pytest.mark.parametrize("n,fmt,adm,eps", [
    (29183, "h", "std", 1e-4), (29185, "h", "std", 1e-4),   # the gather's line; short sums, many of them
    (8000, "h", "hodlr", 1e-6),                             # long sums
    (29200, "uh", "std", 1e-4),                             # weighted sums
    (33, "h", "std", 1e-6),
])
def test_panel_columns_equal_single_products(n, fmt, adm, eps):
    from paper_2405_03456_gb300 import build, hm
    build.build()
    r = 32 + 9
    M = hm.HMatrix(synth.sphere_points(n), "laplace", 64, 2.0, fmt, eps, adm=adm)
    try:
        M.compress(eps, "aflp")
        x = torch.from_numpy(synth.rhs(n, r, seed=5).T.copy()).cuda().t()
        y0 = torch.from_numpy(synth.rhs(n, r, seed=6).T.copy()).cuda().t()
        y = y0.t().contiguous().t()
        M.matvec(0.75, x, 0.5, y)
        assert M.sync_status() == 0
        for k in (0, 3, 17, 31, 32, 40):
            ys = y0[:, k].contiguous()
            M.matvec(0.75, x[:, k].contiguous(), 0.5, ys)
            assert float((y[:, k] - ys).norm() / ys.norm()) <= 1e-6, k
    finally:
        M.close()
