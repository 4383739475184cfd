"""Batches of a few right-hand sides in the forms that other entry points and options
give them: launches whose warps take more pieces than one load of copy descriptors
(32), the adjoint, HODLR and BLR trees, graph replay.  Every column equals its single
product to 1e-9: a batch runs a single product's operations in the same order inside
a piece, and only the float-float order of a chunk's pieces may differ (about 2^-44;
a coefficient that then rounds to another FP32 multiplier, with probability about
2^-20, moves by 2^-24 of itself)."""
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


@pytest.mark.parametrize("n,kernel,fmt,adm,leaf,eps,counts,adjoint,graph", [
    (40000, "laplace", "h", "std", 8, 1e-4, (4, 8), False, False),     # up to 51 (column dots) and 118 pieces a warp
    (24000, "laplace", "h", "std", 8, 1e-8, (2, 4), False, False),     # the same, float-float
    (2001, "laplace_w", "h", "std", 32, 1e-6, (2, 5, 8), True, False),
    (1500, "laplace_w", "uh_sep", "std", 64, 1e-6, (3,), True, False),
    (1200, "laplace_w", "h2", "std", 32, 1e-8, (4,), True, True),
    (3000, "laplace", "h", "hodlr", 64, 1e-6, (3, 8), False, False),
    (1100, "laplace", "h", "blr", 128, 1e-6, (2, 7), False, True),
    (2500, "laplace", "uh", "std", 64, 1e-6, (4, 6), False, True),
])
def test_batch_forms_equal_single_products(n, kernel, fmt, adm, leaf, eps, counts, adjoint, graph):
    from paper_2405_03456_gb300 import build, hm
    build.build()
    M = hm.HMatrix(synth.sphere_points(n), kernel, leaf, 2.0, fmt, eps, adm=adm)
    try:
        M.compress(eps, "aflp")
        for r in counts:
            x = torch.from_numpy(synth.rhs(n, r, seed=r).T.copy()).cuda().t()
            y0 = torch.from_numpy(synth.rhs(n, r, seed=50 + r).T.copy()).cuda().t()
            M.graph(graph)
            y = y0.t().contiguous().t()
            for _ in range(2 if graph else 1):   # captured, then replayed
                y.copy_(y0)
                M.matvec(0.75, x, -0.5, y, adjoint=adjoint)
            assert M.sync_status() == 0
            M.graph(False)
            for k in range(r):
                ys = y0[:, k].contiguous()
                M.matvec(0.75, x[:, k].contiguous(), -0.5, ys, adjoint=adjoint)
                assert float((y[:, k] - ys).norm()) <= 1e-9 * float(ys.norm()), (r, k)
    finally:
        M.close()
