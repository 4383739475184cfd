"""Products issued back to back without a synchronisation, each reading what the
one before wrote (the vectors swapped, beta != 0): a kernel that starts before its
predecessor ends must see all of its results, so that the chain equals the same
chain synchronised after every product bit for bit."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


@pytest.mark.parametrize("fmt,n,eps,nrhs", [
    ("h", 4099, 1e-6, 1), ("h", 4099, 1e-6, 4), ("h", 4099, 1e-6, 32), ("h2", 4099, 1e-6, 1), ("uh", 1500, 1e-6, 8),
    ("h", 3001, 1e-8, 1), ("h", 3001, 1e-8, 4),
])
def test_chained_products_equal_synchronised_ones(fmt, n, eps, nrhs):
    from paper_2405_03456_gb300 import build, hm
    build.build()
    M = hm.HMatrix(synth.sphere_points(n), "laplace", 64, 2.0, fmt, eps)
    try:
        M.compress(eps, "aflp")
        x0 = torch.from_numpy(synth.rhs(n, nrhs, seed=3).T.copy()).cuda()
        y0 = torch.from_numpy(synth.rhs(n, nrhs, seed=4).T.copy()).cuda()

        def chain(sync):
            u, v = (t.clone()[0] if nrhs == 1 else t.clone().t() for t in (x0, y0))
            for _ in range(16):
                M.matvec(0.25, u, -0.5, v)
                u, v = v, u
                if sync:
                    torch.cuda.synchronize()
            return np.stack([u.cpu().numpy(), v.cpu().numpy()])

        ref = chain(True)
        assert np.isfinite(ref).all()
        for _ in range(4):
            assert np.array_equal(chain(False).view(np.uint64), ref.view(np.uint64))
        assert M.sync_status() == 0
    finally:
        M.close()
