"""The FP64 operator kernel at every rows-per-warp variant (operator rows 3 to 112:
one and two row tiles, with and without a remainder of eight), derivatives
against the oracle.  Tolerance: the rounding of two dot products of K terms,
2 K eps rowsum|W| max|u| per operator, times the chain rule's largest factors."""

import numpy as np
import pytest

from oracle import cff
from paper_1104_3408_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_r,N", [(3, 2), (8, 6), (17, 9), (26, 14), (33, 18), (41, 23), (52, 26), (64, 31), (65, 33),
                                   (9, 55)])
def test_fp64_derivatives_at_every_tile_height(n_r, N):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1104_3408_gb300 import cffyn as cf
    u = inputs.band_limited_fields(n_r, N, 2 * N, n_fields=50, seed=N, bumps=1)
    sh = cf.Shell(n_r, N, 2 * N, 1.8, 11.0, max(0, N - 2), precision=cf.FP64)
    out = torch.empty((3,) + u.shape, dtype=torch.float64, device="cuda")
    sh.derivs(torch.from_numpy(u).cuda(), out)
    ref = cff.cartesian_derivatives(u, 1.8, 11.0)
    jac = (1.0, 1.0 / 1.8, 1.0 / (1.8 * np.sin(0.5 * np.pi / N)))
    bound = sum(j * 2 * w.shape[1] * np.finfo(float).eps * np.abs(w).sum(1).max()
                for j, w in zip(jac, (sh.get_operator(q) for q in range(3)))) * np.abs(u).max()
    sh.destroy()
    assert np.abs(out.cpu().numpy() - ref).max() <= bound
