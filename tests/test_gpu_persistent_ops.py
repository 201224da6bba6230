"""The persistent form of the split-precision operator kernel, which launches of
many tiles take: derivatives and filter at shapes whose launches lie on both
sides of its rule, with ragged tiles, both row-group sizes, the staged radial
epilogue with 48 and 96 rows and the unstaged one (n_r > 80), and at the longest
field of the one-block exponent scan (16 x 16 x 32) and the next above, against
the plain FP64 operators.

Tolerance of the derivatives: the 47-bit fixed point.  Column values are off by
at most 2^-48 2^E <= 2^-47 max|u| and a row's entries by 2^-47 max|W|, so an
operator with K columns is off by at most 2^-46 (rowsum|W| + K max|W|) max|u|;
the chain rule multiplies the three operators by at most 1, 1 / r_in and
1 / (r_in sin theta_0).  The filter's entries are at most of order one and it
rotates a tensor's components into one another: the mixed path's 1e-10 of the
state's maximum."""

import numpy as np
import pytest

from paper_1104_3408_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cf():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1104_3408_gb300 import cffyn
    return cffyn


def _deriv_bound(sh, N, r_in, umax):
    W = [sh.get_operator(w) for w in range(3)]
    jac = (1.0, 1.0 / r_in, 1.0 / (r_in * np.sin(0.5 * np.pi / N)))
    return sum(j * 2.0 ** -46 * (np.abs(w).sum(1).max() + w.shape[1] * np.abs(w).max())
               for j, w in zip(jac, W)) * umax


@pytest.mark.parametrize("n_r,N,fields,rows", [
    (17, 32, 50, 0), (33, 47, 58, 0), (33, 47, 50, 48), (65, 24, 54, 0), (90, 16, 50, 0), (25, 48, 50, 96),
    (16, 16, 50, 0), (17, 16, 58, 0),
])
def test_persistent_launches_match_fp64(cf, n_r, N, fields, rows):
    u = torch.from_numpy(inputs.band_limited_fields(n_r, N, 2 * N, n_fields=fields, seed=n_r, bumps=2)).cuda()
    out = []
    for prec in (cf.MIXED, cf.FP64):
        sh = cf.Shell(n_r, N, 2 * N, 1.8, 11.0, N - 2, n_fields=fields, precision=prec)
        if rows:
            for w in range(5):
                sh.set_operator_rows(w, rows)
        d = torch.empty((3,) + tuple(u.shape), dtype=torch.float64, device="cuda")
        f = torch.empty_like(u)
        sh.derivs(u, d)
        sh.filter(u, f)
        torch.cuda.synchronize()
        out.append((d, f))
        bound = _deriv_bound(sh, N, 1.8, u.abs().amax((1, 2, 3)).cpu().numpy())
        sh.destroy()
    (d, f), (d64, f64) = out
    assert np.isfinite(d.cpu().numpy()).all() and np.isfinite(f.cpu().numpy()).all()
    assert ((d - d64).abs().amax((0, 2, 3, 4)).cpu().numpy() <= bound).all()
    assert float((f - f64).abs().max() / f64.abs().max()) < 1e-10
