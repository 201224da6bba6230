"""The right-hand-side and reconstruction kernels that share a point's tensors out
over several warps (small launches) against those with one thread per point or
tensor group: a small shell stepped alone takes the former, the same shell in a
batch beside a large one the latter, and the states agree bit for bit.  Point
counts with and without a remainder of 32, all field counts, both filter
placements, both precisions."""

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


@pytest.mark.parametrize("n_r,N,fields,kind,mode,prec", [
    (3, 2, 50, 0, 0, 1), (13, 9, 50, 0, 1, 1), (13, 9, 58, 0, 0, 1), (9, 7, 54, 2, 1, 1), (17, 16, 50, 1, 0, 1),
    (7, 5, 58, 0, 0, 0),
])
def test_shared_out_points_match_one_thread_per_point(cf, n_r, N, fields, kind, mode, prec):
    def shell(n_r, N):
        u = torch.from_numpy(inputs.kerr_schild_state(n_r, N, 2 * N, 1.8, 11.0, n_fields=fields, amp=1e-4, ell=2,
                                                      seed=N)).cuda()
        sh = cf.Shell(n_r, N, 2 * N, 1.8, 11.0, max(0, N - 3), n_fields=fields, precision=prec, filter_mode=mode,
                      filter_kind=kind)
        sh.init_gauge_from_state(u)
        return sh, u

    small, u = shell(n_r, N)
    large, v = shell(33, 40)
    alone = u.clone()
    small.rk4_step(alone, 1e-3, 2)
    b = cf.Batch([small, large])
    b.rk4_step([u, v], [1e-3, 1e-3], 2)
    torch.cuda.synchronize()
    assert torch.isfinite(alone).all() and torch.equal(alone, u)
    b.destroy()
    small.destroy()
    large.destroy()
