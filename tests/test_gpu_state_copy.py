"""The copy of a caller's state into a shell's own storage (one word per thread for
small states, four for large ones): the scalar Y filter, which starts with that
copy, against the oracle on both sides of the line and with last blocks that are
partly filled.  A second state in the workspace beforehand shows a word left out
as an error of order one; the tolerances are those of the filter itself."""

import numpy as np
import pytest

import oracle
from paper_1104_3408_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = {0: 1e-12, 1: 1e-10}  # FP64, mixed


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n_r,N", [(3, 3), (25, 22), (25, 23), (26, 24), (33, 23)])
def test_filter_of_a_copied_state(n_r, N, prec):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1104_3408_gb300 import cffyn as cf
    L = max(0, N - 3)
    u = inputs.band_limited_fields(n_r, N, 2 * N, 1.8, 11.0, seed=N)
    ref = oracle.OracleShell(n_r, N, 2 * N, 1.8, 11.0, L, filter_kind="y").filter(u)
    sh = cf.Shell(n_r, N, 2 * N, 1.8, 11.0, L, precision=prec, filter_kind=1)
    v = torch.from_numpy(np.ascontiguousarray(u)).cuda()
    out = torch.empty_like(v)
    sh.filter(v.flip(0).contiguous() + 3.0, out)
    sh.filter(v, out)
    got = out.cpu().numpy()
    sh.destroy()
    err = np.abs(got - ref).reshape(len(u), -1).max(1) / np.abs(ref).reshape(len(u), -1).max(1)
    assert err.max() < TOL[prec], err.max()
