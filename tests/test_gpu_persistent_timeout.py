"""The persistent operator kernel when its waits give up (a wait bound of 0: every
pipeline wait ends at once): each role leaves its loop by itself, the copies,
products and bulk stores already issued are waited for, the tensor memory is freed,
the step reports CFFYN_ETIMEOUT, and with the default bound restored the same
handle steps as before.  One shape for each form of d_r (inputs copied and outputs
staged, staged with 48 and with 96 rows, and above 80 rows the one-item kernel),
large enough that the angular derivatives and the filter run persistently too."""

import pytest

from paper_1104_3408_gb300 import inputs
from test_gpu_persistent_instances import cf, items, line  # noqa: F401 (cf: the fixture)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_r", [17, 24, 49, 81])
def test_persistent_step_reports_timeout_and_recovers(cf, n_r):  # noqa: F811
    N = 2
    while items(100 * N * N) <= 1.05 * max(line(n_r), line(24)):
        N += 1
    sh = cf.Shell(n_r, N, 2 * N, 1.8, 11.0, N - 2)
    u = torch.from_numpy(inputs.kerr_schild_state(n_r, N, 2 * N, 1.8, 11.0, amp=1e-6, ell=2, seed=0)).cuda()
    sh.init_gauge_from_state(u)
    dt = sh.default_dt()
    ref = u.clone()
    sh.rk4_step(ref, dt, 1)
    sh.set_wait_limit(0.0)
    with pytest.raises(cf.CffynError) as ei:
        sh.rk4_step(u.clone(), dt, 1)
    assert ei.value.code == cf.ETIMEOUT and "gave up" in str(ei.value)
    sh.set_wait_limit(-1.0)
    again = u.clone()
    sh.rk4_step(again, dt, 1)
    torch.cuda.synchronize()
    assert torch.isfinite(again).all() and torch.equal(again, ref)
    sh.destroy()
