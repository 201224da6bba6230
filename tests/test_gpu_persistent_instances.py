"""Every instance of the persistent operator kernel that d_r has: outputs staged as
one tile beside copied inputs (odd n_r up to 39), staged alone with 48 rows (even
n_r, 41..47) and with 96 (up to 80), and the one-item kernel that it has above.
The shapes are sized from the device's SM count and from the lines read off the rule
itself, so that a changed line keeps them on the persistent side; every one has a
ragged last tile.

FP64 words in: the derivatives against the plain FP64 operators, within the bound of
the 47-bit fixed point (an operator with K columns: 2^-46 (rowsum|W| + K max|W|)
max|u|; the chain rule multiplies the three by at most 1, 1 / r_in and 1 / (r_in
sin theta_0)).  Pairs in: an RK4 step of shells stacked in a batch, whose launches
are persistent, against the shells one by one, whose d_r is not, bit for bit."""

import os
import re

import numpy as np
import pytest

from paper_1104_3408_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# n_r: one, two and three k-steps, the ends of each form's range
N_R = [4, 9, 24, 33, 39, 40, 41, 48, 49, 80, 81, 96]


@pytest.fixture(scope="module")
def cf():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1104_3408_gb300 import cffyn
    return cffyn


def line(n_r):
    """Items (tiles of 128 columns) above which d_r runs on the persistent kernel."""
    import paper_1104_3408_gb300 as pkg
    with open(os.path.join(os.path.dirname(pkg.__file__), "csrc", "ops.cu")) as fh:
        per_sm = re.search(r"return items > \(rows != 48 \? (\d+) : dr \? (\d+) : \d+\) \* \(long long\)sh->sm_count;",
                           fh.read())
    return int(per_sm.group(1 if n_r > 48 else 2)) * torch.cuda.get_device_properties(0).multi_processor_count


def items(columns):
    return -(-columns // 128)


@pytest.mark.parametrize("n_r", N_R)
def test_derivatives_of_fp64_words(cf, n_r):
    N = 2
    while items(100 * N * N) <= 1.05 * line(n_r) or 100 * N * N % 128 == 0:
        N += 1
    u = torch.from_numpy(inputs.band_limited_fields(n_r, N, 2 * N, n_fields=50, seed=n_r, bumps=1)).cuda()
    out = []
    for prec in (cf.MIXED, cf.FP64):
        sh = cf.Shell(n_r, N, 2 * N, 1.8, 11.0, N - 2, precision=prec)
        d = torch.empty((3,) + tuple(u.shape), dtype=torch.float64, device="cuda")
        sh.derivs(u, d)
        out.append(d)
        jac = (1.0, 1.0 / 1.8, 1.0 / (1.8 * np.sin(0.5 * np.pi / N)))
        bound = sum(j * 2.0 ** -46 * (np.abs(w).sum(1).max() + w.shape[1] * np.abs(w).max())
                    for j, w in zip(jac, (sh.get_operator(q) for q in range(3)))) * float(u.abs().max())
        sh.destroy()
    assert float((out[0] - out[1]).abs().max()) <= bound


# (54 and 58 fields: the gauge fields' right-hand sides and time derivatives are zero)
@pytest.mark.parametrize("n_r,fields", [(n, 50) for n in N_R] + [(17, 54), (17, 58), (24, 58), (49, 54), (49, 58)])
def test_stacked_steps_of_pairs(cf, n_r, fields):
    N = 18 if n_r <= 48 else 12
    M = 2
    while items(2 * fields * N * N * M) <= 1.05 * line(n_r) or 2 * fields * N * N * M % 128 == 0:
        M += 1
    assert items(2 * fields * N * N) <= line(n_r)
    shells, us = [], []
    for q in range(M):
        u = torch.from_numpy(inputs.kerr_schild_state(n_r, N, 2 * N, 1.8, 11.0, n_fields=fields, amp=1e-4, ell=2,
                                                      seed=q)).cuda()
        shells.append(cf.Shell(n_r, N, 2 * N, 1.8, 11.0, N - 2, n_fields=fields))
        shells[-1].init_gauge_from_state(u)
        us.append(u)
    alone = [u.clone() for u in us]
    dt = shells[0].default_dt()
    for sh, u in zip(shells, alone):
        sh.rk4_step(u, dt, 1)
    b = cf.Batch(shells)
    assert b.units() == 1
    b.rk4_step(us, [dt] * M, 1)
    torch.cuda.synchronize()
    for x, y in zip(us, alone):
        assert torch.isfinite(x).all() and torch.equal(x, y)
    b.destroy()
    for sh in shells:
        sh.destroy()
