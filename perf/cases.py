"""Timed cases of the framework: what a user's program has the library do, from
the paper's smallest single black hole runs to the largest benchmarked shell.

Every case goes through the Python binding (paper_1104_3408_gb300.cffyn).  Each
pass of a stepping case starts from the case's state (copied into the stepped
buffer, as a program that works through independent problems does), so passes
are alike.  Kinds: "step" (RK4 steps of one shell), "rhs", "derivs", "filter",
"nest" (RK4 steps of two nested shells), "batch" (RK4 steps of uneven shells).

exact() restates the method (Bruegmann, arXiv:1104.3408) in plain torch and
numpy FP64, without the framework: grid and differentiation matrices (Secs.
2.1-2.3), the spin-weighted filter (Secs. 3.4, 3.5), the GHG right-hand side
with its outer boundary condition (App. A), RK4 (Sec. 2.5) and the
characteristic coupling of nested shells.
"""

import itertools
import math

import numpy as np
import torch

PAIRS = [(0, 0), (0, 1), (0, 2), (0, 3), (1, 1), (1, 2), (1, 3), (2, 2), (2, 3), (3, 3)]
FILTERS = {"yn": 0, "y": 1, "yg": 2}
RHS_OPS = 7168  # FP64-equivalent operations of the right-hand side per point


def _shell(kind, n_r, n_theta, L, r_out=11.0, fields=50, precision="mixed", filter="yn", placement="substep",
           courant=0.25, steps=1, amp=1e-4, ell=4):
    return dict(kind=kind, n_r=n_r, n_theta=n_theta, L=L, r_out=r_out, fields=fields, precision=precision,
                filter=filter, placement=placement, courant=courant, steps=steps, amp=amp, ell=ell)


def listed():
    return [
        # the paper's smallest R10 run: the Yn filter with n_f = 4 after every
        # step, dt = 4 min dx, 20 steps between two samples of the monitor
        dict(name="r10_13x9x18", **_shell("step", 13, 9, 4, 11.8, placement="step", courant=4.0, steps=20,
                                          amp=1e-6, ell=2)),
        # R10 as two nested shells coupled on their common sphere
        dict(name="nest_2x13x9x18", **_shell("nest", 13, 9, 4, 11.8, placement="step", courant=1.0, steps=10,
                                             amp=1e-6, ell=2)),
        # a finer odd-sized R10 grid with the graded component-wise filter
        dict(name="r10_yg_25x15x30", **_shell("step", 25, 15, 10, 11.8, filter="yg", placement="step", courant=4.0,
                                              steps=5, amp=1e-6, ell=2)),
        # a middle-sized shell, Yn filter on every stage
        dict(name="step_25x24x48", **_shell("step", 25, 24, 22, steps=2)),
        # the plain FP64 path that the mixed path is checked against
        dict(name="step_fp64_17x16x32", **_shell("step", 17, 16, 14, precision="fp64")),
        # operator micro-benchmark: Cartesian derivatives and the Yn filter of
        # 50 band-limited fields
        dict(name="derivs_33x32x64", **_shell("derivs", 33, 32, 30)),
        dict(name="filter_33x32x64", **_shell("filter", 33, 32, 30)),
        # one right-hand side of the benchmark shell (monitoring, own integrators)
        dict(name="rhs_33x48x96", **_shell("rhs", 33, 48, 46, amp=1e-3)),
        # the benchmark shell: one RK4 step, Yn filter on every stage
        dict(name="step_33x48x96", **_shell("step", 33, 48, 46)),
        # independent shells of uneven resolution advanced together
        dict(name="batch_8", kind="batch", grids="17x16,25x16,17x24,17x24,33x24,25x32,25x32,33x48", L=-2, r_out=11.0,
             fields=50, precision="mixed", filter="yn", placement="substep", courant=0.25, steps=2, amp=1e-4, ell=4),
        # the largest shell: 58 fields with an evolved gauge
        dict(name="step_65x96x192_58f", **_shell("step", 65, 96, 94, 41.0, fields=58)),
    ]


def _between(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "rhs", "derivs", "filter", "nest", "batch"])
    small = kind in ("nest", "batch")
    n_theta, n_r = _between(rng, 8, 32 if small else 90), _between(rng, 9, 33 if small else 65)
    points = 2 * n_r * n_theta ** 2
    r10 = rng.random() < 0.3
    c = _shell(kind, n_r, n_theta, n_theta - 5 if r10 else n_theta - 2, rng.choice([11.0, 11.8, 21.0]),
               fields=rng.choice([50, 50, 54, 58]), filter=rng.choice(["yn", "yn", "yn", "y", "yg"]),
               placement="step" if r10 else "substep", courant=1.0 if r10 else 0.25,
               steps=rng.choice([5, 10, 20]) if points < 8000 else (2 if points < 60000 else 1),
               amp=1e-6 if r10 else 1e-4, ell=2 if r10 else 4)
    if points < 60000 and rng.random() < 0.15:
        c["precision"] = "fp64"
    if kind == "rhs":
        c["amp"] = 1e-3
    if kind == "batch":
        c.pop("n_r"), c.pop("n_theta")
        grids = [(rng.choice([17, 25, 33]), rng.choice([16, 24, 32])) for _ in range(rng.randint(2, 4))]
        c["grids"] = ",".join("%dx%d" % g for g in grids + [grids[0]] * rng.randint(0, 2))
        c["L"], c["fields"] = -2, 50
    return c


# ---------------------------------------------------------------------------
# Inputs

def _grids(case):
    """(n_r, n_theta, r_in, r_out) of the case's shells."""
    if case["kind"] == "batch":
        return [(*map(int, g.split("x")), 1.8, case["r_out"]) for g in case["grids"].split(",")]
    n_r, N, r1 = case["n_r"], case["n_theta"], case["r_out"]
    if case["kind"] == "nest":
        mid = 0.5 * (1.8 + r1)
        return [(n_r, N, 1.8, mid), (n_r, N, mid, r1)]
    return [(n_r, N, 1.8, r1)]


def _degree(case, N):
    return case["L"] if case["L"] >= 0 else N + case["L"]


def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _points(n_r, N, r_in, r_out):
    k, i, j = (torch.arange(n, dtype=torch.float64, device=_dev()) for n in (n_r, N, 2 * N))
    r = 0.5 * (r_out + r_in) - 0.5 * (r_out - r_in) * torch.cos(math.pi * k / (n_r - 1))
    return r, math.pi * (i + 0.5) / N, math.pi * j / N


def _normal(theta, phi):
    """n_i = x_i / r on the sphere: [3, J, N]."""
    st, ct = torch.sin(theta)[None], torch.cos(theta)[None]
    sp, cp = torch.sin(phi)[:, None], torch.cos(phi)[:, None]
    return torch.stack([st * cp, st * sp, ct.expand(len(phi), -1)])


def _ghg_state(n_r, N, r_in, r_out, fields, amp, ell, seed, center, width):
    """Schwarzschild in Kerr-Schild form (mass 1) plus a smooth perturbation of
    degree <= ell on every sphere; Phi_iab = d_i g_ab, Pi_ab for d_t g_ab = 0."""
    r, theta, phi = _points(n_r, N, r_in, r_out)
    n = _normal(theta, phi)[..., None].expand(-1, -1, -1, n_r)
    R = r.expand(n.shape[1:])
    X = n * R
    f = 2.0 / R
    l4 = torch.cat([torch.ones_like(R)[None], n])
    eye = torch.eye(3, dtype=torch.float64, device=R.device)
    coef = np.random.default_rng(seed)
    xs = X / center
    G = torch.exp(-((R - center) / width) ** 2)
    dG = -2.0 * (R - center) / width ** 2 * G
    monos = [m for m in itertools.product(range(ell + 1), repeat=3) if sum(m) <= ell]
    powers = [[xs[i] ** e for e in range(ell + 1)] for i in range(3)]
    u = torch.zeros((fields,) + tuple(R.shape), dtype=torch.float64, device=R.device)
    dl = torch.zeros((3, 4) + tuple(R.shape), dtype=torch.float64, device=R.device)
    for i in range(3):
        for j in range(3):
            dl[i, j + 1] = (eye[i, j] - n[i] * n[j]) / R
    for s, (a, b) in enumerate(PAIRS):
        Q, dQ = torch.zeros_like(R), torch.zeros_like(X)
        for c, m in zip(coef.standard_normal(len(monos)) / math.sqrt(len(monos)), monos):
            Q += c * powers[0][m[0]] * powers[1][m[1]] * powers[2][m[2]]
            for i in range(3):
                if m[i]:
                    e = [m[q] - (q == i) for q in range(3)]
                    dQ[i] += c * m[i] / center * powers[0][e[0]] * powers[1][e[1]] * powers[2][e[2]]
        eta = (-1.0 if a == 0 else 1.0) if a == b else 0.0
        u[s] = eta + f * l4[a] * l4[b] + amp * G * Q
        for i in range(3):
            u[20 + 10 * i + s] = (-f / R * n[i] * l4[a] * l4[b] + f * (dl[i, a] * l4[b] + l4[a] * dl[i, b])
                                  + amp * (dG * n[i] * Q + G * dQ[i]))
    alpha, bu = _three_plus_one(_sym(u[:10]))[:2]
    for s in range(10):
        u[10 + s] = sum(bu[i] * u[20 + 10 * i + s] for i in range(3)) / alpha
    return u


def _smooth_fields(n_r, N, r_in, r_out, fields, seed):
    """Band-limited fields: six von-Mises bumps on the sphere, each times a
    Chebyshev series in r with coefficients falling as 10^(-q/4)."""
    rng = np.random.default_rng(seed)
    r, theta, phi = _points(n_r, N, r_in, r_out)
    put = lambda a: torch.from_numpy(a).to(r.device)  # noqa: E731
    e = rng.standard_normal((fields, 6, 3))
    e = put(e / np.linalg.norm(e, axis=-1, keepdims=True))
    kappa, w = put(rng.uniform(1.0, 6.0, (fields, 6, 1, 1))), put(rng.standard_normal((fields, 6, 1, 1)))
    c = put(rng.standard_normal((fields, 6, n_r)) * 10.0 ** (-np.arange(n_r) / 4.0))
    x = torch.acos(((2.0 * r - r_in - r_out) / (r_out - r_in)).clamp(-1.0, 1.0))
    cheb = torch.cos(torch.arange(n_r, dtype=torch.float64, device=r.device)[:, None] * x)
    ang = w * torch.exp(kappa * (torch.einsum("fbx,xji->fbji", e, _normal(theta, phi)) - 1.0))
    return torch.einsum("fbji,fbk->fjik", ang, c @ cheb).contiguous()


def _states(case, seed):
    out = []
    grids = _grids(case)
    r0, r1 = grids[0][2], grids[-1][3]
    for q, (n_r, N, a, b) in enumerate(grids):
        if case["kind"] in ("derivs", "filter"):
            out.append(_smooth_fields(n_r, N, a, b, case["fields"], seed))
        else:
            # a batch's shells hold different perturbations, nested shells one
            s = seed * 1009 + q if case["kind"] == "batch" else seed
            out.append(_ghg_state(n_r, N, a, b, case["fields"], case["amp"], case["ell"], s,
                                  0.5 * (r0 + r1), (r1 - r0) / 8.0))
    return out


# ---------------------------------------------------------------------------
# The calls

def prepare(case, seed):
    from paper_1104_3408_gb300 import cffyn
    shells, u0 = [], _states(case, seed)
    for (n_r, N, a, b), u in zip(_grids(case), u0):
        sh = cffyn.Shell(n_r, N, 2 * N, a, b, _degree(case, N), n_fields=case["fields"],
                         precision=cffyn.MIXED if case["precision"] == "mixed" else cffyn.FP64,
                         filter_mode=cffyn.FILTER_STEP if case["placement"] == "step" else cffyn.FILTER_SUBSTEP,
                         courant=case["courant"], filter_kind=FILTERS[case["filter"]])
        if case["kind"] not in ("derivs", "filter"):
            sh.init_gauge_from_state(u)
        shells.append(sh)
    s = dict(case=case, shells=shells, u0=u0)
    if case["kind"] == "derivs":
        s["out"] = torch.empty((3,) + tuple(u0[0].shape), dtype=torch.float64, device=u0[0].device)
    else:
        s["out"] = [torch.empty_like(u) for u in u0]
    if case["kind"] == "nest":
        s["group"] = cffyn.Nest(shells)
    if case["kind"] == "batch":
        s["group"] = cffyn.Batch(shells)
    return s


def run(state):
    case, sh, u0, out = state["case"], state["shells"], state["u0"], state["out"]
    if case["kind"] == "derivs":
        return sh[0].derivs(u0[0], out)
    if case["kind"] == "filter":
        return sh[0].filter(u0[0], out[0])
    if case["kind"] == "rhs":
        return sh[0].rhs(u0[0], out[0])
    for u, v in zip(out, u0):
        u.copy_(v)
    if case["kind"] == "nest":
        return state["group"].rk4_step(out, 0.0, case["steps"])
    if case["kind"] == "batch":
        return state["group"].rk4_step(out, None, case["steps"])
    return sh[0].rk4_step(out[0], 0.0, case["steps"])


def work(case):
    """The state read once and the result written once; the dense operators'
    and the right-hand side's own FP64 operations."""
    nv, nbytes, flops = case["fields"], 0.0, 0.0
    for n_r, N, _, _ in _grids(case):
        points = 2 * n_r * N * N
        nbytes += 8.0 * nv * points * (4 if case["kind"] == "derivs" else 2)
        derivs = 2 * n_r + 4 * N + 4 * N
        filt = 4 * N + 2 * (_degree(case, N) + 1) + 4 * N
        rhs = derivs * nv + RHS_OPS
        if case["kind"] == "derivs":
            flops += points * nv * derivs
        elif case["kind"] == "filter":
            flops += points * nv * filt
        elif case["kind"] == "rhs":
            flops += points * rhs
        else:
            flops += case["steps"] * points * (4 * rhs + (4 if case["placement"] == "substep" else 1) * filt * nv)
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------
# The method in plain FP64

def _sym(block):
    """Ten symmetric pairs -> [4, 4, ...]."""
    out = torch.empty((4, 4) + tuple(block.shape[1:]), dtype=block.dtype, device=block.device)
    for s, (a, b) in enumerate(PAIRS):
        out[a, b] = block[s]
        out[b, a] = block[s]
    return out


def _pack(T):
    return torch.stack([T[a, b] for a, b in PAIRS])


def _three_plus_one(g):
    """alpha, beta^i, gamma^ij, n^a, g^ab (eqs. normal, abgfromgab)."""
    m = g[1:, 1:]
    c = lambda i, j: (m[(i + 1) % 3, (j + 1) % 3] * m[(i + 2) % 3, (j + 2) % 3]  # noqa: E731
                      - m[(i + 1) % 3, (j + 2) % 3] * m[(i + 2) % 3, (j + 1) % 3])
    det = sum(m[0, j] * c(0, j) for j in range(3))
    gi = torch.stack([torch.stack([c(j, i) / det for j in range(3)]) for i in range(3)])
    bu = torch.stack([sum(gi[i, j] * g[0, j + 1] for j in range(3)) for i in range(3)])
    alpha = torch.sqrt(sum(g[0, i + 1] * bu[i] for i in range(3)) - g[0, 0])
    n = torch.cat([torch.ones_like(alpha)[None], -bu]) / alpha
    g4 = -torch.einsum("a...,b...->ab...", n, n)
    g4[1:, 1:] += gi
    return alpha, bu, gi, n, g4


class _Method:
    """One shell of the method (see the module's docstring)."""

    def __init__(self, case, grid):
        n_r, N, a, b = grid
        self.N, self.J, self.nv, self.kind = N, 2 * N, case["fields"], case["filter"]
        self.L = _degree(case, N)
        self.r, self.theta, self.phi = _points(n_r, N, a, b)
        dev = self.r.device
        fourier = lambda n: torch.tensor(  # noqa: E731
            [[0.0 if i == j else (-1.0) ** (i + j) / (2.0 * math.tan(math.pi * (i - j) / n)) for j in range(n)]
             for i in range(n)], dtype=torch.float64, device=dev)
        x = [-math.cos(math.pi * k / (n_r - 1)) for k in range(n_r)]
        c = [2.0 if k in (0, n_r - 1) else 1.0 for k in range(n_r)]
        D = np.array([[0.0 if i == j else c[i] / c[j] * (-1.0) ** (i + j) / (x[i] - x[j]) for j in range(n_r)]
                      for i in range(n_r)])
        D -= np.diag(D.sum(axis=1))
        self.Dr = torch.from_numpy(2.0 * D / (b - a)).to(dev)
        self.Df = fourier(self.J)  # phi, and theta over the double cover (2 N points)
        self.n = _normal(self.theta, self.phi)
        st, sp, cp = torch.sin(self.theta)[None, :, None], torch.sin(self.phi)[:, None, None], torch.cos(self.phi)[:, None, None]
        ct = torch.cos(self.theta)[None, :, None]
        one = torch.ones_like(self.r).expand(self.J, N, n_r)
        rr = self.r[None, None, :]
        self.jac = [[(v * one).reshape(-1) for v in row] for row in (
            (st * cp, ct * cp / rr, -sp / (rr * st)), (st * sp, ct * sp / rr, cp / (rr * st)), (ct, -st / rr, 0.0 * rr))]
        self.F = {}
        th0, dphi = math.pi * 0.5 / N, math.pi / N
        self.dx = min(float(self.r[1] - self.r[0]), 2.0 * a * math.sin(th0) * math.sin(0.5 * dphi))
        self.H = self.dH = None

    def derivs(self, u):
        """Cartesian derivatives [3, fields, J, N, n_r] (eqs. D1-D3, dvdx)."""
        nf = u.shape[0]
        ext = torch.cat([u, torch.roll(u, -self.N, 1).flip(2)], 2)
        d = (u @ self.Dr.T, torch.matmul(self.Df[:self.N], ext), torch.matmul(self.Df, u.reshape(nf, self.J, -1)).reshape(u.shape))
        d = [v.reshape(nf, -1) for v in d]
        out = torch.stack([sum(j * v for j, v in zip(row, d)) for row in self.jac])
        return out.reshape((3,) + tuple(u.shape))

    def christoffel(self, Pi, Phi, alpha, bu, g4):
        d = torch.cat([(-alpha * Pi + torch.einsum("iP,iabP->abP", bu, Phi))[None], Phi])
        G = 0.5 * (d.permute(2, 0, 1, 3) + d.permute(2, 1, 0, 3) - d)  # [c, a, b]
        return G, torch.einsum("abP,cabP->cP", g4, G)

    def split(self, u):
        f = u.reshape(u.shape[0], -1)
        return _sym(f[:10]), _sym(f[10:20]), torch.stack([_sym(f[20 + 10 * i:30 + 10 * i]) for i in range(3)])

    def start(self, u):
        """The gauge source H_a = -Gamma_a (eq. gauge): fixed, or into the state."""
        g, Pi, Phi = self.split(u)
        alpha, bu, _, _, g4 = _three_plus_one(g)
        H = -self.christoffel(Pi, Phi, alpha, bu, g4)[1].reshape((4,) + tuple(u.shape[1:]))
        u = u.clone()
        if self.nv > 50:
            u[50:54] = H
            u[54:] = 0.0
        else:
            self.H, self.dH = H, self.derivs(H)
        return u

    def rhs(self, u, outer=True):
        """Eqs. gdot, Phidot, Pidot with gamma_0 = gamma_2 = 1, gamma_1 = -1,
        and the freeze-incoming condition of App. A.2 on the outer sphere."""
        du = self.derivs(u)
        H, dH = (self.H, self.dH) if self.nv == 50 else (u[50:54], du[:, 50:54])
        H, dH, f = H.reshape(4, -1), dH.reshape(3, 4, -1), u.reshape(self.nv, -1)
        g, Pi, Phi = self.split(u)
        al, bu, gi, n, g4 = _three_plus_one(g)
        G, Gc = self.christoffel(Pi, Phi, al, bu, g4)
        d = [self.split(du[k]) for k in range(3)]
        dg, dPi = torch.stack([v[0] for v in d]), torch.stack([v[1] for v in d])
        dPhi = torch.stack([v[2] for v in d])
        del d, du
        dH4 = torch.cat([f[54:58][None] if self.nv == 58 else torch.zeros_like(dH[:1]), dH])
        DH = dH4 - torch.einsum("cP,cabP->abP", torch.einsum("cdP,dP->cP", g4, H), G)
        C = H + Gc
        nPhi = torch.einsum("cP,icdP->idP", n, Phi)
        nnPhi = torch.einsum("dP,idP->iP", n, nPhi)
        dtPhi = (torch.einsum("kP,kiabP->iabP", bu, dPhi) - al * dPi + al * dg - al * Phi
                 + 0.5 * al * nnPhi[:, None, None] * Pi
                 + al * torch.einsum("ikP,kabP->iabP", torch.einsum("jkP,ijP->ikP", gi, nPhi[:, 1:]), Phi))
        up = torch.einsum("cdP,iacP->iadP", g4, Phi)
        Q = torch.einsum("jadP,jbdP->abP", torch.einsum("ijP,iadP->jadP", gi, up), Phi)
        Q = Q - torch.einsum("adP,bdP->abP", torch.einsum("cdP,acP->adP", g4, Pi), Pi)
        GG = torch.einsum("efP,adeP->adfP", g4, torch.einsum("cdP,aceP->adeP", g4, G))
        Q = Q - torch.einsum("adfP,bdfP->abP", GG, G)
        nPi = torch.einsum("cP,cdP->dP", n, Pi)
        nlo = torch.zeros_like(n)
        nlo[0] = -al
        nC = torch.einsum("aP,bP->abP", nlo, C)
        dtPi = (torch.einsum("kP,kabP->abP", bu, dPi) - al * torch.einsum("ikP,kiabP->abP", gi, dPhi) - torch.einsum("kP,kabP->abP", bu, dg)
                + 2.0 * al * Q - al * (DH + DH.transpose(0, 1)) - 0.5 * al * torch.einsum("dP,dP->P", n, nPi) * Pi
                - al * torch.einsum("jP,jabP->abP", torch.einsum("iP,ijP->jP", nPi[1:], gi), Phi)
                + al * (nC + nC.transpose(0, 1) - g * torch.einsum("cP,cP->P", n, C)) + torch.einsum("iP,iabP->abP", bu, Phi))
        dtg = -al * Pi + torch.einsum("iP,iabP->abP", bu, Phi)
        out = torch.zeros_like(f)
        out[:10], out[10:20] = _pack(dtg), _pack(dtPi)
        for i in range(3):
            out[20 + 10 * i:30 + 10 * i] = _pack(dtPhi[i])
        if self.nv == 58:
            out[50:54] = f[54:58]
        out = out.reshape(u.shape)
        if outer:
            o = out[..., -1]
            sl, su = self.sphere_normal(u[..., -1])
            w = o[10:20] + sum(su[i] * o[20 + 10 * i:30 + 10 * i] for i in range(3))
            phi = [0.5 * sl[i] * (w - o[:10]) for i in range(3)]
            out[10:20, ..., -1] = 0.5 * (o[:10] + w)
            for i in range(3):
                out[20 + 10 * i:30 + 10 * i, ..., -1] = phi[i]
        return out

    def sphere_normal(self, u):
        """s_i and s^i of a sphere from the state on it (u[fields, J, N])."""
        gi = _three_plus_one(_sym(u[:10]))[2]
        sl = self.n / torch.sqrt(torch.einsum("ij...,i...,j...->...", gi, self.n, self.n))
        return sl, torch.einsum("ij...,j...->i...", gi, sl)

    def projectors(self, L):
        """F^n_m for n = 0..3 and every |m| < N in the order of the FFT (eq.
        FasPfQ with the recursion of eq. Yninc), [4, J, N, N]; F^-n_m = F^n_-m."""
        if L in self.F:
            return self.F[L]
        N = self.N
        th = self.theta.cpu().numpy()
        x, s = np.cos(th), np.sin(th)
        m = np.arange(-(N - 1), N)
        P = np.zeros((4, N, 2 * N - 1, N))  # n, l, m, theta
        sect = 1.0 / math.sqrt(4.0 * math.pi)
        for l in range(N):
            if l:
                sect *= -math.sqrt((2 * l + 1.0) / (2 * l))
                for q in range(l):
                    v = x * P[0, l - 1, N - 1 + q]
                    if l - 2 >= q:
                        v = v - math.sqrt(((l - 1.0) ** 2 - q * q) / (4.0 * (l - 1.0) ** 2 - 1.0)) * P[0, l - 2, N - 1 + q]
                    P[0, l, N - 1 + q] = math.sqrt((4.0 * l * l - 1.0) / (l * l - q * q)) * v
            P[0, l, N - 1 + l] = sect * s ** l
            for q in range(1, l + 1):
                P[0, l, N - 1 - q] = (-1.0) ** q * P[0, l, N - 1 + q]
        for n in range(1, 4):
            for l in range(n, N):
                ok = np.abs(m) <= l
                mm = m[ok][:, None]
                al = math.sqrt((l - n + 1.0) / (l + n))
                be = np.sqrt((2 * l + 1.0) / (2 * l - 1.0) * (l + n - 1.0) * (l * l - mm * mm) / (l + n)) / l
                P[n, l, ok] = al * (mm / l - x) / s * P[n - 1, l, ok] + be / s * P[n - 1, l - 1, ok]
        P = np.moveaxis(P, 1, 3)  # n, m, theta, l
        F = np.zeros((4, 2 * N, N, N))
        F[:, m % (2 * N)] = P[..., :L + 1] @ np.linalg.pinv(P, rcond=N * 2.3e-16)[..., :L + 1, :]
        self.F[L] = torch.from_numpy(F).to(self.r.device)
        return self.F[L]

    def project(self, f, n, L):
        """Complex functions f[c, J, N, n_r] of spin n."""
        F = self.projectors(L)[abs(n)]
        if n < 0:
            F = torch.roll(F.flip(0), 1, 0)
        c = torch.fft.fft(f, dim=1)
        c = torch.complex(torch.matmul(F, c.real), torch.matmul(F, c.imag))
        return torch.fft.ifft(c, dim=1)

    def tensor(self, T, rank):
        """Yn filter of a Cartesian tensor [3, .., 3, J, N, n_r] (Sec. 3.4)."""
        st, ct = torch.sin(self.theta)[None], torch.cos(self.theta)[None]
        sp, cp = torch.sin(self.phi)[:, None], torch.cos(self.phi)[:, None]
        m = torch.complex(torch.stack([ct * cp, ct * sp, (-st).expand(self.J, -1)]),
                          torch.stack([-sp.expand(-1, self.N), cp.expand(-1, self.N), 0.0 * st * sp])) / math.sqrt(2.0)
        legs = torch.stack([self.n.to(m.dtype), m, m.conj()])[..., None]  # spins 0, 1, -1
        back = torch.stack([legs[0], legs[2], legs[1]])
        C = T.to(m.dtype)
        for q in range(rank):  # leg q to the triad
            C = torch.stack([sum(legs[A, a] * C.select(q, a) for a in range(3)) for A in range(3)], q)
        for tau in itertools.product(range(3), repeat=rank):
            C[tau] = self.project(C[tau][None], sum((0, 1, -1)[A] for A in tau), self.L)[0]
        for q in range(rank):
            C = torch.stack([sum(back[A, a] * C.select(q, A) for A in range(3)) for a in range(3)], q)
        return C.real

    def filter(self, u):
        out = u.clone()
        if self.kind != "yn":
            for s in range(self.nv):
                d = (0 if (s - 50) % 4 == 0 else 1) if s >= 50 else sum(q > 0 for q in PAIRS[s % 10]) + (s >= 20)
                L = min(self.L + d, self.N - 1) if self.kind == "yg" else self.L
                out[s] = self.project(u[s][None].to(torch.complex128), 0, L)[0].real
            return out
        sym = [[PAIRS.index((min(a, b), max(a, b))) for b in range(4)] for a in range(4)]
        i3 = range(3)
        spots = [(1, [20 + 10 * i for i in i3]), (2, [20 + 10 * i + sym[0][j + 1] for i in i3 for j in i3]),
                 (3, [20 + 10 * i + sym[j + 1][k + 1] for i in i3 for j in i3 for k in i3])]
        for b in (0, 10):
            spots += [(0, [b]), (1, [b + sym[0][i + 1] for i in i3]),
                      (2, [b + sym[i + 1][j + 1] for i in i3 for j in i3])]
        for b in range(50, self.nv, 4):
            spots += [(0, [b]), (1, [b + 1, b + 2, b + 3])]
        for rank, at in spots:
            T = u[at].reshape((3,) * rank + tuple(u.shape[1:]))
            out[at] = self.tensor(T, rank).reshape((len(at),) + tuple(u.shape[1:]))
        return out


def _all_rhs(ms, us):
    k = [m.rhs(u, outer=q == len(ms) - 1) for q, (m, u) in enumerate(zip(ms, us))]
    for q in range(len(ms) - 1):  # characteristic coupling on the common sphere
        a, b = k[q][..., -1], k[q + 1][..., 0]
        sl, su = ms[q].sphere_normal(us[q][..., -1])
        dot = lambda v: sum(su[i] * v[20 + 10 * i:30 + 10 * i] for i in range(3))  # noqa: E731
        sa, sb = dot(a), dot(b)
        w0, wp, wm = a[:10], a[10:20] - a[:10] + sa, b[10:20] - b[:10] - sb
        c = a.clone()
        c[10:20] = 0.5 * (wp + wm) + w0
        for i in range(3):
            c[20 + 10 * i:30 + 10 * i] = sl[i] * (0.5 * (wp - wm)) + b[20 + 10 * i:30 + 10 * i] - sl[i] * sb
        k[q][..., -1] = c
        k[q + 1][..., 0] = c
    return k


def _advance(case, ms, us):
    dt = case["courant"] * min(m.dx for m in ms)

    def stage(vs):
        k = _all_rhs(ms, vs)
        return [m.filter(x) for m, x in zip(ms, k)] if case["placement"] == "substep" else k

    for _ in range(case["steps"]):
        k1 = stage(us)
        acc = k1
        k = k1
        for w, c in ((2.0, 0.5), (2.0, 0.5), (1.0, 1.0)):
            k = stage([u + c * dt * x for u, x in zip(us, k)])
            acc = [p + w * x for p, x in zip(acc, k)]
        us = [u + dt / 6.0 * p for u, p in zip(us, acc)]
        if case["placement"] == "step":
            us = [m.filter(u) for m, u in zip(ms, us)]
    return us


def exact(case, seed):
    us = _states(case, seed)
    ms = [_Method(case, g) for g in _grids(case)]
    if case["kind"] == "derivs":
        return ms[0].derivs(us[0])
    if case["kind"] == "filter":
        return ms[0].filter(us[0])
    us = [m.start(u) for m, u in zip(ms, us)]
    if case["kind"] == "rhs":
        return ms[0].rhs(us[0])
    if case["kind"] == "batch":
        return [_advance(case, [m], [u])[0] for m, u in zip(ms, us)]
    us = _advance(case, ms, us)
    return us if case["kind"] == "nest" else us[0]
