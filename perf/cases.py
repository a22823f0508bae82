"""The work that is measured: time steps, nonlinear terms, banded solves and adjoint steps of
the Taylor-Couette solver through its Python entry points (paper_1311_2481_gb300.tc.Plan and
adjoint.final_energy), over the sizes that its configurations, tests and benchmark use.

A case names its call ("op"), the resolution (N_r radial nodes, modes m = 0..M and k = -K..K
on a P_theta x P_z grid; 0: the default 3M or 3K), the flow and the precision form.  `exact`
restates the method in plain torch in 64 bits (FFTs, dense solves, autograd for the adjoint).
"""
import math

import numpy as np
import torch

from paper_1311_2481_gb300 import adjoint, tc

DEV = "cuda"
L_Z = 2 * math.pi / 3.16
SYSTEMS = {"p": tc.TC_P_STAR, "u+": tc.TC_U_PLUS, "u-": tc.TC_U_MINUS, "uz": tc.TC_U_Z, "phi": tc.TC_PHI}


def _case(name, op, N_r, M, K, mixed=False, m_p=1, P_theta=0, P_z=0, Re_i=1000.0, Re_o=0.0, **more):
    return dict(name=name, op=op, N_r=N_r, M=M, K=K, mixed=mixed, m_p=m_p, P_theta=P_theta, P_z=P_z,
                Re_i=Re_i, Re_o=Re_o, **more)


def listed():
    qk = math.sqrt(0.5)   # quasi-Keplerian: Omega_o / Omega_i = eta^1.5, so Re_o = sqrt(eta) Re_i
    return [
        # the nonlinear term alone at the size of a first smoke run: one call's latency
        _case("nonlinear tiny", "nonlinear", 16, 4, 8, Re_i=50.0),
        # a step of the small validation runs (hundreds of thousands of steps, launch-bound)
        _case("step small", "step", 32, 8, 16, Re_i=50.0),
        # the throughput workload: production runs at moderate Reynolds number, both forms
        _case("step", "step", 64, 32, 64),
        _case("step mixed", "step", 64, 32, 64, mixed=True),
        # the same from host memory, as a program that keeps its state outside the device calls it
        _case("step from host", "step_host", 64, 32, 64),
        # a grid with no power-of-two structure and a rotational symmetry, as users of m_p > 1 set it
        _case("nonlinear ragged", "nonlinear", 45, 25, 50, m_p=6, P_theta=81, P_z=162),
        # the paper's own timing grid (P_z is not three times a power of two)
        _case("nonlinear 32x576x972", "nonlinear", 32, 192, 320, P_z=972),
        # high radial resolution: the per-stage banded solves, both forms
        _case("step tall", "step", 256, 64, 128, Re_i=1e4, Re_o=1e4 * qk),
        _case("step tall mixed", "step", 256, 64, 128, mixed=True, Re_i=1e4, Re_o=1e4 * qk),
        # one banded system for every mode
        _case("solve", "solve", 128, 32, 64, system="u+"),
        # backward: one adjoint step of the optimal-perturbation workload
        _case("adjoint step", "adjoint", 96, 32, 64, Re_i=2000.0),
        # forward and backward of a short checkpointed run, through autograd
        _case("gradient of a run", "gradient", 32, 8, 16, Re_i=50.0, steps=8, checkpoint=4),
    ]


def _grid(n):
    """Smallest 2^a 3^b >= 3 n."""
    best = None
    for a in range(14):
        for b in range(9):
            v = 2 ** a * 3 ** b
            if v >= 3 * n and (best is None or v < best):
                best = v
    return best


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the same ranges: any node count, mode counts and grids 2^a 3^b of at least 3/2."""
    op, mixed = rng.choice([("nonlinear", False), ("step", False), ("step", False), ("step", True),
                            ("adjoint", False), ("solve", False)])
    while True:
        N_r, M, K = _log_int(rng, 12, 256), _log_int(rng, 2, 192), _log_int(rng, 4, 320)
        cost = N_r * M * K * {"nonlinear": 1, "step": 1, "adjoint": 2.5, "solve": 0.5}[op]
        if cost <= 1.9e6:
            break
    c = _case("", op, N_r, M, K, mixed=mixed, m_p=rng.choice([1, 1, 1, 6]), P_theta=_grid(M), P_z=_grid(K),
              Re_i=float(_log_int(rng, 50, 2000) if M >= 12 else 50))
    if op == "solve":
        c["system"] = rng.choice(sorted(SYSTEMS))
    del c["name"]
    return c


# ------------------------------------------------------------------------------ inputs

def _dt(c):
    """A quarter of the advective limit of the fastest wall, and less: runs stay bounded."""
    return 0.1 / (max(abs(c["Re_i"]), 0.5 * abs(c["Re_o"])) * c["M"] * c["m_p"])


def _nodes(n):
    """Clustered radial nodes between r = 1 and 2 (gap 1, eta = 0.5, clustering 0.5)."""
    j = np.arange(n, dtype=np.longdouble)
    x = -np.cos(np.longdouble(math.pi) * 0 + np.arccos(np.longdouble(-1)) * j / (n - 1))
    return np.longdouble(1.5) + np.arcsin(np.longdouble(0.5) * x) / (2 * np.arcsin(np.longdouble(0.5)))


def _field(c, g, amp, base=True):
    """Couette flow plus a divergence-free perturbation curl(g(r) a) with a Gaussian spectrum of
    random phases, of RMS amp * Re_i: (u_+, u_-, u_z) coefficients [3][N_r][M+1][2K+1]."""
    N, M, K = c["N_r"], c["M"], c["K"]
    r = torch.from_numpy(_nodes(N).astype(np.float64)).to(DEV)[:, None, None]
    m = torch.arange(M + 1, device=DEV, dtype=torch.float64)[:, None]
    k = torch.arange(-K, K + 1, device=DEV, dtype=torch.float64)[None, :]
    a = torch.complex(*torch.randn((2, 3, M + 1, 2 * K + 1), generator=g, device=DEV, dtype=torch.float64))
    a = a * torch.exp(-(m / max(M / 4, 0.5)) ** 2 - (k / max(K / 4, 0.5)) ** 2)
    a[:, 0] = 0.5 * (a[:, 0] + a[:, 0].flip(-1).conj())   # the m = 0 line of real fields
    a[:, 0, K] = 0
    im, ik = 1j * c["m_p"] * m, 1j * (2 * math.pi / L_Z) * k
    w = (r - 1) ** 2 * (2 - r) ** 2
    dw = 2 * (r - 1) * (2 - r) ** 2 - 2 * (r - 1) ** 2 * (2 - r)
    ur = im * a[2] * w / r - ik * a[1] * w
    ut = ik * a[0] * w - a[2] * dw
    u = torch.stack([ur + 1j * ut, ur - 1j * ut, a[1] * (w / r + dw) - im * a[0] * w / r])
    e = 0.5 * (u[0].abs() ** 2 + u[1].abs() ** 2) + u[2].abs() ** 2
    e[:, 1:] *= 2
    u *= amp * c["Re_i"] / torch.sqrt(e.sum() / N)
    if base:
        eta, Re_i, Re_o = 0.5, c["Re_i"], c["Re_o"]
        C1, C2 = (Re_o - eta * Re_i) / (1 + eta), eta * (Re_i - eta * Re_o) / ((1 - eta) * (1 - eta * eta))
        U = C1 * r[:, 0, 0] + C2 / r[:, 0, 0]
        u[0, :, 0, K] = 1j * U
        u[1, :, 0, K] = -1j * U
    return u


def _inputs(c, seed):
    """(u, extra): the velocity, and the right-hand side or the adjoint fields where the call takes them."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    u = _field(c, g, 0.01)
    if c["op"] == "solve":
        x = _field(c, g, 0.01, base=False)[0 if c["system"] == "u+" else 1].contiguous()
        return u, x * (1.5 / _dt(c))
    if c["op"] == "adjoint":
        return u, [_field(c, g, 0.01, base=False) for _ in range(3)]
    return u, None


def prepare(c, seed):
    u, extra = _inputs(c, seed)
    plan = tc.Plan(c["N_r"], c["M"], c["K"], c["m_p"], 0.5, c["Re_i"], c["Re_o"], L_Z, _dt(c),
                   P_theta=c["P_theta"], P_z=c["P_z"], precision=tc.TC_MIXED if c["mixed"] else tc.TC_FP64,
                   no_adjoint=c["op"] not in ("adjoint", "gradient"))
    s = {"op": c["op"], "plan": plan, "u": u, "case": c}
    if c["op"] in ("step", "step_host"):
        s["st"] = plan.step(tc.State(plan, u), 0)   # with the history that a run has
        if c["op"] == "step_host":
            st = s["st"]
            s["host"] = {k: t.cpu().pin_memory() for k, t in
                         (("u", st.u), ("u_prev", st.u_prev), ("N_prev", st.N_prev), ("p", st.p))}
            s["host"]["started"] = True
            s["out"] = {k: torch.empty_like(s["host"][k], pin_memory=True) for k in ("u", "p")}
    elif c["op"] == "solve":
        s["rhs"] = extra
    elif c["op"] == "adjoint":
        s["bar"] = tc.StateBar(*extra)
        s["fwd"] = plan.step(tc.State(plan, u), 0)
    return s


def run(s):
    op, plan = s["op"], s["plan"]
    if op == "nonlinear":
        return plan.nonlinear(s["u"])
    if op == "step":
        st = plan.step(s["st"], 1)
        return {"u": st.u, "u_prev": st.u_prev, "N_prev": st.N_prev, "p": st.p}
    if op == "step_host":
        plan.step_host(s["st"], s["host"], s["out"], 1)
        return s["out"]
    if op == "solve":
        return plan.helmholtz_solve(SYSTEMS[s["case"]["system"]], s["rhs"])
    if op == "adjoint":
        b = plan.adjoint_step(s["fwd"], s["bar"])
        return {"u": b.u, "u_prev": b.u_prev, "N_prev": b.N_prev}
    x = s["u"].detach().requires_grad_(True)
    J = adjoint.final_energy(x, plan, s["case"]["steps"], s["case"]["checkpoint"])
    J.backward()
    g, x.grad = x.grad, None
    return {"J": J.detach(), "grad": g}


# ------------------------------------------------------------------------------ least work

def _grids(c):
    return c["P_theta"] or 3 * c["M"], c["P_z"] or 3 * c["K"]


def _nonlinear_flops(c, z_lines, t_lines, per_point):
    Pt, Pz = _grids(c)
    N, M1, S = c["N_r"], c["M"] + 1, c["N_r"] * (c["M"] + 1) * (2 * c["K"] + 1)
    return (z_lines * N * M1 * 5 * Pz * math.log2(Pz) + t_lines * N * Pz * 5 * Pt * math.log2(Pt)
            + per_point * N * Pt * Pz + 3 * 36 * S)


def work(c):
    N, M, K, op = c["N_r"], c["M"], c["K"], c["op"]
    S = N * (M + 1) * (2 * K + 1)                 # complex values of a scalar field
    fac = 8 * 13 * N * (M + 1) * (K + 1)          # one set of banded LU factors with fill
    nl = _nonlinear_flops(c, 12, 7.5, 25)
    lin = S * (5 * 52 + 4 * 36 + 60)              # five substitutions, four stencils, the rest
    if op == "nonlinear":
        return {"bytes": 6 * 16 * S, "flops": nl}
    if op == "solve":
        return {"bytes": 2 * 16 * S + fac, "flops": 52 * S}
    if op == "step":                              # u, u_prev, N_prev in; these and p out
        return {"bytes": 19 * 16 * S + 4 * fac, "flops": nl + lin}
    if op == "step_host":
        return {"bytes": 13 * 16 * S + 4 * fac, "flops": nl + lin}
    adj = _nonlinear_flops(c, 21, 13.5, 60) + lin
    if op == "adjoint":                           # u and three adjoint fields in, three out
        return {"bytes": 21 * 16 * S + 4 * fac, "flops": adj}
    n = c["steps"]
    return {"bytes": n * (40 * 16 * S + 8 * fac), "flops": n * (2 * (nl + lin) + adj)}


# ------------------------------------------------------------------------------ exact values

def _weights(x0, xs, deriv):
    """FD weights of the derivative at x0 on the nodes xs (moment conditions, longdouble)."""
    n = len(xs)
    h = max(abs(x - x0) for x in xs)
    A = [[((x - x0) / h) ** q for x in xs] for q in range(n)]
    b = [np.longdouble(math.factorial(deriv)) if q == deriv else np.longdouble(0) for q in range(n)]
    for i in range(n):
        p = max(range(i, n), key=lambda t: abs(A[t][i]))
        A[i], A[p], b[i], b[p] = A[p], A[i], b[p], b[i]
        for t in range(i + 1, n):
            f = A[t][i] / A[i][i]
            A[t] = [x - f * y for x, y in zip(A[t], A[i])]
            b[t] -= f * b[i]
    w = [np.longdouble(0)] * n
    for i in reversed(range(n)):
        w[i] = (b[i] - sum(A[i][j] * w[j] for j in range(i + 1, n))) / A[i][i]
    return [float(x / h ** deriv) for x in w]


class _Method:
    """The discretisation in plain torch: FFTs on the padded grid, dense radial matrices."""

    def __init__(self, c, solves):
        self.c, N = c, c["N_r"]
        self.M, self.K, (self.Pt, self.Pz) = c["M"], c["K"], _grids(c)
        x = _nodes(N)
        D = np.zeros((2, N, N))
        for j in range(N):
            h = min(j, N - 1 - j, 4)
            idx = range(5) if j == 0 else range(N - 5, N) if j == N - 1 else range(j - h, j + h + 1)
            for d in (1, 2):
                D[d - 1, j, list(idx)] = _weights(x[j], [x[i] for i in idx], d)
        as_t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(DEV)
        self.D1, self.D2 = as_t(D[0]), as_t(D[1])
        self.r = as_t(x.astype(np.float64))
        self.ir = (1 / self.r)[:, None, None]
        self.mm = c["m_p"] * torch.arange(self.M + 1, device=DEV, dtype=torch.float64)[:, None]
        self.kk = 2 * math.pi / L_Z * torch.arange(-self.K, self.K + 1, device=DEV, dtype=torch.float64)
        self.A = {n: self.matrix(n) for n in solves}

    def matrix(self, n):
        N, c, ir = self.c["N_r"], self.c, 1 / self.r
        eye = torch.eye(N, device=DEV, dtype=torch.float64)
        mm, ka = self.mm[:, :, None, None], self.kk[self.K:][None, :, None, None]
        L = (self.D2 + ir[:, None] * self.D1) - mm ** 2 * torch.diag(ir ** 2) - ka ** 2 * eye
        if n == "p":
            L[:, :, 0], L[:, :, -1] = self.D1[0], self.D1[-1]
            L[0, 0, -1] = eye[-1]
            return L
        s = {"u+": 1.0, "u-": -1.0, "uz": 0.0}[n]
        A = 1.5 / _dt(c) * eye - L + abs(s) * torch.diag(ir ** 2) + s * 2 * mm * torch.diag(ir ** 2)
        A[:, :, 0], A[:, :, -1] = eye[0], eye[-1]
        return A

    def solve(self, n, b):
        K = self.K
        bp, bm = b[..., K:], b[..., :K + 1].flip(-1)              # k = |k| and -|k|: one matrix
        B = torch.stack([bp.real, bp.imag, bm.real, bm.imag], -1).permute(1, 2, 0, 3)
        x = torch.linalg.solve(self.A[n], B).permute(2, 0, 1, 3)
        return torch.cat([torch.complex(x[..., 2], x[..., 3])[..., 1:].flip(-1), torch.complex(x[..., 0], x[..., 1])], -1)

    def d(self, D, a):
        return torch.tensordot(D.to(a.dtype), a, dims=([1], [0]))

    def phys(self, a):
        z = a.new_zeros(a.shape[:-1] + (self.Pz,))
        z[..., :self.K + 1] = a[..., self.K:]
        z[..., self.Pz - self.K:] = a[..., :self.K]
        t = a.new_zeros(a.shape[:-2] + (self.Pt, self.Pz))
        z = torch.fft.ifft(z, dim=-1) * self.Pz
        t[..., 0, :] = z[..., 0, :]
        t[..., 1:self.M + 1, :] = 2 * z[..., 1:, :]
        return torch.fft.ifft(t, dim=-2).real * self.Pt

    def spec(self, f):
        t = torch.fft.fft(f, dim=-2)[..., :self.M + 1, :] / self.Pt
        z = torch.fft.fft(t, dim=-1) / self.Pz
        return torch.cat([z[..., self.Pz - self.K:], z[..., :self.K + 1]], -1)

    def nonlinear(self, u):
        comps = [(u[0] + u[1]) / 2, (u[0] - u[1]) / 2j, u[2]]
        v = [self.phys(a) for a in comps]
        r = self.ir
        adv = [v[0] * self.phys(self.d(self.D1, a)) + v[1] * r * self.phys(1j * self.mm * a)
               + v[2] * self.phys(1j * self.kk * a) for a in comps]
        n = [self.spec(f) for f in (adv[0] - v[1] * v[1] * r, adv[1] + v[1] * v[0] * r, adv[2])]
        return torch.stack([n[0] + 1j * n[1], n[0] - 1j * n[1], n[2]])

    def div(self, v):
        vr = (v[0] + v[1]) / 2
        return self.d(self.D1, vr) + vr * self.ir + self.mm * (v[0] - v[1]) * self.ir / 2 + 1j * self.kk * v[2]

    def grad(self, f):
        d, t = self.d(self.D1, f), self.mm * f * self.ir
        return torch.stack([d - t, d + t, 1j * self.kk * f])

    def lap_r(self, u):
        def lap(a, s):
            return (self.d(self.D2, a) + self.d(self.D1, a) * self.ir
                    - ((self.mm ** 2 + 1 + 2 * s * self.mm) * self.ir ** 2 + self.kk ** 2) * a)
        return (lap(u[0], 1) + lap(u[1], -1)) / 2

    def advance(self, u, up, n, n0, bc=1.0):
        K, w = self.K, 2 * n - n0
        g = -(w[0] + w[1]) / 2 + 2 * self.lap_r(u) - self.lap_r(up)
        b = torch.cat([g[:1], -self.div(w)[1:-1], g[-1:]])
        keep = torch.ones_like(b.real)
        keep[-1, 0, K] = 0
        p = self.solve("p", b * keep)
        rhs = (4 * u - up) / (2 * _dt(self.c)) - w - self.grad(p)
        wall = torch.zeros_like(rhs)
        for j, Re in ((0, self.c["Re_i"]), (-1, self.c["Re_o"])):
            wall[0, j, 0, K], wall[1, j, 0, K] = 1j * Re * bc, -1j * Re * bc
        rhs = torch.cat([wall[:, :1], rhs[:, 1:-1], wall[:, -1:]], 1)
        us = torch.stack([self.solve(s, rhs[i]) for i, s in enumerate(("u+", "u-", "uz"))])
        b = self.div(us)
        f = self.solve("p", torch.cat([0 * b[:1], b[1:-1], 0 * b[-1:]]))
        return us - self.grad(f), p + 1.5 / _dt(self.c) * f

    def start(self, u):
        n = self.nonlinear(u)
        up = 2.5 * u - 1.5 * self.advance(u, u, n, n)[0]
        return up, self.nonlinear(up)

    def energy(self, u):
        K, r, N = self.K, self.r, self.c["N_r"]
        eta, Re_i, Re_o = 0.5, self.c["Re_i"], self.c["Re_o"]
        C1, C2 = (Re_o - eta * Re_i) / (1 + eta), eta * (Re_i - eta * Re_o) / ((1 - eta) * (1 - eta * eta))
        U = torch.zeros_like(u)
        U[0, :, 0, K], U[1, :, 0, K] = 1j * (C1 * r + C2 / r), -1j * (C1 * r + C2 / r)
        e = u - U
        e = 0.5 * (e[0].abs() ** 2 + e[1].abs() ** 2) + e[2].abs() ** 2
        w = torch.zeros_like(r)
        w[:-1] += (r[1:] - r[:-1]) / 2
        w[1:] += (r[1:] - r[:-1]) / 2
        cm = torch.full_like(self.mm, 2.0)
        cm[0] = 1
        return 0.5 * (w * r * (cm * e).sum((1, 2))).sum()


def exact(c, seed):
    op = c["op"]
    u, extra = _inputs(c, seed)
    if op == "nonlinear":
        return _Method(c, ()).nonlinear(u)
    if op == "solve":
        n = {"phi": "p"}.get(c["system"], c["system"])
        return _Method(c, (n,)).solve(n, extra)
    if c["N_r"] ** 2 * (c["M"] + 1) * (c["K"] + 1) > 6e8:
        return None                            # the dense matrices of every mode
    x = _Method(c, ("p", "u+", "u-", "uz"))
    if op in ("step", "step_host"):
        up, n0 = x.start(u)
        n = x.nonlinear(u)
        un, p = x.advance(u, up, n, n0)
        return {"u": un, "p": p} if op == "step_host" else {"u": un, "u_prev": u, "N_prev": n, "p": p}
    if op == "adjoint":
        v = u.clone().requires_grad_(True)
        up, n0 = (torch.zeros_like(u).requires_grad_(True) for _ in range(2))
        n = x.nonlinear(v)
        un, _ = x.advance(v, up, n, n0, bc=0.0)
        loss = sum((torch.view_as_real(b) * torch.view_as_real(o)).sum() for b, o in zip(extra, (un, v, n)))
        g = torch.autograd.grad(loss, (v, up, n0))
        return {"u": g[0], "u_prev": g[1], "N_prev": g[2]}
    v = u.clone().requires_grad_(True)
    up, n0 = x.start(v)
    a = v
    for _ in range(c["steps"]):
        n = x.nonlinear(a)
        a, up, n0 = x.advance(a, up, n, n0)[0], a, n
    J = x.energy(a)
    return {"J": J.detach(), "grad": torch.autograd.grad(J, v)[0]}
