"""Every call on plans of 3 to 9 radial rows (fd_order 2 to 8): below 9 rows the padded stencils begin
before the first row, with weight 0."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O
from paper_1311_2481_gb300 import inputs as I

pytestmark = pytest.mark.gpu
LZ = 2 * math.pi / 3.16
ROWS = [(3, 2), (4, 2), (5, 2), (5, 4), (6, 4), (7, 6), (8, 2), (8, 6), (9, 8)]


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.fixture(scope="module")
def tc():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1311_2481_gb300 import build, tc as t
    build.build()
    return t


def case(N_r, fd):
    cfg = dict(N_r=N_r, M=3, K=4, m_p=1, eta=0.5, Re_i=50.0, Re_o=10.0, L_z=LZ, dt=1e-3, fd_order=fd)
    ops = O.Operators(O.Params(**cfg))
    u0 = I.initial_state(ops.r, 3, 4, 1, LZ, 0.5, 50.0, 10.0, kind="broadband", amp=1e-2, seed=3)
    return cfg, ops, u0


@pytest.mark.parametrize("split", [-1, 1])
@pytest.mark.parametrize("N_r,fd", ROWS)
def test_steps_solves_and_diagnostics(tc, N_r, fd, split):
    """The bounds of the same calls at more rows: 1e-10 for two steps, rounding for the rest."""
    cfg, ops, u0 = case(N_r, fd)
    plan = tc.Plan(**cfg, pc_split=split, no_adjoint=True)
    st = tc.State(plan, torch.from_numpy(u0).cuda())
    plan.step(st, 2)
    ref = O.run(ops, O.cold_state(u0), 2)
    for k in ("u", "p"):
        assert rel(getattr(st, k).cpu().numpy(), getattr(ref, k)) <= 1e-10, k
    d, u = plan.diagnostics(st.u), st.u.cpu().numpy()
    T = O.torque(ops, u)
    assert d.finite and abs(d.energy - O.perturbation_energy(ops, u)) <= 1e-12 * d.energy
    assert max(abs(d.torque_inner - T[0]), abs(d.torque_outer - T[1])) <= 1e-11 * max(map(abs, T))
    assert abs(d.max_div - O.max_divergence(ops, u)) <= 1e-10 * np.abs(u).max()
    b = I.random_spectral(ops.prm.shape(), 5)
    for which, name in ((tc.TC_P_STAR, "P"), (tc.TC_U_PLUS, "Hp"), (tc.TC_U_MINUS, "Hm"), (tc.TC_U_Z, "Hz")):
        x = plan.helmholtz_solve(which, torch.from_numpy(b).cuda()).cpu().numpy()
        assert rel(x, O.solve_modes(ops, ops.mats[name], b)) <= 1e-12, name


@pytest.mark.parametrize("N_r,fd", ROWS)
def test_mixed_steps(tc, N_r, fd):
    """FP32 transforms of the perturbation: 1e-6 of N, of which a step takes dt."""
    cfg, ops, u0 = case(N_r, fd)
    plan = tc.Plan(**cfg, precision=tc.TC_MIXED, no_adjoint=True)
    st = tc.State(plan, torch.from_numpy(u0).cuda())
    plan.step(st, 2)
    assert rel(st.u.cpu().numpy(), O.run(ops, O.cold_state(u0), 2).u) <= 1e-8


@pytest.mark.parametrize("split", [-1, 1])
@pytest.mark.parametrize("N_r,fd", ROWS)
def test_adjoint_step(tc, N_r, fd, split):
    cfg, ops, u0 = case(N_r, fd)
    st_o = O.step(ops, O.cold_state(u0))
    y = [I.random_spectral((3,) + ops.prm.shape(), seed=s) for s in (21, 22, 23)]
    ref = O.adjoint_step(ops, st_o, *y)
    plan = tc.Plan(**cfg, pc_split=split)
    st = tc.State(plan, torch.from_numpy(st_o.u).cuda())
    st.started = True
    bar = tc.StateBar(*[torch.from_numpy(v).cuda() for v in y])
    plan.adjoint_step(st, bar)
    for got, want in zip((bar.u, bar.u_prev, bar.N_prev), ref):
        assert rel(got.cpu().numpy(), want) <= 1e-11


@pytest.mark.parametrize("mixed", [False, True])
def test_nan_before_the_field_stays_there(tc, mixed):
    """u, u_prev and N_prev inside larger buffers of NaN."""
    cfg, ops, u0 = case(5, 4)
    plan = tc.Plan(**cfg, no_adjoint=True, precision=tc.TC_MIXED if mixed else tc.TC_FP64)
    st = tc.State(plan, torch.from_numpy(u0).cuda())
    plan.step(st, 1)
    n = 8 * ops.prm.shape()[1] * ops.prm.shape()[2]
    inside = tc.State(plan, st.u)
    for k in ("u", "u_prev", "N_prev", "p"):
        v = getattr(st, k)
        buf = torch.full((v.numel() + 2 * n,), float("nan"), dtype=v.dtype, device=v.device)
        w = buf[n:n + v.numel()].view(v.shape)
        w.copy_(v)
        setattr(inside, k, w)
    inside.started = True
    plan.step(inside, 2)
    plan.step(st, 2)
    for k in ("u", "u_prev", "N_prev", "p"):
        assert torch.equal(getattr(inside, k), getattr(st, k)), k
    assert plan.diagnostics(inside.u).finite
