"""The mean mode and the m = 0 lines of the FP64 nonlinear term: the symmetry of real fields holds exactly,
and the azimuthal mean, which drives the mean flow and is far smaller than N_r beside it, is as
accurate as its own terms allow."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1311_2481_gb300 import inputs as I

pytestmark = pytest.mark.gpu
LZ = 2 * math.pi / 3.16


def case(N_r, M, K, amp, **kw):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1311_2481_gb300 import build, tc
    build.build()
    plan = tc.Plan(N_r, M, K, 1, 0.5, 1000.0, 0.0, LZ, 1e-6, no_adjoint=True, **kw)
    u = I.initial_state(plan.nodes(), M, K, 1, LZ, 0.5, 1000.0, 0.0, kind="broadband", amp=amp, seed=5)
    return tc, plan, u


@pytest.mark.parametrize("N_r,M,K,kw", [(12, 4, 8, {}), (33, 8, 16, {}), (20, 25, 50, dict(P_theta=81, P_z=162)),
                                        (16, 2, 320, dict(P_z=972)), (24, 32, 64, dict(stage_rows=7)), (10, 1, 1, {})])
def test_m0_lines_are_those_of_real_fields(N_r, M, K, kw):
    tc, plan, u = case(N_r, M, K, 1e-2, **kw)
    N = plan.nonlinear(torch.from_numpy(u).cuda()).cpu().numpy()
    assert np.array_equal(N[1, :, 0], np.conj(N[0, :, 0, ::-1]))
    assert np.array_equal(N[2, :, 0], np.conj(N[2, :, 0, ::-1]))
    # so u_+ + u_- of the mean mode, and with it the imaginary part of p, stays exactly 0
    st = tc.State(plan, torch.from_numpy(u).cuda())
    plan.step(st, 3)
    assert not st.p[:, 0, K].imag.any()
    assert torch.equal(st.u[0, :, 0, K], st.u[1, :, 0, K].conj())


@pytest.mark.parametrize("amp", [1e-2, 1e-4])
@pytest.mark.parametrize("N_r,M,K,kw", [(12, 4, 8, {}), (33, 8, 16, {}), (20, 25, 50, dict(P_theta=81, P_z=162)),
                                        (16, 2, 320, dict(P_z=972)), (48, 32, 64, dict(stage_rows=7))])
def test_azimuthal_mean(N_r, M, K, kw, amp):
    """Against the Parseval sum in extended precision, <N_t> = <u_r D u_t> + <u_r u_t> / r + <u_z d_z u_t>.  The
    lines hold u_r beside U, at 2^-61 of the sum of their moduli, S = 4 U here: a few units of that,
    random in z, times the mean flow's gradient (D U + U / r), and the products' own rounding, far
    smaller.  8 2^-61 S |D U + U / r|, and the FP64 rounding of the sum's terms."""
    tc, plan, u = case(N_r, M, K, amp, **kw)
    got = plan.nonlinear(torch.from_numpy(u).cuda()).cpu().numpy()[0, :, 0, K].imag
    L = np.longdouble
    r = plan.nodes().astype(L)
    w, c0 = plan.fd_weights(1)
    v = u.astype(np.clongdouble)
    ur, ut, uz = (v[0] + v[1]) / 2, (v[0] - v[1]) / L(2) * np.clongdouble(-1j), v[2]
    d = np.stack([sum(L(w[j, t]) * ut[c0[j] + t] for t in range(9)) for j in range(N_r)])
    kz = (2 * L(math.pi) / L(LZ)) * np.arange(-K, K + 1).astype(L)
    cm = np.where(np.arange(M + 1) == 0, 1, 2).astype(L)[None, :, None]
    # the m = 0 line counts through its real part: it is one already
    terms = cm * (ur * np.conj(d + ut / r[:, None, None]) + uz * np.conj(1j * kz * ut)).real
    want = terms.sum((1, 2))
    U = np.abs(ut[:, 0, K].real)
    bound = 8 * 2.0 ** -61 * 4 * U * np.abs((d[:, 0, K] + ut[:, 0, K] / r).real) + 2.0 ** -50 * np.abs(terms).sum((1, 2))
    err = np.abs(got - want)
    assert (err <= bound)[1:-1].all(), (err / bound).max()


@pytest.mark.parametrize("N_r,M,K,kw", [(12, 4, 8, {}), (33, 8, 16, {}), (20, 25, 50, dict(P_theta=81, P_z=162)),
                                        (10, 2, 384, dict(P_z=1152)), (24, 32, 64, dict(stage_rows=7))])
def test_adjoint_keeps_m0_lines_of_real_fields(N_r, M, K, kw):
    """Of adjoint fields whose m = 0 lines are those of real fields: + and - stay mirrored conjugates (the
    transforms' part exactly, the solves' as x and its conjugate take the same operations), and with
    them D1^T (g_+ + g_-) of the mean mode has no imaginary part for P^{-T} to magnify."""
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1311_2481_gb300 import build, tc
    build.build()
    plan = tc.Plan(N_r, M, K, 1, 0.5, 1000.0, 0.0, LZ, 1e-6, **kw)
    u = I.initial_state(plan.nodes(), M, K, 1, LZ, 0.5, 1000.0, 0.0, kind="broadband", amp=1e-2, seed=5)
    st = tc.State(plan, torch.from_numpy(u).cuda())
    st.started = True
    y = []
    for s in (1, 2, 3):
        v = I.random_spectral((3,) + u.shape[1:], seed=s, hermitian_K=K)
        v[1, :, 0] = np.conj(v[0, :, 0, ::-1])
        v[:2, :, 0, K] = 1j * v[:1, :, 0, K].imag * np.array([1, -1])[:, None]   # the mean mode has no radial part
        y.append(torch.from_numpy(v).cuda())
    bar = tc.StateBar(*y)
    for _ in range(2):
        plan.adjoint_step(st, bar)
        for f in (bar.u, bar.u_prev, bar.N_prev):
            assert torch.equal(f[1, :, 0], f[0, :, 0].flip(-1).conj())
