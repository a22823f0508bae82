"""The fixed-point transforms of the FP64 nonlinear term: every compile-time length and run-time
ones, at the edges of their tiles and bands, against the oracle; exponents; NaN and Inf.

Tolerance 1e-13: the oracle's dense DFTs round at about eps sqrt(P) <= 1e-14 of the row's norm
for P <= 2304, and the fixed-point lines keep 62 bits of the sum of the moduli of a line,
which for n random modes is sqrt(n) of its RMS: n 2^-62 < 1e-15 for n <= 2304."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O
from paper_1311_2481_gb300 import inputs as I

pytestmark = pytest.mark.gpu
LZ = 2 * math.pi / 3.16


@pytest.fixture(scope="module")
def tc():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1311_2481_gb300 import build, tc as t
    build.build()
    return t


def both(tc, N_r, M, K, u=None, seed=3, rows=None, opt={}, **kw):
    cfg = dict(dict(N_r=N_r, M=M, K=K, m_p=1, eta=0.5, Re_i=100.0, Re_o=0.0, L_z=LZ, dt=1e-4), **kw)
    ops = O.Operators(O.Params(**cfg))
    if u is None:
        u = I.random_spectral((3,) + ops.prm.shape(), seed, hermitian_K=K)
        u[1, :, 0] = np.conj(u[0, :, 0, ::-1])   # the m = 0 line of a real field in (u_+, u_-)
    plan = tc.Plan(**cfg, no_adjoint=True, **opt)
    N = plan.nonlinear(torch.from_numpy(u).cuda()).cpu().numpy()
    ref = O.nonlinear(ops, u, rows)
    return (N if rows is None else N[:, rows]), ref, u, plan


def check(N, ref):
    for c in range(3):
        assert np.linalg.norm(N[c] - ref[c]) <= 1e-13 * np.linalg.norm(ref[c]), c


@pytest.mark.parametrize("M,P", [(1, 3), (1, 4), (2, 6), (3, 9), (5, 16), (8, 24), (12, 36), (16, 48), (24, 72), (32, 96),
                                 (48, 144), (64, 192), (96, 288), (128, 384), (192, 576), (256, 768), (384, 1152),
                                 (40, 81), (47, 96), (35, 128), (54, 162), (300, 1024)])
def test_theta_lengths(tc, M, P):
    """P_theta with compile-time and run-time plans, 3/2 grids and grids down to 2M + 1."""
    check(*both(tc, 10, M, 3, P_theta=P, P_z=12)[:2])


@pytest.mark.parametrize("K,P", [(1, 3), (2, 8), (4, 12), (8, 24), (12, 36), (16, 48), (24, 72), (32, 96), (48, 144), (64, 192),
                                 (96, 288), (128, 384), (192, 576), (256, 768), (384, 1152), (512, 1536), (768, 2304),
                                 (40, 81), (95, 192), (161, 324), (320, 972), (700, 2048), (700, 2187)])
def test_z_lengths(tc, K, P):
    check(*both(tc, 10, 2, K, P_theta=6, P_z=P)[:2])


@pytest.mark.parametrize("N_r,fd", [(9, 8), (10, 8), (15, 8), (16, 8), (17, 8), (27, 8), (12, 4), (7, 2)])
def test_radial_tiles(tc, N_r, fd):
    check(*both(tc, N_r, 3, 4, fd_order=fd, m_p=6)[:2])


@pytest.mark.parametrize("rows", [1, 3, 8, 11])
def test_slabs_do_not_change_a_bit(tc, rows):
    a = both(tc, 21, 6, 10, P_z=36)
    b = both(tc, 21, 6, 10, P_z=36, u=a[2], opt=dict(stage_rows=rows))
    assert np.array_equal(a[0], b[0])


@pytest.mark.parametrize("e", [-140, -40, 1, 60, 140])
def test_powers_of_two_scale_exactly(tc, e):
    """N is quadratic: u 2^e gives N 2^2e, bit for bit, as exponents are kept apart from the lines."""
    N, _, u, plan = both(tc, 12, 6, 8)
    got = plan.nonlinear(torch.from_numpy(u * 2.0 ** e).cuda()).cpu().numpy()
    assert np.array_equal(got, N * 2.0 ** (2 * e))


def test_rows_of_very_different_size(tc):
    """Rows scaled by up to 1e100 apart: each row's N has its own exponent."""
    _, _, u, _ = both(tc, 12, 4, 6)
    u = u * (10.0 ** np.array([0, 0, 0, 0, 0, 0, 0, -3, -6, 40, 100, -100.]))[None, :, None, None]
    N, ref, _, _ = both(tc, 12, 4, 6, u=u)
    for j in range(12):
        assert np.linalg.norm(N[:, j] - ref[:, j]) <= 1e-13 * np.linalg.norm(ref[:, j]), j


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_rows(tc, bad):
    """A NaN or Inf makes N of its row NaN throughout, and of the rows whose stencil reaches it;
    rows out of reach keep their values (through the FP64 stencil where they share a tile of 8
    rows with its window, bit for bit elsewhere)."""
    N, ref, u, plan = both(tc, 40, 4, 6)
    v = u.copy()
    v[1, 20, 2, 5] = bad
    got = plan.nonlinear(torch.from_numpy(v).cuda()).cpu().numpy()
    assert np.isnan(got[:, 20]).all()
    near = [*range(8, 16), *range(25, 32)]      # the stencils of rows 16 .. 24 reach row 20
    check(got[:, near], ref[:, near])
    for j in (*range(0, 8), *range(32, 40)):
        assert np.array_equal(got[:, j], N[:, j]), j


def test_zero_and_mean_flow_only(tc):
    N, ref, _, _ = both(tc, 12, 4, 6, u=np.zeros((3, 12, 5, 13), np.complex128))
    assert not N.any()
    ops = O.Operators(O.Params(N_r=12, M=4, K=6, m_p=1, eta=0.5, Re_i=100.0, Re_o=0.0, L_z=LZ, dt=1e-4))
    u = I.base_state(ops.r, 4, 6, 0.5, 100.0, 0.0)
    N, ref, _, _ = both(tc, 12, 4, 6, u=u)
    assert np.linalg.norm(N - ref) <= 1e-14 * np.linalg.norm(ref)


@pytest.mark.parametrize("N_r,M,P_t,K,P_z,rows", [(11, 12, 36, 27, 81, 0), (10, 5, 16, 40, 243, 0), (10, 2, 6, 320, 972, 0),
                                                  (10, 2, 6, 384, 1152, 4), (12, 40, 81, 4, 12, 5), (10, 4, 12, 2, 6, 0),
                                                  (10, 24, 72, 6, 18, 3), (10, 96, 288, 4, 12, 0)])
def test_adjoint_lengths(tc, N_r, M, P_t, K, P_z, rows):
    """The transposed transforms at lengths with one z per block, odd tiles, one line per block
    (P_z > 768) and run-time plans, against the oracle's adjoint step.  1e-11 as the other
    adjoint tests ask: the oracle's own solves round at that level."""
    cfg = dict(N_r=N_r, M=M, K=K, m_p=1, eta=0.5, Re_i=50.0, Re_o=0.0, L_z=LZ, dt=1e-3)
    ops = O.Operators(O.Params(**cfg, P_theta=P_t, P_z=P_z))
    u0 = I.initial_state(ops.r, M, K, 1, LZ, 0.5, 50.0, 0.0, kind="box", amp=1e-2)
    st = O.State(u0, u0, u0, None, True)
    y = [I.random_spectral((3,) + ops.prm.shape(), seed=s) for s in (1, 2, 3)]
    ref = O.adjoint_step(ops, st, *y)
    plan = tc.Plan(**cfg, P_theta=P_t, P_z=P_z, stage_rows=rows)
    fwd = tc.State(plan, torch.from_numpy(u0))
    fwd.started = True
    bar = tc.StateBar(*[torch.from_numpy(v).cuda() for v in y])
    plan.adjoint_step(fwd, bar)
    for got, want in zip((bar.u, bar.u_prev, bar.N_prev), ref):
        assert np.linalg.norm(got.cpu().numpy() - want) <= 1e-11 * np.linalg.norm(want)
