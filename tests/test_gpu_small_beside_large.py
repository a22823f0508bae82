"""d_theta lines far below the mean flow: the exponent of a theta line weighted by m m_p comes from its
m > 0 entries alone."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu
LZ = 2 * math.pi / 3.16


@pytest.mark.parametrize("e", [-30, -96, -97, -100, -110])
def test_d_theta_far_below_the_mean(e):
    """u = (0, U, 1 + 2^e (w e^{i theta} + cc)): N_z at (1, 0) is i U w 2^e / r and nothing else.  N_z is
    held to 2^-62 of the largest exponent among its terms, here at least that of u_r d_r u_z:
    u_r = 0 counts as up to 2^-30 U, d_r of the constant as the stencil's rounding, up to 2^-40
    at 12 rows.  So 2^(-30 - 40 - 62 + 4) U beside 2^(e - 1) U: 1e-5 at e = -110."""
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1311_2481_gb300 import build, tc
    build.build()
    N, M, K = 12, 4, 6
    plan = tc.Plan(N, M, K, 1, 0.5, 50.0, 0.0, LZ, 1e-3, no_adjoint=True)
    r = plan.nodes()
    rng = np.random.default_rng(7)
    w = np.exp(2j * math.pi * rng.random(N))
    u = np.zeros((3, N, M + 1, 2 * K + 1), np.complex128)
    u[0, :, 0, K], u[1, :, 0, K] = 1j * 3.0, -1j * 3.0
    u[2, :, 0, K] = 1.0
    u[2, :, 1, K] = w * 2.0 ** e
    got = plan.nonlinear(torch.from_numpy(u).cuda()).cpu().numpy()[2, :, 1, K]
    want = 1j * 3.0 * w * 2.0 ** e / r
    assert np.abs(got - want).max() <= 1e-5 * np.abs(want).max()
