"""tc_helmholtz_solve on plans that force the fused steps 2-5 at many rows: the columns of 16 modes
exceed a block's shared memory from about 900 rows on."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1311_2481_gb300 import inputs as I

pytestmark = pytest.mark.gpu
LZ = 2 * math.pi / 3.16


@pytest.mark.parametrize("N_r", [193, 384, 385, 896, 897, 1000, 1537, 2048])
def test_solve_at_many_rows(N_r):
    """Against the host substitution with the same plan's factors: two forms of a backward-stable
    elimination, which for these Helmholtz matrices (3 / (2 dt) on the diagonal, condition below
    1e9) agree to 1e-16 times their condition and more."""
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1311_2481_gb300 import build, tc
    build.build()
    cfg = dict(N_r=N_r, M=1, K=2, m_p=1, eta=0.5, Re_i=50.0, Re_o=0.0, L_z=LZ, dt=1e-4, pc_split=-1)
    plan, host = tc.Plan(**cfg, no_adjoint=True), tc.Plan(**cfg, host_only=True)
    b = I.random_spectral((N_r, 2, 5), 5)
    rhs = torch.from_numpy(b).cuda()
    x = plan.helmholtz_solve(tc.TC_U_Z, rhs)
    assert torch.equal(x, plan.helmholtz_solve(tc.TC_U_Z, rhs, rhs))
    x = x.cpu().numpy()
    for m in range(2):
        for k in range(-2, 3):
            ref = sum(f * host.solve_host(tc.TC_U_Z, m, abs(k), np.ascontiguousarray(p), 1)
                      for f, p in ((1, b[:, m, k + 2].real), (1j, b[:, m, k + 2].imag)))
            assert np.linalg.norm(x[:, m, k + 2] - ref) <= 1e-7 * np.linalg.norm(ref)
