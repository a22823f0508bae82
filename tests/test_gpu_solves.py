"""tc_helmholtz_solve in two partitions (N_r >= 16 on plans of the fused steps-2-5 kernel) and in
one, at the edges of both, ragged blocks of modes included, against the oracle's elimination."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O
from paper_1311_2481_gb300 import inputs as I

pytestmark = pytest.mark.gpu
LZ = 2 * math.pi / 3.16


@pytest.mark.parametrize("N_r,M,K", [(15, 4, 6), (16, 1, 1), (17, 3, 8), (33, 2, 4), (64, 4, 9), (192, 2, 3), (193, 2, 3)])
def test_solves_match_oracle(N_r, M, K):
    """Error bound: both sides are backward-stable eliminations, which differ by up to a small
    multiple of eps cond(A) (the Poisson matrices grow as N_r^2 with the clustering)."""
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1311_2481_gb300 import build, tc
    build.build()
    cfg = dict(N_r=N_r, M=M, K=K, m_p=1, eta=0.5, Re_i=50.0, Re_o=0.0, L_z=LZ, dt=1e-3)
    ops = O.Operators(O.Params(**cfg))
    plan = tc.Plan(**cfg, no_adjoint=True)
    b = I.random_spectral(ops.prm.shape(), 5)
    for which, name in ((tc.TC_P_STAR, "P"), (tc.TC_U_PLUS, "Hp"), (tc.TC_U_MINUS, "Hm"), (tc.TC_U_Z, "Hz"), (tc.TC_PHI, "P")):
        ref = O.solve_modes(ops, ops.mats[name], b)
        rhs = torch.from_numpy(b).cuda()
        x = plan.helmholtz_solve(which, rhs)
        inplace = plan.helmholtz_solve(which, rhs, rhs)
        cond = max(np.linalg.cond(ops.mats[name][m, k]) for m, k in ((0, 0), (M, K), (0, K)))
        err = np.linalg.norm(x.cpu().numpy() - ref) / np.linalg.norm(ref)
        assert err <= 1e-12 + 1e-17 * cond, (name, err, cond)
        assert torch.equal(x, inplace)
