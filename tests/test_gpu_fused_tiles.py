"""The fused steps 2-5 with fixed-point stencils, in blocks of 16 and of 8 modes: every remainder of the
tiles of 4 rows, and columns steep enough that single rows and whole tiles are left to FP64 sums."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O
from paper_1311_2481_gb300 import inputs as I

pytestmark = pytest.mark.gpu
LZ = 2 * math.pi / 3.16


@pytest.mark.parametrize("kind", ["broadband", "zero"])
@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("N_r,m_p", [(48, 1), (49, 6), (50, 1), (51, 6), (97, 6), (100, 1)])
def test_steps_match_oracle(N_r, m_p, mixed, kind):
    """The bounds of the same steps with fewer modes: the rounding of the wall Laplacian (weights of
    order N_r^4) in p; FP32 transforms of the perturbation in the mixed form."""
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1311_2481_gb300 import build, tc
    build.build()
    M, K = 21, 64
    # the rule of the fixed-point stencils (48 rows, 256 threads per SM), with a margin
    T = 16 if N_r <= 96 else 8
    threads = -(-(M + 1) * (2 * K + 1) // T) * (256 if T == 16 else 128)
    assert threads >= 1.1 * 256 * torch.cuda.get_device_properties(0).multi_processor_count
    cfg = dict(N_r=N_r, M=M, K=K, m_p=m_p, eta=0.5, Re_i=50.0, Re_o=0.0, L_z=LZ, dt=2e-5)
    ops = O.Operators(O.Params(**cfg, P_theta=64, P_z=192))
    u0 = I.initial_state(ops.r, M, K, m_p, LZ, 0.5, 50.0, 0.0, kind="broadband", amp=1e-2 if kind == "broadband" else 0.0,
                         seed=3)
    ref = O.run(ops, O.cold_state(u0), 2)
    plan = tc.Plan(**cfg, P_theta=64, P_z=192, no_adjoint=True, precision=tc.TC_MIXED if mixed else tc.TC_FP64)
    st = tc.State(plan, torch.from_numpy(u0).cuda())
    plan.step(st, 2)
    for k in ("u", "p"):
        a, b = getattr(st, k).cpu().numpy(), getattr(ref, k)
        bound = 1e-10 * N_r / 48 if not mixed else 1e-8 if k == "u" else 1e-5
        assert np.linalg.norm(a - b) <= bound * np.linalg.norm(b), k
