"""The fused steps 2-5 with many modes, in blocks of 16 and of 8: FP64 stencils with a column for the sum of
u_+ and u_- (below 76 rows, 56 in the mixed form) and fixed-point ones, at every remainder of their tiles
of 4 rows, with columns steep enough that single rows and whole tiles are left to FP64 sums."""
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
@pytest.mark.parametrize("N_r,m_p", [(48, 1), (49, 6), (50, 1), (51, 6), (56, 6), (57, 1), (58, 6), (59, 1),
                                     (75, 6), (76, 6), (77, 1), (78, 6), (79, 1), (97, 6), (100, 1)])
def test_steps_match_oracle(N_r, m_p, mixed, kind):
    """The bounds of the same steps with fewer modes: the rounding of the wall Laplacian (weights of
    order N_r^4) in p; FP32 transforms of the perturbation in the mixed form."""
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1311_2481_gb300 import build, tc
    build.build()
    M, K = 21, 64
    # enough modes for the fixed-point stencils (256 threads per SM), with a margin
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


def test_blocks_without_room_for_the_sum():
    """Two blocks of 8 modes of 180 rows per SM, too few warps for the fixed-point form: FP64 stencils of
    u_+ + u_- term by term."""
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1311_2481_gb300 import build, tc
    build.build()
    cfg = dict(N_r=180, M=18, K=40, m_p=1, eta=0.5, Re_i=50.0, Re_o=0.0, L_z=LZ, dt=2e-5)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert sms < -(-19 * 81 // 8) < 2 * sms
    ops = O.Operators(O.Params(**cfg, P_theta=54, P_z=128))
    u0 = I.initial_state(ops.r, 18, 40, 1, LZ, 0.5, 50.0, 0.0, kind="broadband", amp=1e-2, seed=3)
    ref = O.run(ops, O.cold_state(u0), 2)
    plan = tc.Plan(**cfg, P_theta=54, P_z=128, no_adjoint=True)
    st = tc.State(plan, torch.from_numpy(u0).cuda())
    plan.step(st, 2)
    for k in ("u", "p"):
        a, b = getattr(st, k).cpu().numpy(), getattr(ref, k)
        assert np.linalg.norm(a - b) <= 1e-10 * 180 / 48 * np.linalg.norm(b), k
