"""The radial stencils of steps 2-5 in fixed point, fused (from 48 rows on, with enough modes to share
the FP64 pipe) and per stage, against the oracle: node counts at the edges of the tiles of rows and of the wall zones,
an azimuthal symmetry that makes columns fall off steeply, and a field that is zero but for the
mean flow."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O
from paper_1311_2481_gb300 import inputs as I

pytestmark = pytest.mark.gpu
LZ = 2 * math.pi / 3.16


@pytest.mark.parametrize("kind", ["broadband", "zero"])
@pytest.mark.parametrize("split", [-1, 1])
@pytest.mark.parametrize("N_r,m_p", [(9, 1), (12, 1), (13, 6), (16, 1), (23, 6), (32, 1), (49, 6)])
def test_steps_match_oracle(N_r, m_p, split, kind):
    """Bound: the rounding of the wall Laplacian (weights of order N_r^4) in p, as between any two
    forms of these stages."""
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1311_2481_gb300 import build, tc
    build.build()
    cfg = dict(N_r=N_r, M=18, K=64, m_p=m_p, eta=0.5, Re_i=50.0, Re_o=0.0, L_z=LZ, dt=1e-4)
    ops = O.Operators(O.Params(**cfg))
    u0 = I.initial_state(ops.r, 18, 64, m_p, LZ, 0.5, 50.0, 0.0, kind="broadband", amp=1e-2 if kind == "broadband" else 0.0,
                         seed=3)
    ref = O.run(ops, O.cold_state(u0), 2)
    plan = tc.Plan(**cfg, pc_split=split, no_adjoint=True)
    st = tc.State(plan, torch.from_numpy(u0).cuda())
    plan.step(st, 2)
    for k in ("u", "p"):
        a, b = getattr(st, k).cpu().numpy(), getattr(ref, k)
        assert np.linalg.norm(a - b) <= 1e-10 * np.linalg.norm(b), k


@pytest.mark.parametrize("N_r,m_p", [(9, 1), (18, 6), (19, 1), (20, 6), (25, 1), (32, 1)])
def test_adjoint_step_matches_oracle(N_r, m_p):
    """Blocks of 16 modes with idle warps beside the substitutions, node counts that end within the
    chunks of factor rows.  The bound of the adjoint steps with fewer modes."""
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1311_2481_gb300 import build, tc
    build.build()
    cfg = dict(N_r=N_r, M=18, K=64, m_p=m_p, eta=0.5, Re_i=50.0, Re_o=0.0, L_z=LZ, dt=1e-3)
    ops = O.Operators(O.Params(**cfg))
    u0 = I.initial_state(ops.r, 18, 64, m_p, LZ, 0.5, 50.0, 0.0, kind="broadband", amp=1e-2, seed=4)
    st_o = O.step(ops, O.cold_state(u0))
    y = [I.random_spectral((3,) + ops.prm.shape(), seed=s) for s in (21, 22, 23)]
    ref = O.adjoint_step(ops, st_o, *y)
    plan = tc.Plan(**cfg)
    st = tc.State(plan, torch.from_numpy(st_o.u).cuda())
    st.u_prev.copy_(torch.from_numpy(st_o.u_prev))
    st.N_prev.copy_(torch.from_numpy(st_o.N_prev))
    st.started = True
    bar = tc.StateBar(*[torch.from_numpy(v).cuda() for v in y])
    plan.adjoint_step(st, bar)
    for got, want in zip((bar.u, bar.u_prev, bar.N_prev), ref):
        assert np.linalg.norm(got.cpu().numpy() - want) <= 1e-11 * np.linalg.norm(want)
