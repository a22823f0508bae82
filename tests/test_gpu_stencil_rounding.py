"""Rounding of the radial derivative, row by row: u_r = 1 and u_z = f(r) in the mean mode alone make
N_z = d_r f there.  Columns that are smooth, vanish at the walls, oscillate or rise by 2^192 across the gap."""
import math
from fractions import Fraction

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu
LZ = 2 * math.pi / 3.16

COLUMNS = {
    "couette": lambda r: 100 / 3 * (4 / r - r),
    "smooth": lambda r: 1 + 0.3 * np.sin(3 * r),
    "walls": lambda r: (r - 1) ** 2 * (2 - r) ** 2,
    "waves": lambda r: (r - 1) ** 2 * (2 - r) ** 2 * np.sin(20 * math.pi * r),
    "gauss": lambda r: np.exp(-((r - 1.5) / 0.1) ** 2),
    "r^32": lambda r: r ** 32.0,
    "r^-32": lambda r: r ** -32.0,
    "r^192": lambda r: r ** 192.0,
    "r^-192": lambda r: r ** -192.0,
    "noise": lambda r: np.random.default_rng(3).standard_normal(len(r)),
}


@pytest.mark.parametrize("N_r", [45, 64, 96, 256])
@pytest.mark.parametrize("name", sorted(COLUMNS))
def test_derivative_rounds_like_an_fp64_sum(name, N_r):
    """u = 2^-53.  A sum of 9 FP64 FMAs is off by at most 9 u sum |w f|, and by 0.3 to 2 of it as a rule.
    Fixed point drops what lies 2^-60 below the window's largest value; rows whose next
    neighbours are more than 2^-3 below it are left to FP64 sums, and these neighbours' weights are at
    least 2^-2.4 of sum |w|, so that is 2^-53.6 sum |w f| (standard deviation): 4 u sum |w f| holds
    both.  8 u of the result for the transforms and their scale.  In norm the column is as good
    as 2 u of its terms."""
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1311_2481_gb300 import build, tc
    build.build()
    plan = tc.Plan(N_r, 1, 1, 1, 0.5, 50.0, 0.0, LZ, 1e-3, P_theta=6, P_z=108, no_adjoint=True)
    f = COLUMNS[name](plan.nodes())
    w, c0 = plan.fd_weights(1)
    u = np.zeros((3, N_r, 2, 3), np.complex128)
    u[0, :, 0, 1] = u[1, :, 0, 1] = 1.0
    u[2, :, 0, 1] = f
    got = plan.nonlinear(torch.from_numpy(u).cuda()).cpu().numpy()[2, :, 0, 1]
    assert not got.imag.any()
    U = 2.0 ** -53
    err, terms = np.zeros(N_r), np.zeros(N_r)
    for j in range(N_r):
        t = [Fraction(float(w[j, q])) * Fraction(float(f[c0[j] + q])) for q in range(9)]
        d = sum(t)
        err[j], terms[j] = abs(Fraction(float(got.real[j])) - d), sum(abs(x) for x in t)
        assert err[j] <= U * (4 * terms[j] + 8 * abs(float(d))), (j, err[j] / (U * terms[j]))
    assert np.linalg.norm(err) <= 2 * U * np.linalg.norm(terms)
