"""tc_nonlinear_noalloc on plans whose staging lines fit the static array but whose rows are many: the
exponents that count are those of the staged rows, and a mixed plan's nonlinear term has none."""
import ctypes
import math

import pytest

torch = pytest.importorskip("torch")

from paper_1311_2481_gb300 import inputs as I

pytestmark = pytest.mark.gpu
LZ = 2 * math.pi / 3.16


@pytest.mark.parametrize("mixed,M,K,P_theta,P_z,rows", [
    (False, 85, 4, 256, 12, 423),   # 79.9 MiB of lines, 5.4 KB of exponents per row of 2048
    (False, 85, 4, 256, 12, 7),
    (False, 69, 1, 144, 3, 0),      # short lines: the most exponents per byte of lines, all rows
    (True, 93, 1, 192, 3, 0),       # 79.3 MiB of FP32 staging, adjoint regions behind it
])
def test_many_rows(mixed, M, K, P_theta, P_z, rows):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1311_2481_gb300 import build, tc
    build.build()
    plan = tc.Plan(2048, M, K, 1, 0.5, 50.0, 0.0, LZ, 1e-6, P_theta=P_theta, P_z=P_z, stage_rows=rows,
                   no_adjoint=not mixed, precision=tc.TC_MIXED if mixed else tc.TC_FP64)
    u = torch.from_numpy(I.random_spectral((3, 2048, M + 1, 2 * K + 1), 5, hermitian_K=K)).cuda()
    ref = plan.nonlinear(u)
    got = torch.full_like(u, float("nan"))
    lib = tc.load_library()
    st = lib.tc_nonlinear_noalloc(plan.handle, ctypes.c_void_p(u.data_ptr()), ctypes.c_void_p(got.data_ptr()),
                                  ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == tc.TC_OK, lib.tc_plan_last_error(plan.handle)
    torch.cuda.synchronize()
    assert torch.equal(got, ref)
