"""The 2D kernel's slots where they can go wrong: one term, a CTA that is not full, blocks of unequal length, more
terms than resident slots; term ranges and an empty one; RK4.  Against the 2D oracle; bound: the FP32
pipeline's 1e-5 of max |Q| (of the change of f for RK4)."""
import numpy as np
import pytest

import bz_inputs as bi
from oracle import kernels, spectral2d

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
TOL = 1e-5
L, R = 6.62, 6.0


@pytest.fixture(scope="module")
def bz():
    import paper_2004_11239_gb300 as m
    return m


@pytest.mark.parametrize("N,N_rho,M,dtype", [(8, 1, 1, "c128"), (8, 1, 17, "c64"), (16, 3, 3, "c128"), (32, 1, 5, "c64"),
                                             (32, 1, 3, "c128"), (64, 1, 1, "c64"), (64, 1, 3, "c128"), (64, 43, 16, "c64")])
def test_slots(bz, N, N_rho, M, dtype):
    f = bi.random_mixture2d(N, L, 7)
    if dtype == "c64":
        f = f.astype(np.complex64)
    plan = bz.bz_plan_create_ex(N, L, R, 0.0, 0.0, N_rho, M, kernel=bz.BZ_KERNEL_B2, dim=2)
    fd = torch.from_numpy(f).cuda()
    q = torch.full_like(fd, float("nan"))
    bz.bz_collide(plan, fd, q)
    got = q.cpu().numpy().astype(np.complex128)
    op = spectral2d.OraclePlan2D(N, L, R, 0.0, kernels.Kernel2D("b2"), N_rho, M)
    ref = spectral2d.collide2d(op, f.astype(np.complex128))
    assert np.max(np.abs(got - ref)) <= TOL * np.max(np.abs(ref))
    part = 0
    for a, b in ((0, plan.P // 3), (plan.P // 3, plan.P), (plan.P, plan.P)):
        bz.bz_collide_terms(plan, a, b, fd, q)
        part = part + q.cpu().numpy().astype(np.complex128)
    assert np.max(np.abs(part - got)) <= 1e-6 * np.max(np.abs(ref))
    if dtype == "c128" and plan.P < 20:
        bz.bz_step_rk(plan, fd, 0.0, 0.05, 2)
        fr = spectral2d.rk4_2d(op, f, 0.05, 2)
        assert np.max(np.abs(fd.cpu().numpy() - fr)) <= TOL * np.max(np.abs(fr - f))
    plan.close()
