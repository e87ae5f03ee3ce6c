"""h = IFFT(fhat) formed in double-float arithmetic (bz_hff.cu), seen through the operator.

A few terms, so that a wrong line, lane or plane of h shows at every mode.  Data whose modes span many
decades (magnitudes 1e-30 .. 1, signs mixed) exercise the split of doubles; complex64 input takes the other
load; an infinity must still be reported.  Bound: the FP32 pipeline's 1e-5 of max |Q|."""
import numpy as np
import pytest

import bz_inputs as bi
from oracle import kernels, spectral
from oracle import spectral2d

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
TOL = 1e-5


@pytest.fixture(scope="module")
def bz():
    import paper_2004_11239_gb300 as m
    return m


def _decades(shape, seed):
    rng = np.random.default_rng(seed)
    mag = 10.0 ** rng.uniform(-30, 0, size=shape)
    return mag * np.exp(2j * np.pi * rng.random(shape)) * np.where(rng.random(shape) < 0.02, 0.0, 1.0)


@pytest.mark.parametrize("N", [8, 16, 24, 32])
@pytest.mark.parametrize("dtype", ["c128", "c64"])
def test_3d(bz, N, dtype):
    L = 6.62
    f = _decades((N, N, N), N)
    if dtype == "c64":
        f = f.astype(np.complex64)
    plan = bz.bz_plan_create(N, L, 6.0, 0.0, 0.5, 1, 4)
    fd = torch.from_numpy(f).cuda()
    q = torch.empty_like(fd)
    bz.bz_collide(plan, fd, q)
    ref = spectral.collide(spectral.OraclePlan(N, L, 6.0, 0.0, kernels.Kernel("family", 0.5), 1, 4),
                           f.astype(np.complex128))
    err = np.max(np.abs(q.cpu().numpy() - ref)) / np.max(np.abs(ref))
    assert err <= TOL, err
    assert bz.bz_plan_check_finite(plan) == 0
    f = f.copy()
    f[1, 2, 3] = np.inf
    bz.bz_collide(plan, torch.from_numpy(f).cuda(), q)
    assert bz.bz_plan_check_finite(plan) == 1
    plan.close()


@pytest.mark.parametrize("N", [8, 16, 32, 64])
def test_2d(bz, N):
    L = 6.62
    f = _decades((N, N), N + 1)
    plan = bz.bz_plan_create_ex(N, L, 6.0, 0.0, 0.0, 1, 5, kernel=bz.BZ_KERNEL_B2, dim=2)
    fd = torch.from_numpy(f).cuda()
    q = torch.empty_like(fd)
    bz.bz_collide(plan, fd, q)
    ref = spectral2d.collide2d(spectral2d.OraclePlan2D(N, L, 6.0, 0.0, kernels.Kernel2D("b2"), 1, 5), f)
    err = np.max(np.abs(q.cpu().numpy() - ref)) / np.max(np.abs(ref))
    assert err <= TOL, err
    plan.close()
