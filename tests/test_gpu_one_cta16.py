"""k_fused with one CTA a term (N = 16), whose fhat column, h pencil and sums are kept in tensor memory, where it can go
wrong: a few terms, fewer and more terms than resident CTAs, term ranges, both data forms, both precisions of h;
and beside another kernel that holds tensor memory.  Against the oracle; bound: the FP32 pipeline's 1e-5."""
import numpy as np
import pytest

import bz_inputs as bi
from oracle import kernels, spectral

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
TOL = 1e-5
N, L = 16, 10.0
R = bi.R_from_L(L)


@pytest.fixture(scope="module")
def bz():
    import paper_2004_11239_gb300 as m
    return m


def _rel(a, b):
    return np.max(np.abs(a - b)) / np.max(np.abs(b))


@pytest.mark.parametrize("real", [False, True])
@pytest.mark.parametrize("N_rho,M,h,dtype", [(1, 8, 0, "c128"), (5, 12, 2, "c64"), (26, 12, 0, "c64"), (33, 32, 0, "c128")])
def test_collide_and_term_ranges(bz, real, N_rho, M, h, dtype):
    fhat = bi.random_fhat(N, seed=31, scale=1e-3)
    if dtype == "c64":
        fhat = fhat.astype(np.complex64)
    plan = bz.bz_plan_create_ex(N, L, R, -1.0, 0.5, N_rho, M, h_precision=h,
                                data=bz.BZ_DATA_REAL if real else bz.BZ_DATA_COMPLEX)
    assert bz.bz_plan_pipeline(plan)["cluster"] == 1
    f = torch.from_numpy(fhat).cuda()
    q = torch.full_like(f, float("nan"))
    bz.bz_collide(plan, f, q)
    got = q.cpu().numpy().astype(np.complex128)
    op = spectral.OraclePlan(N, L, R, -1.0, kernels.Kernel("family", 0.5), N_rho, M)
    ref = (spectral.collide_real if real else spectral.collide)(op, fhat.astype(np.complex128))
    err = _rel(got, ref)
    print(f"k_fused<16, 1> P={plan.P} real={real} h={h} {dtype}: rel_Linf={err:.2e}")
    assert err <= TOL
    total = 0
    for a, b in ((0, 2), (2, plan.P), (plan.P, plan.P)):
        bz.bz_collide_terms(plan, a, b, f, q)
        total = total + q.cpu().numpy().astype(np.complex128)
    assert _rel(total, got) <= 1e-6
    plan.close()


def test_beside_another_kernel_with_tensor_memory(bz):
    """Batches at N = 16 and collides at N = 32 on two streams give the bits that each gives alone."""
    small = bz.bz_plan_create(N, L, R, 0.0, 0.5, 16, 12)
    batch = bz.bz_batch_create(small, 64, 0)
    big = bz.bz_plan_create(32, L, R, 0.0, 0.5, 16, 12)
    f16 = torch.from_numpy(np.stack([bi.random_mixture(N, L, seed=b) for b in range(64)])).cuda()
    f32 = torch.from_numpy(bi.random_mixture(32, L, seed=3)).cuda()
    q16, q32 = torch.zeros_like(f16), torch.zeros_like(f32)
    slots = list(range(64))
    bz.bz_batch_collide(batch, slots, f16, q16)
    bz.bz_collide(big, f32, q32)
    torch.cuda.synchronize()
    want16, want32 = q16.clone(), q32.clone()
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for _ in range(10):
        with torch.cuda.stream(streams[0]):
            bz.bz_batch_collide(batch, slots, f16, q16)
        with torch.cuda.stream(streams[1]):
            bz.bz_collide(big, f32, q32)
    torch.cuda.synchronize()
    assert torch.equal(q16, want16) and torch.equal(q32, want32)
    batch.close()
    small.close()
    big.close()
