"""The one-term-per-SM kernel of complex plans at N = 32 (k_cube32, what such a plan runs by default) where its items
can go wrong: one term, fewer and more terms than SMs, a last item that is not full; term ranges, RK4,
batches, the padded form on its grid.  Against the oracle; bound: the FP32 pipeline's 1e-5."""
import numpy as np
import pytest

import bz_inputs as bi
from oracle import kernels, spectral

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
TOL = 1e-5
N, L = 32, 10.0
R = bi.R_from_L(L)


@pytest.fixture(scope="module")
def bz():
    import paper_2004_11239_gb300 as m
    return m


def _plan(bz, gamma, s, N_rho, M):
    p = bz.bz_plan_create(N, L, R, gamma, s, N_rho, M)
    assert bz.bz_plan_pipeline(p)["kernel"] == "k_cube32"
    return p


def _rel(a, b):
    return np.max(np.abs(a - b)) / np.max(np.abs(b))


@pytest.mark.parametrize("N_rho,M,data,dtype", [(1, 1, "random", "c128"), (3, 9, "random", "c64"), (17, 9, "mixture", "c128"),
                                                (9, 18, "random", "c64"), (7, 49, "random", "c128")])
def test_collide_and_term_ranges(bz, N_rho, M, data, dtype):
    fhat = bi.random_fhat(N, seed=72, scale=1e-3) if data == "random" else bi.random_mixture(N, L, seed=6)
    if dtype == "c64":
        fhat = fhat.astype(np.complex64)
    plan = _plan(bz, -1.0, 0.5, N_rho, M)
    f = torch.from_numpy(fhat).cuda()
    q = torch.full_like(f, float("nan"))
    bz.bz_collide(plan, f, q)
    got = q.cpu().numpy().astype(np.complex128)
    op = spectral.OraclePlan(N, L, R, -1.0, kernels.Kernel("family", 0.5), N_rho, M)
    err = _rel(got, spectral.collide(op, fhat.astype(np.complex128)))
    print(f"k_cube32 P={plan.P} {data} {dtype}: rel_Linf={err:.2e}")
    assert err <= TOL
    total = 0
    for a, b in ((0, 1), (1, plan.P), (plan.P, plan.P)):
        bz.bz_collide_terms(plan, a, b, f, q)
        total = total + q.cpu().numpy().astype(np.complex128)
    assert _rel(total, got) <= 1e-6
    plan.close()


def test_rk4_and_batches(bz):
    plan = _plan(bz, 0.0, 0.5, 3, 9)
    f = np.stack([bi.random_mixture(N, L, seed=500 + b) for b in range(5)])
    op = {g: spectral.OraclePlan(N, L, R, g, kernels.Kernel("family", 0.5), 3, 9) for g in (0.0, -1.0)}
    one = torch.from_numpy(f[0]).cuda()
    bz.bz_step_rk(plan, one, 0.0, 0.05, 2)
    assert _rel(one.cpu().numpy() - f[0], spectral.rk4(op[0.0], f[0], 0.05, 2) - f[0]) <= TOL
    for dtype in (torch.complex128, torch.complex64):
        batch = bz.bz_batch_create(plan, 5, 0)
        bz.bz_batch_set_gamma(batch, 3, -1.0)
        fd = torch.from_numpy(f).cuda().to(dtype)
        qd = torch.zeros_like(fd)
        bz.bz_batch_collide(batch, [3, 0], fd, qd)
        q = qd.cpu().numpy()
        for slot, g in ((3, -1.0), (0, 0.0)):
            assert _rel(q[slot], spectral.collide(op[g], fd[slot].cpu().numpy().astype(np.complex128))) <= TOL
        assert not q[1].any()
        alone = torch.zeros_like(fd)
        bz.bz_batch_collide(batch, [3], fd, alone)
        assert np.array_equal(alone[3].cpu().numpy(), q[3])
        if dtype == torch.complex128:
            bz.bz_batch_step_rk(batch, [3, 0], fd, 0.05, 1)
            g1 = fd.cpu().numpy()
            for slot, g in ((3, -1.0), (0, 0.0)):
                assert _rel(g1[slot] - f[slot], spectral.rk4(op[g], f[slot], 0.05, 1) - f[slot]) <= TOL
            assert np.array_equal(g1[1], f[1])
        batch.close()
    plan.close()


def test_padded_grid(bz):
    n = 16
    fhat = bi.random_mixture(n, L, seed=3)
    plan = bz.bz_plan_create_ex(n, L, R, 0.0, 0.5, 2, 9, conv=bz.BZ_CONV_PADDED)
    assert bz.bz_plan_pipeline(plan)["kernel"] == "k_cube32"
    f = torch.from_numpy(fhat).cuda()
    q = torch.empty_like(f)
    bz.bz_collide(plan, f, q)
    ref = bz.bz_plan_create_ex(n, L, R, 0.0, 0.5, 2, 9, conv=bz.BZ_CONV_PADDED, cluster=8)
    r = torch.empty_like(f)
    bz.bz_collide(ref, f, r)
    assert bz.bz_plan_pipeline(ref)["kernel"] == "k_fused"
    assert _rel(q.cpu().numpy(), r.cpu().numpy()) <= TOL
    plan.close()
    ref.close()
