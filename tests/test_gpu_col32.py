"""The one-term-per-SM kernel of real-data plans at N = 32 (k_col32, what such a plan runs by default):
collides, term ranges, RK4 steps and batches against the oracle's real-data reading at the sizes
where its items and tables can go wrong (fewer terms than SMs, a last item that is not full, single
terms), on data with content on the Nyquist planes.  Bounds as for the other FP32 kernels: 1e-5 of
max |Q|, the FP32 pipeline's bar."""
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


def _plan(bz, gamma, s, N_rho, M, **kw):
    p = bz.bz_plan_create_ex(N, L, R, gamma, s, N_rho, M, data=bz.BZ_DATA_REAL, **kw)
    assert bz.bz_plan_pipeline(p)["kernel"] == "k_col32"
    return p


def _rel(a, b):
    return np.max(np.abs(a - b)) / np.max(np.abs(b))


@pytest.mark.parametrize("N_rho,M,data,dtype", [(1, 2, "random", "c128"), (2, 12, "random", "c64"),
                                                (9, 18, "mixture", "c128"), (5, 32, "random", "c128")])
def test_collide_and_term_ranges(bz, N_rho, M, data, dtype):
    fhat = bi.random_fhat(N, seed=71, scale=1e-3) if data == "random" else bi.random_mixture(N, L, seed=5)
    if dtype == "c64":
        fhat = fhat.astype(np.complex64)
    plan = _plan(bz, -1.0, 0.5, N_rho, M)
    f = torch.from_numpy(fhat).cuda()
    q = torch.empty_like(f)
    bz.bz_collide(plan, f, q)
    got = q.cpu().numpy().astype(np.complex128)
    op = spectral.OraclePlan(N, L, R, -1.0, kernels.Kernel("family", 0.5), N_rho, M)
    ref = spectral.collide_real(op, fhat.astype(np.complex128))
    err = _rel(got, ref)
    print(f"k_col32 P={plan.P} {data} {dtype}: rel_Linf={err:.2e}")
    assert err <= TOL
    ny = spectral.nyquist_mask(N)
    assert np.array_equal(spectral.mirror(got)[~ny], np.conj(got)[~ny])
    assert got[0, 0, 0] == 0
    total = 0
    for a, b in ((0, 2), (2, plan.P), (plan.P, plan.P)):
        r = torch.empty_like(f)
        bz.bz_collide_terms(plan, a, b, f, r)
        total = total + r.cpu().numpy().astype(np.complex128)
    assert _rel(total, got) <= 1e-6
    plan.close()


def test_fp32_h_and_rk4(bz):
    fhat = bi.random_mixture(N, L, seed=9)
    op = spectral.OraclePlan(N, L, R, 0.0, kernels.Kernel("family", 0.5), 3, 12)
    ref = spectral.collide_real(op, fhat)
    f = torch.from_numpy(fhat).cuda()
    plan = _plan(bz, 0.0, 0.5, 3, 12, h_precision=bz.BZ_H_FP32)
    q = torch.empty_like(f)
    bz.bz_collide(plan, f, q)
    assert _rel(q.cpu().numpy(), ref) <= 2.5e-5         # the bar of FP32 h on an under-resolved mixture
    plan.close()
    plan = _plan(bz, 0.0, 0.5, 3, 12)
    fr = spectral.rk4_real(op, fhat, 0.05, 2)
    bz.bz_step_rk(plan, f, 0.0, 0.05, 2)
    assert _rel(f.cpu().numpy() - fhat, fr - fhat) <= TOL
    plan.close()


@pytest.mark.parametrize("cap,N_rho,M", [(3, 2, 12), (7, 3, 2)])
def test_batches(bz, cap, N_rho, M):
    plan = _plan(bz, 0.0, 0.5, N_rho, M)
    batch = bz.bz_batch_create(plan, cap, 0)
    gam = {2: -1.0, 0: 0.0}
    for slot, g in gam.items():
        bz.bz_batch_set_gamma(batch, slot, g)
    f = np.stack([bi.random_fhat(N, seed=500 + b, scale=1e-3) for b in range(cap)])
    fd = torch.from_numpy(f).cuda()
    qd = torch.zeros_like(fd)
    bz.bz_batch_collide(batch, [2, 0], fd, qd)
    q = qd.cpu().numpy()
    for slot, g in gam.items():
        op = spectral.OraclePlan(N, L, R, g, kernels.Kernel("family", 0.5), N_rho, M)
        assert _rel(q[slot], spectral.collide_real(op, f[slot])) <= TOL
    assert not q[1].any()
    alone = torch.zeros_like(fd)
    bz.bz_batch_collide(batch, [2], fd, alone)
    assert np.array_equal(alone[2].cpu().numpy(), q[2])
    bz.bz_batch_step_rk(batch, [2, 0], fd, 0.05, 1)
    g = fd.cpu().numpy()
    for slot, gm in gam.items():
        op = spectral.OraclePlan(N, L, R, gm, kernels.Kernel("family", 0.5), N_rho, M)
        assert _rel(g[slot] - f[slot], spectral.rk4_real(op, f[slot], 0.05, 1) - f[slot]) <= TOL
    assert np.array_equal(g[1], f[1])
    batch.close()
    plan.close()
