"""The chunked pipeline at N = 48 and 64 (bz_lines.cu) where its splits can go wrong: fewer terms than a chunk, than
the accumulating pass's splits, one term; chunks that do not divide the terms, one and several of
them on two streams; an empty range; data with content on the Nyquist planes.  Against the oracle at
every mode; bound: the FP32 pipeline's 1e-5 of max |Q|, 2e-5 for FP32 h on unresolved data."""
import numpy as np
import pytest

import bz_inputs as bi
from oracle import kernels, spectral

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
L = 10.0
R = bi.R_from_L(L)


@pytest.fixture(scope="module")
def bz():
    import paper_2004_11239_gb300 as m
    return m


@pytest.mark.parametrize("N,real,N_rho,M,chunk", [
    (48, False, 1, 1, 0), (48, True, 1, 2, 0), (48, True, 2, 8, 3), (48, False, 1, 9, 4),
    (64, False, 1, 1, 0), (64, True, 1, 2, 0), (64, True, 1, 8, 1), (64, False, 1, 4, 3),
])
def test_chunks(bz, N, real, N_rho, M, chunk):
    fhat = bi.random_fhat(N, seed=90 + N, scale=1e-3)
    plan = bz.bz_plan_create_ex(N, L, R, -1.0, 0.5, N_rho, M, data=int(real), chunk_terms=chunk)
    assert bz.bz_plan_pipeline(plan)["pipeline"] == "chunked"
    f = torch.from_numpy(fhat).cuda()
    q = torch.full_like(f, float("nan"))
    bz.bz_collide(plan, f, q)
    got = q.cpu().numpy()
    op = spectral.OraclePlan(N, L, R, -1.0, kernels.Kernel("family", 0.5), N_rho, M)
    ref = (spectral.collide_real if real else spectral.collide)(op, fhat)
    err = np.max(np.abs(got - ref)) / np.max(np.abs(ref))
    print(f"lines N={N} real={real} P={plan.P} chunk={chunk}: rel_Linf={err:.2e}")
    assert err <= 2e-5
    if real:
        ny = spectral.nyquist_mask(N)
        assert np.array_equal(spectral.mirror(got)[~ny], np.conj(got)[~ny])
    bz.bz_collide(plan, f, q)                               # nothing is left over from the last call
    assert np.array_equal(q.cpu().numpy(), got)
    bz.bz_collide_terms(plan, 0, 0, f, q)
    assert not q.cpu().numpy().any()
    plan.close()
