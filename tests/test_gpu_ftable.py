"""The plan's weight table (Legendre series) against single entries (the theta rule summed directly).

Both evaluate c_p F(k, r, qhat) / N^3 in FP64 and the table rounds it to FP32, so an entry may differ
by half an FP32 ulp (2^-24 relative) and by the rounding of two different FP64 sums of a few hundred
terms, for which 1e-11 of the term's largest weight is allowed."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("N,N_rho,M,R,L,kernel,s,theta0", [
    (8, 1, 1, 6.0, 6.62, 0, 0.5, 0.0),          # one term
    (8, 5, 9, 6.0, 6.62, 0, 0.75, 0.0),         # a partial group of terms
    (16, 3, 12, 9.0616, 10.0, 0, 0.25, 0.0),
    (24, 4, 18, 9.0616, 10.0, 2, 0.0, 0.0),     # b8
    (32, 4, 12, 6.0, 6.62, 7, 0.0, 0.0),        # Debye-Yukawa, a kink in the angle
    (32, 2, 32, 6.0, 6.62, 0, 0.5, 0.785),      # angular cutoff: no Taylor part
    (48, 2, 12, 9.0616, 10.0, 0, 0.0, 0.0),
    (64, 3, 12, 9.0616, 10.0, 0, 0.5, 0.0),     # the longest series in use
    (16, 2, 8, 60.0, 6.62, 0, 0.5, 0.0),        # R far beyond the box: phases of several hundred
    (16, 3, 4, 1e-3, 10.0, 0, 0.5, 0.0),        # a tiny ball: the first terms only
])
def test_table_equals_entries(N, N_rho, M, R, L, kernel, s, theta0):
    import paper_2004_11239_gb300 as bz
    plan = bz.bz_plan_create_ex(N, L, R, 0.0, s, N_rho, M, kernel=kernel, theta0=theta0)
    alpha = bz.bz_plan_alpha(plan, 0, plan.P).cpu().numpy().astype(np.complex128)
    c = bz.bz_plan_terms(plan)[4]
    rng = np.random.default_rng(7)
    for p in sorted({0, plan.P // 2, plan.P - 1}):
        k = rng.integers(0, N, size=(300, 3))
        k[:8] = [(0, 0, 0), (0, 0, 1), (N // 2, N // 2, N // 2), (N // 2, 0, 1), (0, N // 2, N - 1), (1, 0, 0),
                 (N - 1, 0, 0), (N - 1, N - 1, N - 1)]
        F = bz.bz_ftable_entries(plan, torch.from_numpy(k.astype(np.int32)).cuda().contiguous(),
                                 torch.full((len(k),), p, dtype=torch.int32, device="cuda")).cpu().numpy()
        ref = c[p] * F / N ** 3
        got = alpha[p][k[:, 0], k[:, 1], k[:, 2]]
        top = np.max(np.abs(c[p] * F)) / N ** 3
        err = np.abs(got - ref)
        assert np.all(err <= 2.0 ** -23 * np.abs(ref) + 1e-11 * top), (p, err.max() / top)
    plan.close()
