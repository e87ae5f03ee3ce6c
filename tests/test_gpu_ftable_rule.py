"""The weight table of a caller's sphere rule whose points are unit to a few digits, against single entries.

Where a mode is parallel to a point longer than 1 by d, k.qhat is beyond |k|: the entries sum the theta rule with
k - (k.qhat) qhat cut off at zero there, and the table's series takes cos chi = 1.  Both move by at most about d relative
to the term's largest weight (2 d allowed, beside the FP32 rounding), not by z d, z = pi r |k| / (2L)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("N,R", [(64, 6.0), (16, 60.0)])        # series up to and beyond 160 terms
def test_points_longer_than_one(N, R):
    import paper_2004_11239_gb300 as bz
    xyz = np.array([(0.26727, 0.53453, 0.80179), (-0.26727, -0.53453, -0.80179), (0.57736, 0.57735, 0.57735),
                    (0.6, 0.8, 0.0)])
    k = [np.array((1, 2, 3)), np.array((1, 2, 3)), np.array((1, 1, 1)), np.array((3, 4, 0))]
    plan = bz.bz_plan_create_ex(N, 6.62, R, 0.0, 0.5, 2, 4, sphere=(xyz, np.full(4, np.pi)))
    alpha = bz.bz_plan_alpha(plan, 0, plan.P).cpu().numpy().astype(np.complex128)
    c = bz.bz_plan_terms(plan)[4]
    rng = np.random.default_rng(3)
    for p in range(plan.P):
        d = abs(np.linalg.norm(xyz[p % 4]) - 1.0)
        top_m = (N // 2 - 1) // int(k[p % 4].max())
        idx = np.concatenate([np.outer([m for m in range(-top_m, top_m + 1) if m], k[p % 4]) % N,
                              rng.integers(0, N, size=(100, 3))])
        F = bz.bz_ftable_entries(plan, torch.from_numpy(idx.astype(np.int32)).cuda().contiguous(),
                                 torch.full((len(idx),), p, dtype=torch.int32, device="cuda")).cpu().numpy()
        ref = c[p] * F / N ** 3
        err = np.abs(alpha[p][idx[:, 0], idx[:, 1], idx[:, 2]] - ref)
        top = np.max(np.abs(ref))
        assert np.all(err <= 2.0 ** -23 * np.abs(ref) + (2.0 * d + 1e-11) * top), (p, d, np.max(err) / top)
    plan.close()
