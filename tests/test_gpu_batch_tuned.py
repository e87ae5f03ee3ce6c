"""Terms per item of batches on the cluster kernels when the caller names none: the smallest that costs a full batch
nothing, as one active slot takes as long as one item (64 at most where 128 and more win under 1%)."""
import pytest

import bz_inputs as bi

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("N,N_rho,M,capacity", [(16, 12, 32, 150), (16, 32, 32, 150), (8, 4, 8, 40)])
def test_tuned_split(N, N_rho, M, capacity):
    import paper_2004_11239_gb300 as bz
    L = 10.0
    plan = bz.bz_plan_create(N, L, bi.R_from_L(L), 0.0, 0.5, N_rho, M)
    batch = bz.bz_batch_create(plan, capacity, 0)
    assert 1 <= batch.terms_per_item <= 64
    f = torch.zeros((capacity, N, N, N), dtype=torch.complex128, device="cuda")
    f[0] = torch.from_numpy(bi.random_mixture(N, L, seed=4)).cuda()
    g = f.clone()
    bz.bz_batch_step_rk(batch, [0], f, 0.01, 1)
    one = g[0].clone()
    bz.bz_step_rk(plan, one, 0.0, 0.01, 1)
    # the change over the step, up to the grouping of the sums
    assert float((f[0] - one).abs().max() / (one - g[0]).abs().max()) <= 1e-6
    batch.close()
    plan.close()
