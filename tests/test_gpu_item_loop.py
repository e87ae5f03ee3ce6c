"""Batches whose CTAs take several work items each, of several instances with data and gamma of their own: the sums, h
and twiddles that an item leaves behind must not reach the next.  More than two items a CTA, not a multiple;
slots whose items come first, second and third against the oracle (1e-5, the FP32 pipeline's bar), and each as it is
alone, to the bit."""
import numpy as np
import pytest

import bz_inputs as bi
from oracle import kernels, spectral

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
L = 10.0
R = bi.R_from_L(L)


@pytest.mark.parametrize("N,real,slots,terms", [(32, False, 21, 1), (32, True, 21, 1), (32, False, 31, 8),
                                                   (16, False, 43, 1), (16, True, 80, 2), (24, False, 25, 1)])
def test_several_items_a_cta(N, real, slots, terms):
    import paper_2004_11239_gb300 as bz
    plan = bz.bz_plan_create_ex(N, L, R, 0.0, 0.5, 2, 12, data=bz.BZ_DATA_REAL if real else bz.BZ_DATA_COMPLEX)
    batch = bz.bz_batch_create(plan, slots, terms)
    items = slots * -(-plan.P // batch.terms_per_item)
    ctas = bz.bz_plan_pipeline(plan)["clusters"]
    assert items > 2 * ctas and items % ctas
    f = np.stack([bi.random_mixture(N, L, seed=700 + b) * (1.0 + 0.1 * b) for b in range(slots)])
    gammas = [-1.0 if b % 3 == 1 else 0.0 for b in range(slots)]
    for b, g in enumerate(gammas):
        bz.bz_batch_set_gamma(batch, b, g)
    fd = torch.from_numpy(f).cuda()
    q, alone = torch.zeros_like(fd), torch.zeros_like(fd)
    order = list(range(slots))[::-1]
    bz.bz_batch_collide(batch, order, fd, q)
    op = {g: spectral.OraclePlan(N, L, R, g, kernels.Kernel("family", 0.5), 2, 12) for g in (0.0, -1.0)}
    collide = spectral.collide_real if real else spectral.collide
    for b in (order[0], order[slots // 2], order[slots // 2 + 1], order[-1]):
        ref = collide(op[gammas[b]], f[b])
        assert np.max(np.abs(q[b].cpu().numpy() - ref)) / np.max(np.abs(ref)) <= 1e-5, b
        bz.bz_batch_collide(batch, [b], fd, alone)
        assert torch.equal(alone[b], q[b])
    batch.close()
    plan.close()
