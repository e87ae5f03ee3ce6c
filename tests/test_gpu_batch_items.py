"""The terms per item that a caller asks for, on the kernels that run a term on one SM (N = 32): a quarter of them (half where
a full batch would have too many items), at least one; the sums are those of a single collide up to the rounding of their grouping (1e-6 of max|Q|)."""
import numpy as np
import pytest

import bz_inputs as bi

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("real", [False, True])
@pytest.mark.parametrize("capacity,asked,taken", [(3, 1, 1), (3, 5, 2), (3, 32, 8), (3, 4096, 36), (200, 4, 2)])
def test_terms_per_item(real, capacity, asked, taken):
    import paper_2004_11239_gb300 as bz
    N, L = 32, 10.0
    plan = bz.bz_plan_create_ex(N, L, bi.R_from_L(L), 0.0, 0.5, 3, 12,
                                data=bz.BZ_DATA_REAL if real else bz.BZ_DATA_COMPLEX)
    batch = bz.bz_batch_create(plan, capacity, asked)
    assert batch.terms_per_item == taken
    f = torch.from_numpy(np.stack([bi.random_mixture(N, L, seed=40 + b) for b in range(3)])).cuda()
    f = torch.cat([f, torch.zeros(capacity - 3, N, N, N, dtype=f.dtype, device="cuda")])
    q, one = torch.zeros_like(f), torch.zeros_like(f[0])
    bz.bz_batch_collide(batch, [2, 0], f, q)
    for slot in (0, 2):
        bz.bz_collide(plan, f[slot].contiguous(), one)
        assert float((q[slot] - one).abs().max() / one.abs().max()) <= 1e-6
    batch.close()
    plan.close()
