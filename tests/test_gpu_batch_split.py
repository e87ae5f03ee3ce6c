"""Work items of batches on the one-term-per-SM kernels (N = 32) when the caller names no size: fine enough for one
active slot, few enough for a full batch; and the server's account of what they take."""
import time

import numpy as np
import pytest

import bz_inputs as bi

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
N, L = 32, 10.0
R = bi.R_from_L(L)


@pytest.mark.parametrize("real", [False, True])
@pytest.mark.parametrize("capacity,N_rho,M", [(1, 3, 12), (32, 6, 32), (150, 3, 12), (150, 6, 32), (700, 1, 12)])
def test_automatic_split(real, capacity, N_rho, M):
    """One active slot's item has at most 18 terms unless 32 waves of items are reached (their sums take memory); its
    result is that of a single collide up to the grouping of the sums (1e-6 of max |Q|)."""
    import paper_2004_11239_gb300 as bz
    plan = bz.bz_plan_create_ex(N, L, R, 0.0, 0.5, N_rho, M, data=bz.BZ_DATA_REAL if real else bz.BZ_DATA_COMPLEX)
    batch = bz.bz_batch_create(plan, capacity, 0)
    sms, tb = torch.cuda.get_device_properties(0).multi_processor_count, batch.terms_per_item
    assert capacity * -(-plan.P // tb) <= max(capacity, 32 * sms)
    assert tb <= 18 or capacity * -(-plan.P // (tb - 1)) > 32 * sms
    f = torch.zeros((capacity, N, N, N), dtype=torch.complex64, device="cuda")
    f[capacity - 1] = torch.from_numpy(bi.random_mixture(N, L, seed=4)).cuda().to(f.dtype)
    q, one = torch.zeros_like(f), torch.empty_like(f[0])
    bz.bz_batch_collide(batch, [capacity - 1], f, q)
    bz.bz_collide(plan, f[capacity - 1].contiguous(), one)
    assert float((q[capacity - 1] - one).abs().max() / one.abs().max()) <= 1e-6
    batch.close()
    plan.close()


@pytest.mark.parametrize("real", [False, True])
def test_server_accounts_for_the_items(real):
    """A group's share of the budget covers what its plan and batch allocate."""
    import paper_2004_11239_gb300 as bz
    server = bz.bz_server_create(32 << 30, max_batch=8, terms_per_item=4)
    f = bi.random_mixture(N, L, seed=6)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    t = bz.bz_submit(server, fhat0=f, N=N, L=L, R=R, gamma=0.0, s=0.5, N_rho=16, M=32, t0=0.0, t_end=0.02, dt=0.02,
                     data=bz.BZ_DATA_REAL if real else bz.BZ_DATA_COMPLEX)
    end = time.time() + 60
    while bz.bz_poll(server, t, N) is None and time.time() < end:
        time.sleep(0.01)
    took = free - torch.cuda.mem_get_info()[0]
    assert took <= bz.bz_server_stats(server)["hbm_used"]
    server.close()
