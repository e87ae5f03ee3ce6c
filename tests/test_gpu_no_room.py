"""A plan at N = 32 whose second weight table finds no memory takes the cluster kernels, as it did before it had one.

All but 414 MiB is reserved first.  8 N^3 P = 256 MiB of weights and what else a plan has (some 4 MiB with one term a
chunk) fit; of the rest the complex form wants 256 for its second table, the real one 144 and 21 for the items' sums, where
its pair tables take 140."""
import pytest

import bz_inputs as bi

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
N, L = 32, 10.0
R = bi.R_from_L(L)


@pytest.mark.parametrize("real", [False, True])
def test_falls_back_to_clusters(real):
    import paper_2004_11239_gb300 as bz
    args = (N, L, R, 0.0, 0.5)
    data = bz.BZ_DATA_REAL if real else bz.BZ_DATA_COMPLEX
    for kw in ({}, {"cluster": 8, "ctas_per_sm": 2 if real else 0}):                 # loads every kernel
        bz.bz_plan_create_ex(*args, 1, 8, data=data, **kw).close()
    full = bz.bz_plan_create_ex(*args, 32, 32, data=data, chunk_terms=1)
    f = torch.from_numpy(bi.random_mixture(N, L, seed=9)).cuda()
    q, r = torch.empty_like(f), torch.empty_like(f)
    bz.bz_collide(full, f, q)
    assert bz.bz_plan_pipeline(full)["kernel"] == ("k_col32" if real else "k_cube32")
    full.close()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - (414 << 20), dtype=torch.uint8, device="cuda")
    try:
        plan = bz.bz_plan_create_ex(*args, 32, 32, data=data, chunk_terms=1)
    finally:
        del hold
        torch.cuda.empty_cache()
    kernel = bz.bz_plan_pipeline(plan)["kernel"]
    assert kernel in (("k_fused", "k_pair3", "chunked") if real else ("k_fused", "chunked"))
    bz.bz_collide(plan, f, r)
    assert float((q - r).abs().max() / q.abs().max()) <= 1e-5
    plan.close()
