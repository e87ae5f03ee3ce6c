"""Complex collides at N = 32 of few terms run on k_fused's clusters, those of more on k_cube32, in one plan.

On both sides of the line between the two (a resident cluster for each term), against the same terms of a plan that
asks for clusters: bit-equal where the plan takes the clusters itself, within the FP32 pipeline's 1e-5 of
max |Q| where it takes k_cube32."""
import pytest

import bz_inputs as bi

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
N, L = 32, 10.0
R = bi.R_from_L(L)


@pytest.mark.parametrize("dtype", [torch.complex64, torch.complex128])
def test_both_sides_of_the_line(dtype):
    import paper_2004_11239_gb300 as bz
    plan = bz.bz_plan_create(N, L, R, -1.0, 0.5, 17, 18)
    ref = bz.bz_plan_create_ex(N, L, R, -1.0, 0.5, 17, 18, cluster=8)
    G, sms = bz.bz_plan_pipeline(ref)["clusters"], bz.bz_plan_pipeline(plan)["clusters"]
    f = torch.from_numpy(bi.random_mixture(N, L, seed=12)).cuda().to(dtype)
    q, r = torch.empty_like(f), torch.empty_like(f)
    for n in (1, G - 1, G, G + 1, sms, sms + 1, plan.P - 3):
        bz.bz_collide_terms(plan, 3, 3 + n, f, q)
        bz.bz_collide_terms(ref, 3, 3 + n, f, r)
        assert torch.equal(q, r) if n < G else float((q - r).abs().max() / r.abs().max()) <= 1e-5, n
    plan.close()
    ref.close()


@pytest.mark.parametrize("conv", [0, 1])
def test_padded_and_rk4(conv):
    import paper_2004_11239_gb300 as bz
    n = 16 if conv else 32
    plans = [bz.bz_plan_create_ex(n, L, R, 0.0, 0.5, 3, 8, conv=conv, cluster=c) for c in (0, 8)]
    f = torch.from_numpy(bi.random_mixture(n, L, seed=2)).cuda()
    out = []
    for p in plans:
        q, x = torch.empty_like(f), f.clone()
        bz.bz_collide(p, f, q)
        if not conv:
            bz.bz_step_rk(p, x, 0.0, 0.05, 2)
        out.append((q, x))
        p.close()
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
