"""complex64 input whose address is a multiple of 4 but not of 8 (an odd offset into an array of floats), through the C
ABI: the same result as from an aligned copy, on every pipeline."""
import ctypes

import pytest

import bz_inputs as bi

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
L = 10.0


@pytest.mark.parametrize("N,kw", [(16, dict(pipeline=2)), (48, {}), (48, dict(data=1)), (16, dict(h_precision=2)), (16, {}),
                                  (16, dict(data=1)), (32, {}), (32, dict(data=1)), (24, {}), (32, dict(precision=1)),
                                  (16, dict(dim=2, kernel=4))])
def test_odd_address(N, kw):
    import paper_2004_11239_gb300 as bz
    plan = bz.bz_plan_create_ex(N, L, bi.R_from_L(L), 0.0, 0.0 if kw.get("dim") else 0.5, 4, 12, **kw)
    f = torch.from_numpy(bi.random_mixture(N, L, seed=5)).cuda().to(torch.complex64)
    if kw.get("dim"):
        f = f[0].contiguous()
    flat = torch.view_as_real(f).reshape(-1)
    odd = torch.zeros(flat.numel() + 2, dtype=torch.float32, device="cuda")
    odd[1:-1] = flat
    q, r = torch.empty_like(f), torch.empty_like(f)
    bz.bz_collide(plan, f, q)
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert odd.data_ptr() % 8 == 0
    status = bz.lib.bz_collide(plan.handle, ctypes.c_void_p(odd.data_ptr() + 4), ctypes.c_void_p(r.data_ptr()),
                               bz.BZ_C64, stream)
    assert status == 0
    assert torch.equal(q, r)
    plan.close()
