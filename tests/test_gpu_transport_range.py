"""Free streaming of complex64 cells over FP32's range: the sums over a line are taken in numbers of FP32's exponents,
so the kernel scales by a power of two and results of scaled cells are the scaled results, to the bit."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("N,nx", [(8, 8), (16, 32), (24, 24), (32, 16), (32, 32)])
@pytest.mark.parametrize("k", [124, -90])
def test_scaled_cells(N, nx, k):
    import paper_2004_11239_gb300 as bz
    g = torch.Generator().manual_seed(N * nx)
    f = torch.randn((nx, N, N, N, 2), generator=g).clamp(-4, 4)      # sums of 2^124 of them leave FP32, results do not
    out = []
    for s in (1.0, 2.0 ** k):
        c = torch.view_as_complex((f * s).contiguous()).cuda()
        bz.bz_transport_x(N, 6.62, nx, 4.0, c, 0.37)
        out.append(torch.view_as_real(c).double() / s)
    assert torch.isfinite(out[0]).all()
    # results that are below FP32's smallest normal number once scaled have lost bits
    m = out[0].abs() * 2.0 ** k >= 2.0 ** -126
    assert m.float().mean() > 0.99 and torch.equal(out[0][m], out[1][m])
