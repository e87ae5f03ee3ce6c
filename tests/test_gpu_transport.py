"""Free streaming (bz_transport_x) at every pairing of line lengths that takes another path."""
import numpy as np
import pytest

from oracle import inhom

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def bz():
    import paper_2004_11239_gb300 as m
    return m


@pytest.mark.parametrize("N,nx", [(8, 8), (8, 32), (16, 24), (24, 8), (24, 24), (32, 16), (32, 32)])
@pytest.mark.parametrize("dtype", ["c128", "c64"])
def test_streaming_every_line_length(bz, N, nx, dtype):
    """Every pairing of line lengths' code paths (fewer and more cells than modes), both signs of t, against the
    FP64 oracle: FP64 cells to 1e-13 of max |f| (eight transforms' roundings), complex64 cells to the
    rounding of the result, 2^-24 a component (1e-7 allowed)."""
    L, Lx, t = 6.62, 4.0, -0.37
    rng = np.random.default_rng(N * nx)
    f = rng.standard_normal((nx, N, N, N)) + 1j * rng.standard_normal((nx, N, N, N))
    if dtype == "c64":
        f = f.astype(np.complex64)
    fd = torch.from_numpy(f).cuda()
    bz.bz_transport_x(N, L, nx, Lx, fd, t)
    ref = inhom.transport(f.astype(np.complex128), L, Lx, t)
    err = np.max(np.abs(fd.cpu().numpy() - ref)) / np.max(np.abs(ref))
    assert err <= (1e-13 if dtype == "c128" else 1e-7), err
