"""The rounding of the fused kernels' transforms, seen through whole collides: the mean over six inputs of the relative
2-norm error against 64 bits.  Radix-4 decimation in frequency gives the first figure, radix 2 with its
differences as 2a - (a + wb) the second; the bound is between them."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("N,N_rho,M,gamma,s,R,real,radix4,radix2", [
    (16, 32, 32, 0.0, 0.5, 6.0, False, 1.77e-7, 1.98e-7),
    (16, 32, 32, 0.0, 0.5, 6.0, True, 1.75e-7, 1.95e-7),
    (24, 24, 12, -1.0, 0.25, 9.0616, False, 2.87e-7, 3.36e-7),
])
def test_error_of_collides(N, N_rho, M, gamma, s, R, real, radix4, radix2):
    from perf import cases
    case = dict(kind="collide", N=N, N_rho=N_rho, M=M, gamma=gamma, s=s, R=R, real=real)
    total = 0.0
    for seed in range(1, 7):
        state = cases.prepare(case, seed)
        q = cases.run(state).to(torch.complex128)
        ref = cases.exact(case, seed)
        total += float((q - ref).norm() / ref.norm())
        state["plan"].close()
    print(f"N={N} real={real}: {total / 6:.3e}")
    assert total / 6 <= (radix4 * radix2) ** 0.5
