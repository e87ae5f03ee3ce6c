"""The arithmetic of h = IFFT(fhat): double-float by default, FP64 where BZ_H_FP64 asks for it (FP32 stores both).

The default has to round as FP64 does: a stored value can differ only where some 45 bits leave its rounding open, by one
FP32 ulp of a few values, far below 2^-24 of max |Q|; with low parts lost every value would be off by about
1e-7 max |h|, which moves Q by some 1e-6 on data that the grid does not resolve.  And FP64 has to be FP64: a sum of
1 + 2^-24 + 2^-52 lies above the middle between two FP32 numbers in 53 bits and on it in 47."""
import numpy as np
import pytest

import bz_inputs as bi

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
L = 10.0
FORMS = [(3, 8, 0), (3, 16, 0), (3, 16, 1), (3, 24, 0), (3, 32, 0), (3, 32, 1), (2, 8, 0), (2, 16, 0), (2, 32, 0), (2, 64, 0)]


def _collides(dim, N, data, f):
    import paper_2004_11239_gb300 as bz
    out = []
    for h in (bz.BZ_H_AUTO, bz.BZ_H_FP64):
        if dim == 2:
            plan = bz.bz_plan_create_ex(N, L, bi.R_from_L(L), 0.0, 0.0, 2, 12, kernel=bz.BZ_KERNEL_B2, dim=2, h_precision=h)
        else:
            plan = bz.bz_plan_create_ex(N, L, bi.R_from_L(L), 0.0, 0.5, 2, 12, data=data, h_precision=h)
        q = torch.empty_like(f)
        bz.bz_collide(plan, f, q)
        out.append(q)
        plan.close()
    return out


@pytest.mark.parametrize("dim,N,data", FORMS)
@pytest.mark.parametrize("dtype", [torch.complex64, torch.complex128])
def test_default_rounds_as_fp64(dim, N, data, dtype):
    if dim == 3:
        f = bi.random_mixture(N, L, seed=63)
    else:
        rng = np.random.default_rng(63)
        f = (rng.standard_normal((N, N)) + 1j * rng.standard_normal((N, N))) * 10.0 ** rng.uniform(-9, 0, (N, N))
    q, ref = _collides(dim, N, data, torch.from_numpy(f).cuda().to(dtype))
    assert float((q - ref).abs().max() / ref.abs().max()) <= 2.0 ** -24


@pytest.mark.parametrize("dim,N,data", FORMS)
def test_fp64_is_fp64(dim, N, data):
    f = np.zeros((N,) * dim, complex)
    eps = 2.0 ** -24 + 2.0 ** -52
    f[(0,) * dim] = 1.0
    if data:                                   # Hermitian: the two modes add up to eps where their phase is 1
        f[(1,) + (0,) * (dim - 1)] = f[(N - 1,) + (0,) * (dim - 1)] = eps / 2
    else:
        f[(1,) + (0,) * (dim - 1)] = eps
    q, ref = _collides(dim, N, data, torch.from_numpy(f).cuda())
    assert not torch.equal(q, ref)


@pytest.mark.parametrize("dtype", [torch.complex64, torch.complex128])
def test_fp32_h_of_real_data(dtype):
    """BZ_H_FP32 of real data at N = 32 takes the launches of the other arithmetics (h and the kernel's inputs in two) and
    stays within 2.5e-5 of max |Q| of them on data that the grid does not resolve."""
    import paper_2004_11239_gb300 as bz
    f = torch.from_numpy(bi.random_mixture(32, L, seed=63)).cuda().to(dtype)
    out = []
    for h in (bz.BZ_H_AUTO, bz.BZ_H_FP32):
        plan = bz.bz_plan_create_ex(32, L, bi.R_from_L(L), -1.0, 0.5, 2, 12, data=bz.BZ_DATA_REAL, h_precision=h)
        q = torch.empty_like(f)
        bz.bz_collide(plan, f, q)
        assert bz.bz_plan_last_launches(plan) == 4
        out.append(q)
        plan.close()
    err = float((out[0] - out[1]).abs().max() / out[0].abs().max())
    assert 0 < err <= 2.5e-5, err


@pytest.mark.parametrize("data", [0, 1])
@pytest.mark.parametrize("dtype", [torch.complex64, torch.complex128])
def test_fp64_on_one_sm_kernels_and_batches(data, dtype):
    """At N = 32 with enough terms for k_cube32 (its layouts of fhat and h), and of two slots of a batch."""
    import paper_2004_11239_gb300 as bz
    f = torch.stack([torch.from_numpy(bi.random_mixture(32, L, seed=s)) for s in (63, 64, 65)]).cuda().to(dtype)
    out = []
    for h in (bz.BZ_H_AUTO, bz.BZ_H_FP64):
        plan = bz.bz_plan_create_ex(32, L, bi.R_from_L(L), 0.0, 0.5, 4, 12, data=data, h_precision=h)
        one, q = torch.empty_like(f[0]), torch.zeros_like(f)
        bz.bz_collide(plan, f[0].clone(), one)
        batch = bz.bz_batch_create(plan, 3, 0)
        bz.bz_batch_collide(batch, [2, 0], f, q)
        batch.close()
        plan.close()
        out.append((one, q))
    for a, b in zip(*out):
        assert float((a - b).abs().max() / b.abs().max()) <= 2.0 ** -24
    assert not out[1][1][1].any() and out[1][1][2].any()
    assert float((out[1][0] - out[1][1][0]).abs().max() / out[1][0].abs().max()) <= 1e-6
