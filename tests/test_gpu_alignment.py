"""The operators on arrays that start at any element: real arrays off the 8-byte (FP64 16-byte)
grid and images off the 16-byte (32-byte) one, in every form of the lateral passes and with
nz = nk and nz > nk, against the same call on aligned arrays.  The arithmetic is the same
where the form is (whole and half spectra differ by rounding): 2e-6 and 1e-14 of the
largest value."""
import numpy as np
import pytest

from paper_1905_06058_gb300 import inputs as I
from test_gpu_calibration import torch   # noqa: F401

pytestmark = pytest.mark.gpu


def off_grid(torch, shape, dtype):   # noqa: F811
    """A contiguous tensor that starts one element after an allocation."""
    n = int(np.prod(shape))
    t = torch.zeros(n + 1, dtype=dtype, device="cuda")[1:].view(shape)
    assert t.is_contiguous() and t.data_ptr() % 512 == t.element_size()
    return t


@pytest.mark.parametrize("prec,tol", [("fp32", 2e-6), ("fp64", 1e-14)])
@pytest.mark.parametrize("nx,ny", [(2, 1), (24, 1), (64, 1), (256, 1), (1024, 1), (1536, 1), (24, 8),
                                   (64, 24)])
@pytest.mark.parametrize("nk,nz", [(32, 32), (32, 64)])
def test_operators_at_any_element(torch, prec, tol, nx, ny, nk, nz):   # noqa: F811
    from paper_1905_06058_gb300.isam import Plan
    g = I.small_bscan(seed=71, nx=nx, ny=ny, nk=nk, nz=nz).geom
    plan = Plan(g, precision=prec)
    x = torch.from_numpy(I.random_image(plan.image_shape, 5)).cuda().to(plan.cplx_dtype)
    y = torch.from_numpy(I.random_spectra(plan.spec_shape, 6)).cuda().to(plan.real_dtype)
    a, b = plan.forward(x), plan.adjoint(y)
    x1, y1 = off_grid(torch, x.shape, x.dtype), off_grid(torch, y.shape, y.dtype)
    a1, b1 = off_grid(torch, y.shape, y.dtype), off_grid(torch, x.shape, x.dtype)
    x1.copy_(x)
    y1.copy_(y)
    plan.forward(x1, out=a1)
    plan.adjoint(y1, out=b1)
    plan.close()
    assert float((a1 - a).abs().max()) <= tol * float(a.abs().max())
    assert float((b1 - b).abs().max()) <= tol * float(b.abs().max())


@pytest.mark.parametrize("prec,tol", [("fp32", 2e-6), ("fp64", 1e-14)])
def test_residual_at_any_element(torch, prec, tol):   # noqa: F811
    from paper_1905_06058_gb300.isam import Plan
    plan = Plan(I.small_bscan(seed=78, nx=32, nk=64).geom, precision=prec)
    x = torch.from_numpy(I.random_image(plan.image_shape, 5)).cuda().to(plan.cplx_dtype)
    y = torch.from_numpy(I.random_spectra(plan.spec_shape, 6)).cuda().to(plan.real_dtype)
    v, r = plan.data_fidelity(x, y)
    y1, r1 = off_grid(torch, y.shape, y.dtype), off_grid(torch, y.shape, y.dtype)
    y1.copy_(y)
    v1, _ = plan.data_fidelity(x, y1, r_out=r1)
    plan.close()
    assert v1 == pytest.approx(v, rel=tol)
    assert float((r1 - r).abs().max()) <= tol * float(r.abs().max())
