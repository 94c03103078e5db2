"""TV solves at a lambda so small that the dual's |q| = |grad w| / (8 tau) squared is beyond the
plan's largest number.  z lies within 8 tau of u (|p| <= 1, four terms of two parts), so
the image is that of lambda = 0 to rounding: 1e-6 (FP32), 1e-14 (FP64) of its norm."""
import numpy as np
import pytest

from paper_1905_06058_gb300 import inputs as I
from test_gpu_calibration import torch   # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,lam,tol", [("fp32", 1e-20, 1e-6), ("fp32", 1e-24, 1e-6),
                                          ("fp64", 1e-170, 1e-14)])
@pytest.mark.parametrize("iters,steps", [(1, 1), (1, 20), (3, 20)])
def test_image_of_no_prior(torch, prec, lam, tol, iters, steps):   # noqa: F811
    from paper_1905_06058_gb300.isam import Plan
    g = I.small_bscan(seed=72, nx=64, nk=64, nz=64).geom
    plan = Plan(g, precision=prec)
    y = torch.from_numpy(1e3 * I.random_spectra(plan.spec_shape, 7)).cuda().to(plan.real_dtype)
    kw = dict(max_iter=iters, L=2.5, prior="tv", prior_iters=steps)
    ref, _ = plan.solve(y, lambda_rel=0.0, **kw)
    got, info = plan.solve(y, lambda_abs=lam, **kw)
    plan.close()
    assert info["status"] == 0
    assert float((got - ref).norm()) <= tol * float(ref.norm())
