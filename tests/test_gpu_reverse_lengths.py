"""The reverse pass's kernels over the lengths of their forms, against the oracle: the
parameter sums of every spectral length (64, 256 and 512 threads a block, whole and part
loads), with columns whose band is partly or wholly evanescent, and the pointwise kernels
at images that end inside a block's first and second half.  Bars as
test_gpu_calibration.py: 1e-5 (FP32) and 1e-10 (FP64) of sum |D||F y||S_x| for the sums,
1e-3 and 1e-7 for the unrolled gradient."""
import numpy as np
import pytest

from oracle import isam_oracle as O
from paper_1905_06058_gb300 import inputs as I
from test_gpu_calibration import dev, grad_bound, torch, types   # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,tol", [("fp32", 1e-5), ("fp64", 1e-10)])
@pytest.mark.parametrize("dx", [1.0, 0.08])
@pytest.mark.parametrize("nk", [16, 32, 64, 128, 256, 512, 1024, 2048])
def test_param_sums(torch, prec, tol, dx, nk):   # noqa: F811
    from paper_1905_06058_gb300.isam import Plan
    g = I.small_bscan(seed=22, nx=8, nk=nk, nz=nk, dx_scale=dx).geom
    op = O.IsamOracle(g, "nufft")
    x, y = I.random_image(op.image_shape, 4), I.random_spectra(op.spec_shape, 5)
    ct, rt = types(prec)
    plan = Plan(g, precision=prec)
    got = plan.param_grad(dev(torch, x, ct), dev(torch, y, rt))
    plan.close()
    assert np.all(np.abs(got - O.param_grad(op, x, y)) <= tol * grad_bound(op, x, y))


@pytest.mark.parametrize("prec,tol", [("fp32", 1e-3), ("fp64", 1e-7)])
@pytest.mark.parametrize("kw", [dict(nx=1, nk=16, nz=16), dict(nx=2, nk=32, nz=32),
                                dict(nx=24, nk=64, nz=64), dict(nx=48, nk=16, nz=64)],
                         ids=lambda k: f"{k['nx']}x{k['nz']}")
def test_unrolled_gradient(torch, prec, tol, kw):   # noqa: F811
    from paper_1905_06058_gb300.isam import Plan
    wl = I.small_bscan(seed=23, **kw)
    op = O.IsamOracle(wl.geom, "nufft")
    s = op.forward(wl.eta)
    zbar = I.random_image(op.image_shape, 6)
    w = I.depth_weights(wl.geom.nz)
    lam, L, K = 0.02 * np.abs(op.adjoint(s)).max(), 1.2, 5
    ref = O.fista_unrolled_vjp(op, s, lam, L, K, zbar, w=w[None, None, :])
    ct, rt = types(prec)
    plan = Plan(wl.geom, precision=prec)
    sd, wd = dev(torch, s, rt), dev(torch, w, rt)
    _, ck = plan.fista_unrolled(sd, lam, L, K, 2, w=wd)
    g, sb = plan.fista_unrolled_vjp(sd, lam, L, K, 2, ck, dev(torch, zbar, ct),
                                    want_s_bar=True, w=wd)
    plan.close()
    assert np.linalg.norm(g - ref.theta_bar) <= tol * np.linalg.norm(ref.theta_bar)
    assert np.linalg.norm(sb.cpu().numpy() - ref.s_bar) <= tol * np.linalg.norm(ref.s_bar)
