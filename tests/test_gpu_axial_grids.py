"""The FP32 axial kernels of runtime lengths (K <= 1024) on both sides of their two register
counts: grids that one round of blocks holds at 96 registers a thread, and larger ones
(4,660 columns' pairs at K <= 256, 2,080 at K = 512, 546 at K = 1024 by the radix-8 passes),
with windows, residue classes (dx_scale 0.4: steps past 2.3 bins) and nz > nk.  The
operators against the oracle and a solve against the FP64 plan's: 1e-5, the bar of the
operators' parity tests."""
import numpy as np
import pytest

from oracle import isam_oracle as O
from paper_1905_06058_gb300 import inputs as I
from test_gpu_calibration import torch   # noqa: F401

pytestmark = pytest.mark.gpu


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("dx", [1.0, 0.4])
@pytest.mark.parametrize("nx,ny,nk,nz,radix", [(24, 16, 64, 64, 16), (96, 96, 32, 32, 16),
                                               (96, 96, 64, 128, 16), (64, 64, 256, 256, 16),
                                               (32, 24, 256, 256, 16), (64, 16, 512, 512, 8),
                                               (64, 32, 512, 512, 8)])
def test_grids(torch, nx, ny, nk, nz, radix, dx):   # noqa: F811
    from paper_1905_06058_gb300.isam import Plan
    g = I.small_bscan(seed=75, nx=nx, ny=ny, nk=nk, nz=nz, dx_scale=dx).geom
    op = O.IsamOracle(g, "nufft")
    x, y = I.random_image(op.image_shape, 10), I.random_spectra(op.spec_shape, 11)
    plan, wide = Plan(g), Plan(g, precision="fp64")
    plan.set_tuning(axial_radix=radix)
    xd = torch.from_numpy(x.astype(np.complex64)).cuda()
    yd = torch.from_numpy(y.astype(np.float32)).cuda()
    assert rel(plan.forward(xd).cpu().numpy(), op.forward(x)) < 1e-5
    assert rel(plan.adjoint(yd).cpu().numpy(), op.adjoint(y)) < 1e-5
    kw = dict(lambda_abs=1.0, L=8.0, max_iter=3)
    z = plan.solve(yd, **kw)[0].cpu().numpy()
    z64 = wide.solve(yd.double(), **kw)[0].cpu().numpy()
    plan.close()
    wide.close()
    assert rel(z, z64) < 1e-5
