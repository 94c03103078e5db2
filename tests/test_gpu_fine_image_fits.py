"""Fits with more image than spectral samples in depth (nz > nk): their loss and gradient are
what rounding leaves of nearly equal numbers, so they follow the order of every sum before
them, and the library keeps that order.  The values in golden/fine_image_fits.txt (a line a
case: its sizes, the loss, the five derivatives) are those of the shared-memory transforms
and residue-class sums that the library had first.

Bar: every 32-bit rounding is the same, so only the sums in 64 bits could differ, by
1e-16 times the number of their terms (below 1e6) and times the gradient's cancellation (the
moments reach 1e-3 of their terms): 1e-7."""
import os

import numpy as np
import pytest

from paper_1905_06058_gb300 import inputs as I
from test_gpu_calibration import torch   # noqa: F401

pytestmark = pytest.mark.gpu
GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "fine_image_fits.txt")

# lateral lengths of both column-split transforms (256, 1024), of radix 8 at fixed (512) and
# other lengths, with a factor of 3 and along y; K = 64 to 4096
CASES = [(128, 1, 256, 512, 8), (256, 1, 512, 1024, 6), (192, 1, 256, 512, 4),
         (512, 1, 64, 128, 6), (1024, 1, 128, 256, 6), (64, 1, 1024, 2048, 6),
         (96, 1, 16, 32, 6), (24, 16, 64, 128, 6), (16, 256, 32, 64, 8)]


def spectra(shape):
    """Whole numbers in [-2048, 2047] from a linear congruential generator."""
    x, out = 12345, np.empty(int(np.prod(shape)), np.float32)
    for i in range(out.size):
        x = (1103515245 * x + 12345) % (1 << 31)
        out[i] = (x >> 16) % 4096 - 2048
    return out.reshape(shape)


def fit(torch, nx, ny, nk, nz, J):   # noqa: F811
    """Loss and gradient (per unit step of an optimiser) of 16 unrolled iterations."""
    from paper_1905_06058_gb300 import calib
    from paper_1905_06058_gb300.isam import Plan
    g = I.Geometry(nx, ny, nk, nz, 4.65e6, 5.03e6, 2.0e-6, 2.0e-6 if ny > 1 else 0.0, 0.1, 4.0e-4,
                   (0.0, 5e-10, -8e-16, 0.0))
    plan = Plan(g, J=J)
    s = torch.from_numpy(spectra(plan.spec_shape)).cuda()
    lam = 1e-6 * plan.max_abs(plan.adjoint(s))
    theta = torch.tensor(list(g.disp) + [g.z0], dtype=torch.float64, requires_grad=True)
    loss = calib.data_fidelity(s, theta, plan, lam, 2.5, 16, 5)
    loss.backward()
    plan.close()
    return [float(loss.detach())] + (theta.grad.numpy() * calib.theta_scales(g)).tolist()


def golden():
    with open(GOLDEN) as f:
        rows = [line.split() for line in f if not line.startswith("#")]
    return {tuple(int(v) for v in r[:5]): [float(v) for v in r[5:]] for r in rows}


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_fit_keeps_its_values(torch, case):   # noqa: F811
    got, ref = np.array(fit(torch, *case)), np.array(golden()[case])
    assert abs(got[0] - ref[0]) <= 1e-7 * abs(ref[0])
    assert np.linalg.norm(got[1:] - ref[1:]) <= 1e-7 * np.linalg.norm(ref[1:])


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_model_is_the_fits_operator(torch, case):   # noqa: F811
    """A z of calib.model is the one whose residual the data term is of, bit for bit, and
    isam_forward's to rounding (1e-6 of its norm)."""
    from paper_1905_06058_gb300 import calib
    from paper_1905_06058_gb300.isam import Plan
    nx, ny, nk, nz, J = case
    g = I.Geometry(nx, ny, nk, nz, 4.65e6, 5.03e6, 2.0e-6, 2.0e-6 if ny > 1 else 0.0, 0.1, 4.0e-4,
                   (0.0, 5e-10, -8e-16, 0.0))
    plan = Plan(g, J=J)
    s = torch.from_numpy(spectra(plan.spec_shape)).cuda()
    z = plan.adjoint(s)
    theta = torch.tensor(list(g.disp) + [g.z0], dtype=torch.float64)
    a = calib.model(z, theta, plan)
    _, r = plan.data_fidelity(z, s)
    f = plan.forward(z)
    plan.close()
    assert torch.equal(a - s, r)
    assert float((a - f).norm()) <= 1e-6 * float(f.norm())
