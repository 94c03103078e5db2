"""The FP64 soft threshold, bit for bit: z = u max(1 - tau / sqrt(x x + y y), 0) with the
correctly rounded root and division and x x + y y rounded once after y y, in the lateral
passes in registers and in shared memory.  u is the first iterate at a threshold that
rounds away, and the threshold's arithmetic is repeated in exact fractions and numpy."""
from fractions import Fraction

import numpy as np
import pytest

from paper_1905_06058_gb300 import inputs as I
from test_gpu_calibration import torch   # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx", [8, 64])
def test_bits(torch, nx):   # noqa: F811
    from paper_1905_06058_gb300.isam import Plan
    g = I.small_bscan(seed=76, nx=nx, nk=64, nz=64).geom
    plan = Plan(g, precision="fp64")
    s = torch.from_numpy(I.random_spectra(plan.spec_shape, 12)).cuda()
    first = lambda lam: plan.solve(s, lambda_abs=lam, L=4.0, max_iter=1)[0].cpu().numpy().ravel()
    u = first(1e-300)
    tau = 0.6 * np.median(np.abs(u))
    z = first(4.0 * tau)
    plan.close()
    yy = u.imag * u.imag
    m2 = np.array([float(Fraction(x) * Fraction(x) + Fraction(b))
                   for x, b in zip(u.real.tolist(), yy.tolist())])
    f = np.maximum(1.0 - tau / np.sqrt(m2), 0.0)
    assert 0.1 < np.mean(f > 0.0) < 0.95
    assert np.array_equal(z.real, u.real * f) and np.array_equal(z.imag, u.imag * f)
