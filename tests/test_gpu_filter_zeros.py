"""A filter B that is zero at single spectral samples: A gives exactly zero there, whatever
the neighbouring samples hold, and the others are the oracle's to 1e-5."""
import numpy as np
import pytest

from oracle import isam_oracle as O
from paper_1905_06058_gb300 import inputs as I
from test_gpu_calibration import torch   # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [dict(nx=L, nk=32, nz=32) for L in (32, 64, 192, 512, 1024)] +
                         [dict(nx=64, ny=8, nk=32, nz=32), dict(nx=64, nk=32, nz=64)],
                         ids=lambda k: "x".join(str(v) for v in k.values()))
def test_zero_samples(torch, kw):   # noqa: F811
    from paper_1905_06058_gb300.isam import Plan
    g = I.small_bscan(seed=77, **kw).geom
    filt = np.ones(((g.ny // 2 + 1) if g.ny > 1 else 1, g.nx // 2 + 1, g.nk), np.complex128)
    filt[..., [0, 7, 12, 31]] = 0.0
    filt[..., [6, 13]] = 1e3
    op = O.IsamOracle(g, "nufft", filt=filt)
    eta = I.random_image(op.image_shape, 13)
    plan = Plan(g)
    plan.set_filter(filt)
    s = plan.forward(torch.from_numpy(eta.astype(np.complex64)).cuda()).cpu().numpy()
    plan.close()
    assert not np.any(s[..., [0, 7, 12, 31]])
    ref = op.forward(eta)
    assert np.linalg.norm(s - ref) <= 1e-5 * np.linalg.norm(ref)
