"""The kernels that keep an A-scan in registers, the FP32 direct reconstruction and
the Haar prox of nz = 256 to 2048, against the oracle: every length, nk below nz, and
numbers of A-scans that do not fill a block (1, 2 and 24; a block takes up to eight).
Bars: 1e-5 (FP32) and 1e-10 (FP64) relative L2 for the direct reconstruction
(test_gpu_direct.py); two FISTA iterations with the prox apply A and A^H twice each
at those bars apiece, so four times them."""
import numpy as np
import pytest

from oracle import isam_oracle as O
from paper_1905_06058_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as T
    if not T.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    return T


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("nk,nz", [(256, 256), (64, 256), (512, 512), (256, 512), (1024, 1024),
                                   (512, 1024), (2048, 2048), (1024, 2048)])
@pytest.mark.parametrize("nx", [1, 2, 24])
def test_direct(torch, nx, nk, nz):
    from paper_1905_06058_gb300.isam import Plan
    g = I.small_bscan(nx=nx, nk=nk, nz=nz, seed=80).geom
    y = I.random_spectra((1, nx, nk), 81).astype(np.float32)
    plan = Plan(g)
    got = plan.dispersion_compensated_ifft(torch.from_numpy(y).cuda()).cpu().numpy()
    plan.close()
    assert rel(got, O.dispersion_compensated_ifft(g, y.astype(np.float64))) < 1e-5


@pytest.mark.parametrize("prec,tol", [("fp32", 4e-5), ("fp64", 4e-10)])
@pytest.mark.parametrize("nz", [128, 256, 512, 1024, 2048])
@pytest.mark.parametrize("nx", [1, 2, 24])
def test_haar(torch, nx, nz, prec, tol):
    from paper_1905_06058_gb300.isam import Plan
    wl = I.small_bscan(nx=nx, nk=64, nz=nz, seed=82, n_points=6)
    ref = O.IsamOracle(wl.geom, "nufft")
    s = I.add_noise(ref.forward(wl.eta), 30.0, np.random.default_rng(83))
    lam = 0.05 * np.abs(ref.adjoint(s)).max()
    res = O.fista(ref.forward, ref.adjoint, s, lam, 4.0, max_iter=2, shape=ref.image_shape,
                  prox=O.haar_prox)
    plan = Plan(wl.geom, precision=prec)
    sd = torch.from_numpy(s.astype(np.float64 if prec == "fp64" else np.float32)).cuda()
    out, _ = plan.solve(sd, lambda_abs=lam, L=4.0, max_iter=2, prior="haar_depth")
    plan.close()
    assert rel(out.cpu().numpy(), res.eta) < tol
