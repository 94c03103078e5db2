"""The window form of the axial kernels' interpolation and scatter against the
oracle, at the edges of the geometries that take it.

A plan takes it when no column is evanescent and the Stolt positions of
neighbouring samples lie less than 2.3 bins apart (dp/dj = 4 kappa / p, largest
at k_min and the largest |q|); otherwise, and in a block whose positions round
out of the windows, the residue-class scatter runs.  Covered: steps of 2 (all
windows alike), 2.2, just below and just above the bound, and evanescent
columns; a column at q = 0 whose positions all sit within rounding of an
integer; the smallest and largest blocks, nk < nz (bins no window reaches) and
nk = nz (windows past one period); every J, both precisions, with and without
the Stolt table.  Bars as in test_gpu_operator.py: 1e-5 (FP32) and 1e-10 (FP64)
relative L2 per application.

At an integer position the J neighbours change, and with them the result, by
up to twice the min-max design's worst-case error (5e-6 at J = 6): there the
oracle itself moves by that much when its positions move by 1e-9 bins, so the
integer geometries get that on top, and the others have 2 k_min / dk at 0.37 of
a bin (the band's own value makes it an integer for every nk)."""
import dataclasses
import math

import numpy as np
import pytest

from oracle import isam_oracle as O
from paper_1905_06058_gb300 import inputs as I

pytestmark = pytest.mark.gpu

TOL = {"fp32": 1e-5, "fp64": 1e-10}


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


def geometry(nx, nk, nz, step, integer=False):
    """A B-scan whose widest step between positions is `step` bins (None: some
    columns evanescent); integer: 2 k_min / dk an integer, so that every position
    of the q = 0 column is one."""
    g = I.small_bscan(nx=nx, nk=nk, nz=nz, seed=50).geom
    dk = (g.k_max - g.k_min) / (nk - 1)
    k_min = (round(2 * g.k_min / dk) + (0.0 if integer else 0.37)) * dk / 2
    g = dataclasses.replace(g, k_min=k_min, k_max=k_min + dk * (nk - 1))
    if step is None:
        dx = math.pi / (2.1 * g.k_min)
    elif step == 2.0:
        dx = 1.0                                    # q / 2k < 1e-6
    else:
        dx = math.pi / (2 * g.k_min * math.sqrt(1 - 4 / step ** 2))
    return dataclasses.replace(g, dx=dx)


def check(torch, g, prec, J, table, more=0.0):
    from paper_1905_06058_gb300.isam import Plan
    ref = O.IsamOracle(g, "nufft", J=J)
    rng = np.random.default_rng(51)
    real, cplx = (np.float64, np.complex128) if prec == "fp64" else (np.float32, np.complex64)
    eta = (rng.standard_normal(ref.image_shape) + 1j * rng.standard_normal(ref.image_shape)).astype(cplx)
    y = rng.standard_normal(ref.spec_shape).astype(real)
    plan = Plan(g, precision=prec, J=J, stolt_table=table)
    a = plan.forward(torch.from_numpy(eta).cuda()).cpu().numpy()
    b = plan.adjoint(torch.from_numpy(y).cuda()).cpu().numpy()
    plan.close()
    assert rel(a, ref.forward(eta.astype(np.complex128))) < TOL[prec] + more
    assert rel(b, ref.adjoint(y.astype(np.float64))) < TOL[prec] + more


@pytest.mark.parametrize("step", [2.0, 2.2, 2.299, 2.301, None], ids=str)
@pytest.mark.parametrize("nk,nz,J", [(16, 16, 4), (16, 16, 8), (64, 128, 6), (256, 256, 6),
                                     (512, 512, 8), (512, 512, 6), (256, 512, 4), (256, 256, 8),
                                     (1024, 1024, 4), (512, 1024, 6),
                                     (2048, 2048, 8)])
def test_steps_fp32(torch, nk, nz, J, step):
    check(torch, geometry(8, nk, nz, step), "fp32", J, True)


@pytest.mark.parametrize("table", [True, False], ids=["table", "evaluated"])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("nk,nz", [(32, 32), (128, 256), (1024, 1024)])
def test_integer_positions(torch, nk, nz, prec, table):
    check(torch, geometry(4, nk, nz, 2.1, integer=True), prec, 6, table, more=2 * 5e-6)


@pytest.mark.parametrize("step", [2.0, 2.299, 2.301, None], ids=str)
@pytest.mark.parametrize("nk,nz,J,table", [(16, 32, 8, False), (256, 256, 6, True),
                                           (1024, 1024, 4, False), (2048, 2048, 6, True)])
def test_steps_fp64(torch, nk, nz, J, table, step):
    check(torch, geometry(8, nk, nz, step), "fp64", J, table)


@pytest.mark.parametrize("integer", [False, True], ids=["", "integer"])
@pytest.mark.parametrize("step", [2.0, 2.299, 2.301, None], ids=str)
@pytest.mark.parametrize("nk,nz,J", [(16, 512, 6), (64, 512, 4), (512, 512, 8), (32, 1024, 6),
                                     (1024, 1024, 4), (1024, 1024, 6), (16, 2048, 8),
                                     (2048, 2048, 6)])
def test_gradient(torch, nk, nz, J, step, integer):
    """The fused kernel where it keeps taps in tensor memory (K = 1024 to 4096), down to
    a few lanes of one warp with samples, through two linear FISTA iterations
    (lambda = 0; A and A^H twice each, so four times the bar, and at integer
    positions four times the jump)."""
    from paper_1905_06058_gb300.isam import Plan
    if integer and J != 6:
        pytest.skip("one J is enough")
    g = geometry(4, nk, nz, step, integer)
    ref = O.IsamOracle(g, "nufft", J=J)
    s = np.random.default_rng(52).standard_normal(ref.spec_shape).astype(np.float32)
    res = O.fista(ref.forward, ref.adjoint, s.astype(np.float64), 0.0, 4.0, max_iter=2,
                  shape=ref.image_shape)
    for table in (True, False):
        plan = Plan(g, J=J, stolt_table=table)
        out, _ = plan.solve(torch.from_numpy(s).cuda(), lambda_rel=0.0, L=4.0, max_iter=2)
        plan.close()
        assert rel(out.cpu().numpy(), res.eta) < 4e-5 + (4 * 2 * 5e-6 if integer else 0.0)
