"""The lateral passes that keep their tile in registers, at every length they take
(FP32: 64 to 1024, 2^p and 3 * 2^p; FP64: 64 to 512, 2^p), along x and along y of a
volume.

A and A^H go through the complex, real-input and real-output passes and are
compared with the oracle (1e-5 relative L2, the bar of test_gpu_operator.py).
The passes of the solve (update from u_hat with depth weights, update with the
norm partials of the stop rule, gradient step and extrapolation of the other
priors) are compared with the radix-8 shared-memory form of the same plan, which
is the same arithmetic in another order: 1e-5 on the image as in
test_gpu_autotune.py, and 1e-3 on r_r, the bar of test_gpu_stop_rule.py.  FP64:
1e-10 (test_gpu_operator.py) for all of them."""
import numpy as np
import pytest

from oracle import isam_oracle as O
from paper_1905_06058_gb300 import inputs as I

pytestmark = pytest.mark.gpu

LENGTHS = [64, 128, 192, 256, 384, 512, 768, 1024]


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


def shape(L, along_y):
    # 16 depth samples: one tile of 16 columns or two of 8; y: 2 x 16 columns
    return dict(nx=2, ny=L, nk=16, nz=16) if along_y else dict(nx=L, nk=16, nz=32)


@pytest.mark.parametrize("along_y", [False, True], ids=["x", "y"])
@pytest.mark.parametrize("L", LENGTHS)
def test_operators(torch, L, along_y):
    from paper_1905_06058_gb300.isam import Plan
    g = I.small_bscan(seed=60, **shape(L, along_y)).geom
    ref = O.IsamOracle(g, "nufft")
    eta = I.random_image(ref.image_shape, 61).astype(np.complex64)
    y = I.random_spectra(ref.spec_shape, 62).astype(np.float32)
    plan = Plan(g)
    a = plan.forward(torch.from_numpy(eta).cuda()).cpu().numpy()
    b = plan.adjoint(torch.from_numpy(y).cuda()).cpu().numpy()
    plan.close()
    assert rel(a, ref.forward(eta.astype(np.complex128))) < 1e-5
    assert rel(b, ref.adjoint(y.astype(np.float64))) < 1e-5


@pytest.mark.parametrize("along_y", [False, True], ids=["x", "y"])
@pytest.mark.parametrize("L", LENGTHS)
def test_solve_passes_match_radix8(torch, L, along_y):
    from paper_1905_06058_gb300.isam import Plan
    g = I.small_bscan(seed=63, **shape(L, along_y)).geom
    plan = Plan(g)
    s = plan.forward(torch.from_numpy(I.random_image(plan.image_shape, 64).astype(np.complex64)).cuda())
    w = torch.from_numpy(I.depth_weights(plan.image_shape[2]).astype(np.float32)).cuda()
    kws = [dict(max_iter=6, w=w), dict(max_iter=6, w=w, tol=1e-300, check_every=3),
           dict(max_iter=3, prior="haar_depth")]
    for kw in kws:
        got = []
        for r in (16, 8):
            plan.set_tuning(lateral_radix=r)
            out, info = plan.solve(s, lambda_rel=0.02, L=4.0, **kw)
            got.append((out.cpu().numpy(), info["rr"]))
        assert rel(got[0][0], got[1][0]) < 1e-5
        assert got[0][1] == pytest.approx(got[1][1], rel=1e-3)
    plan.close()


@pytest.mark.parametrize("along_y", [False, True], ids=["x", "y"])
@pytest.mark.parametrize("L", [64, 128, 256, 512])
def test_fp64(torch, L, along_y):
    from paper_1905_06058_gb300.isam import Plan
    g = I.small_bscan(seed=65, **shape(L, along_y)).geom
    ref = O.IsamOracle(g, "nufft")
    eta = I.random_image(ref.image_shape, 66)
    y = I.random_spectra(ref.spec_shape, 67)
    plan = Plan(g, precision="fp64")
    s = plan.forward(torch.from_numpy(eta).cuda())
    assert rel(s.cpu().numpy(), ref.forward(eta)) < 1e-10
    assert rel(plan.adjoint(torch.from_numpy(y).cuda()).cpu().numpy(), ref.adjoint(y)) < 1e-10
    w = torch.from_numpy(I.depth_weights(plan.image_shape[2])).cuda()
    for kw in (dict(max_iter=5, w=w), dict(max_iter=5, w=w, tol=1e-300, check_every=2),
               dict(max_iter=3, prior="haar_depth")):
        got = []
        for r in (16, 8):
            plan.set_tuning(lateral_radix=r)
            out, info = plan.solve(s, lambda_rel=0.02, L=4.0, **kw)
            got.append((out.cpu().numpy(), info["rr"]))
        assert rel(got[0][0], got[1][0]) < 1e-10
        assert got[0][1] == pytest.approx(got[1][1], rel=1e-10)
    plan.close()


@pytest.mark.parametrize("kw", [dict(nx=L, nk=nk, nz=64) for L in LENGTHS for nk in (32, 64)] +
                         [dict(nx=64, ny=ny, nk=32, nz=32) for ny in (2, 4, 24, 64)] +
                         [dict(nx=192, ny=2, nk=64, nz=64)],
                         ids=lambda k: "x".join(str(v) for v in k.values()))
def test_half_spectra(torch, kw):
    """A and A^H of FP32 plans whose x passes keep half of the Hermitian spectra, with
    columns paired across y at x = 0 and nx/2, against the oracle and the radix-8 form,
    which keeps them whole."""
    from paper_1905_06058_gb300.isam import Plan
    g = I.small_bscan(seed=68, **kw).geom
    ref = O.IsamOracle(g, "nufft")
    eta = I.random_image(ref.image_shape, 69).astype(np.complex64)
    y = I.random_spectra(ref.spec_shape, 70).astype(np.float32)
    plan = Plan(g)
    for r in (16, 8):
        plan.set_tuning(lateral_radix=r)
        a = plan.forward(torch.from_numpy(eta).cuda()).cpu().numpy()
        b = plan.adjoint(torch.from_numpy(y).cuda()).cpu().numpy()
        assert rel(a, ref.forward(eta.astype(np.complex128))) < 1e-5
        assert rel(b, ref.adjoint(y.astype(np.float64))) < 1e-5
    plan.set_tuning(lateral_radix=16)                    # real arrays off the 8-byte grid
    buf = torch.zeros(2 * (y.size + 1), dtype=torch.float32, device="cuda")
    odd = buf[1:1 + y.size].view(y.shape)
    out = buf[y.size + 1 | 1:][:y.size].view(y.shape)
    odd.copy_(torch.from_numpy(y))
    assert rel(plan.adjoint(odd).cpu().numpy(), b) < 2e-5
    plan.forward(torch.from_numpy(eta).cuda(), out=out)
    assert rel(out.cpu().numpy(), a) < 2e-5
    plan.close()
