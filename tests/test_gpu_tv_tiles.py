"""The FP32 total-variation prox, several dual steps per launch on tiles of 64 x 64
pixels with a halo, against the oracle's steps.

Sizes around a tile's inner extent (52 to 62 pixels, by the number of steps):
images smaller than one tile, of one pixel in x, of just over one and of several
tiles, slices of a volume (whose tiles must not mix), with one, few, exactly five,
just over five and twenty dual steps, so that the last launch of one, two and more
launches is met at every parity.  Three FISTA iterations apply A and A^H three
times each at 1e-5 relative L2 apiece (test_gpu_operator.py), so 1e-4 on the image."""
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


@pytest.mark.parametrize("steps", [1, 4, 5, 6, 11, 20])
@pytest.mark.parametrize("kw", [dict(nx=1, nk=64, nz=64), dict(nx=8, nk=16, nz=16),
                                dict(nx=48, nk=32, nz=64), dict(nx=64, nk=128, nz=128),
                                dict(nx=128, nk=64, nz=64), dict(nx=24, ny=4, nk=64, nz=128)],
                         ids=lambda k: "x".join(str(v) for v in k.values()))
def test_tv_solve(torch, kw, steps):
    from paper_1905_06058_gb300.isam import Plan
    wl = I.small_bscan(n_points=12, seed=70, **kw)
    ref = O.IsamOracle(wl.geom, "nufft")
    s = I.add_noise(ref.forward(wl.eta), 30.0, np.random.default_rng(71))
    lam = 0.05 * np.abs(ref.adjoint(s)).max()
    res = O.fista(ref.forward, ref.adjoint, s, lam, 4.0, max_iter=3, shape=ref.image_shape,
                  prox=O.TVProx(steps))
    plan = Plan(wl.geom)
    y = torch.from_numpy(s.astype(np.float32)).cuda()
    for _ in range(2):                       # the dual starts at 0 in every solve
        out, _ = plan.solve(y, lambda_abs=lam, L=4.0, max_iter=3, prior="tv", prior_iters=steps)
        err = np.linalg.norm(out.cpu().numpy() - res.eta) / np.linalg.norm(res.eta)
        assert err < 1e-4
    plan.close()
