"""The stop rule at check intervals around the host's lag of three iterations, and at the
end of a solve: a solve that stops at check k returns bit for bit what a solve with the
same checks that ends at k returns, at its first check, a later one, and one in the last
iterations; then the same plan solves on without stopping."""
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


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("every", [1, 2, 3, 4, 5])
def test_stop_at_interval(torch, every, prec):
    from paper_1905_06058_gb300.isam import Plan
    wl = I.small_bscan(nx=64, nk=64, nz=64, n_points=6, seed=23)
    s = O.IsamOracle(wl.geom, "nufft").forward(wl.eta)
    plan = Plan(wl.geom, precision=prec)
    sd = torch.from_numpy(s.astype(np.float32 if prec == "fp32" else np.float64)).cuda()
    kw = dict(lambda_rel=0.05, L=4.0, check_every=every)
    last = 4 * every
    ends = {k: plan.solve(sd, max_iter=k, tol=1e-300, **kw) for k in range(every, last + 1, every)}
    for k in (every, 2 * every, last):
        tol = ends[k][1]["rr"] * 1.0001
        first = min(j for j in ends if ends[j][1]["rr"] < tol)   # r_r need not fall steadily
        for max_iter in (first, first + 1, first + 2, first + 40):
            z, info = plan.solve(sd, max_iter=max_iter, tol=tol, **kw)
            assert info["iterations"] == first and info["rr"] == ends[first][1]["rr"]
            assert torch.equal(z, ends[first][0])
    z, info = plan.solve(sd, max_iter=last, tol=1e-300, **kw)
    assert info["iterations"] == last and torch.equal(z, ends[last][0])
    plan.close()
