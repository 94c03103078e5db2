"""Plans under an allocator with a budget: arrays that a call can do without (the FP64
coefficient table) give way, and the results are those of plenty of memory (1e-13: the
coefficients are the same polynomials, tabulated or evaluated)."""
import numpy as np
import pytest

from paper_1905_06058_gb300 import inputs as I
from test_gpu_calibration import torch   # noqa: F401

pytestmark = pytest.mark.gpu


class Pool:
    """Device memory for plans: `budget` bytes at once, no block of a size in `refused`."""

    def __init__(self, torch):   # noqa: F811
        from paper_1905_06058_gb300 import isam as B
        self.torch, self.B = torch, B
        self.live, self.budget, self.refused = {}, 1 << 40, ()

    def alloc(self, n):
        if n in self.refused or sum(self.live.values()) + n > self.budget:
            return 0
        p = self.torch.cuda.caching_allocator_alloc(n)
        self.live[p] = n
        return p

    def free(self, p):
        self.live.pop(p)
        self.torch.cuda.caching_allocator_delete(p)

    def __enter__(self):
        self.B.set_allocator(self.alloc, self.free)
        return self

    def __exit__(self, *_):
        self.B.set_allocator()

    def held(self):
        return sum(self.live.values())


NX, NK, J = 32, 64, 6
COEF = (NX // 2 + 1) * NK * J // 2 * 16        # bytes of the table: 8 J a class sample


def solve(plan, s):
    return plan.solve(s, lambda_rel=0.01, L=4.0, max_iter=5)[0]


def test_no_coefficient_table(torch):   # noqa: F811
    from paper_1905_06058_gb300.isam import Plan
    g = I.small_bscan(seed=73, nx=NX, nk=NK).geom
    ref = Plan(g, precision="fp64", J=J)
    s = torch.from_numpy(I.random_spectra(ref.spec_shape, 8)).cuda()
    z = solve(ref, s)
    L = Plan(g, J=J).lipschitz(20, 1e-30)
    ref.close()
    with Pool(torch) as pool:
        whole = Plan(g, precision="fp64", J=J)
        assert COEF in pool.live.values()
        whole.close()
        pool.refused = (COEF,)
        plan = Plan(g, precision="fp64", J=J)
        got = solve(plan, s)
        fp32 = Plan(g, J=J)
        L2 = fp32.lipschitz(20, 1e-30)
        plan.close()
        fp32.close()
        assert not pool.live
    assert float((got - z).norm()) <= 1e-13 * float(z.norm())
    assert L2 == pytest.approx(L, rel=1e-13)


def test_coefficient_table_gives_way(torch):   # noqa: F811
    from paper_1905_06058_gb300.isam import Plan
    g = I.small_bscan(seed=73, nx=NX, nk=NK).geom
    with Pool(torch) as pool:
        ref = Plan(g, precision="fp64", J=J)
        s = torch.from_numpy(I.random_spectra(ref.spec_shape, 8)).cuda()
        z = solve(ref, s)
        most = pool.held()
        ref.close()
        plan = Plan(g, precision="fp64", J=J)
        pool.budget = most - COEF
        got = solve(plan, s)
        assert COEF not in pool.live.values()
        plan.set_model(g.disp, g.z0)            # rebuilds the tables, without room for it
        again = solve(plan, s)
        plan.close()
        assert not pool.live
    assert float((got - z).norm()) <= 1e-13 * float(z.norm())
    assert float((again - z).norm()) <= 1e-13 * float(z.norm())


@pytest.mark.parametrize("addback", [False, True])
def test_tv_without_its_sixth_image(torch, addback):   # noqa: F811
    """FP32 with nk < nz: the two-launch steps in place of the tiles'.  Both round each
    step's arithmetic to 32 bits; 60 steps of rounding 1.2e-7 at |p| <= 1: 1e-5."""
    from paper_1905_06058_gb300.isam import Batch, Plan
    g = I.small_bscan(seed=74, nx=NX, nk=NK, nz=2 * NK).geom
    with Pool(torch) as pool:
        ref = Plan(g)
        s = torch.from_numpy(I.random_spectra(ref.spec_shape, 9).astype(np.float32)).cuda()
        kw = dict(lambda_rel=0.05, L=4.0, max_iter=3, prior="tv", addback=addback)
        z = ref.solve(s, **kw)[0]
        most = pool.held()
        ref.close()
        plan = Plan(g)
        pool.budget = most - z.numel() * z.element_size()
        got = plan.solve(s, **kw)[0]
        again = plan.solve(s, **kw)[0]
        plan.close()
        pool.budget = 1 << 40
        plan = Plan(g)
        pool.refused = (6 * z.numel() * z.element_size(),)
        out = torch.empty_like(z)
        batch = Batch([(plan, s, out, kw)])
        batch.run()
        batch.close()
        plan.close()
        assert not pool.live
    assert float((got - z).norm()) <= 1e-5 * float(z.norm())
    assert torch.equal(got, again)
    assert torch.equal(got, out)


def test_power_iteration_gives_a_large_table_back(torch):   # noqa: F811
    """An FP32 plan holds a table of more than 64 MB while it iterates for L, not after."""
    from paper_1905_06058_gb300.isam import Plan
    g = I.small_bscan(seed=75, nx=64, ny=64, nk=1024).geom
    coef = 33 * 33 * 1024 * 8 * 8
    with Pool(torch) as pool:
        plan = Plan(g, J=8)
        plan.lipschitz(2, 1e-30)                 # FP64 state and its workspace
        kept = pool.held()
        assert coef not in pool.live.values()
        seen = []
        alloc = pool.alloc
        pool.B.set_allocator(lambda n: (seen.append(n), alloc(n))[1], pool.free)
        plan.lipschitz(2, 1e-30)
        assert seen == [coef] and pool.held() == kept
        plan.close()
        assert not pool.live
