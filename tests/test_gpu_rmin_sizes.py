"""The exact radius of many points at once equals that of the same points in
small calls, on both sides of the number of points from which a point gets
fewer warps (1,024)."""
import numpy as np
import pytest
import torch

from paper_2605_01919_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [1024, 1025, 1300])
def test_radius_does_not_depend_on_the_call(m):
    from paper_2605_01919_gb300 import gfs as G
    G.load()
    w = W.union_grid(N=8, tau=1)
    ctx = G.Context(tau=1)
    ctx.build(torch.from_numpy(w.p).cuda(), torch.from_numpy(w.s).cuda())
    rng = np.random.default_rng(m)
    x = torch.from_numpy(rng.uniform(-1, 1, (m, 3))).cuda()
    sigma = torch.from_numpy(rng.integers(-1, 2, m).astype(np.int8)).cuda()
    whole = ctx.exact_rmin(x, sigma)
    parts = torch.cat([ctx.exact_rmin(x[k:k + 100], sigma[k:k + 100]) for k in range(0, m, 100)])
    ctx.close()
    assert torch.isfinite(whole).any() and torch.equal(whole.view(torch.int64), parts.view(torch.int64))
