"""Cell coverage for every number of warps a cell can get (1 up to 3^3 points,
2 for 4^3, 4 for 5^3, 8 beyond), cells inside, across and outside the range of
the FP32 bounds, against the oracle."""
import numpy as np
import pytest
import torch

from paper_2605_01919_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sub", [2, 4, 5, 6])
def test_counts(sub, orc):
    from paper_2605_01919_gb300 import gfs as G
    G.load()
    w = W.union_grid(N=10, up=2, tau=1)
    cells = np.random.default_rng(sub).integers(-6, 16, (120, 3)).astype(np.int32)
    ctx = G.Context(tau=1)
    ctx.build(torch.from_numpy(w.p).cuda(), torch.from_numpy(w.s).cuda())
    got = ctx.cell_coverage(torch.from_numpy(cells).cuda(), [-1.0, -1.0, -1.0], w.h, sub).cpu().numpy()
    ctx.close()
    want = orc.cell_coverage(w.p, w.s, cells, [-1.0, -1.0, -1.0], w.h, sub)
    assert 0 < want.sum() < len(cells) * sub ** 3
    assert np.array_equal(got.astype(np.uint32), want)
