"""Half a million points and more on few samples, packets of 32: the results
of small calls, which take every point alone."""
import numpy as np
import pytest
import torch

from paper_2605_01919_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n, m", [(1, 524289), (100, 524287), (100, 524300), (1024, 524288), (1025, 524288)])
def test_dense_points(n, m):
    from paper_2605_01919_gb300 import gfs as G
    G.load()
    p, s = W.tiny_random(n, n)
    x = torch.from_numpy(np.random.default_rng(m).uniform(-1.05, 1.05, (m, 3))).cuda()
    ctx = G.Context(tau=2)
    ctx.build(torch.from_numpy(p).cuda(), torch.from_numpy(s).cuda())
    whole = ctx.query(x)
    alone = [ctx.query(x[i:i + 24000]) for i in range(0, m, 24000)]
    ctx.close()
    assert torch.equal(whole["s64"].view(torch.int64), torch.cat([o["s64"] for o in alone]).view(torch.int64))
    for key in ("argmin", "flags"):
        assert torch.equal(whole[key], torch.cat([o[key] for o in alone])), key
