"""Fewer query points than samples: packets of close points, the rest point by
point.  The results are those of small calls, which take every point alone."""
import numpy as np
import pytest
import torch

from paper_2605_01919_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [24575, 24576, 24583, 131071, 131072, 131091])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_mixed_sparse_points(m, dtype):
    """Clusters, a slice, repeated points, samples, points outside the box and
    scattered ones in one call, below and above the sizes from which packets
    of 8 and 16 are tried (140,608 samples)."""
    from paper_2605_01919_gb300 import gfs as G
    G.load()
    w = W.union_grid(N=52, tau=1)
    rng = np.random.default_rng(m)
    k = m // 8
    parts = [rng.normal(0.2, 0.01, (2 * k, 3)), rng.normal(-0.4, 0.03, (k, 3)), np.tile(rng.uniform(-1, 1, (1, 3)), (k, 1)),
             w.p[rng.integers(0, w.n, k)], rng.uniform(-1, 1, (k, 3)) * np.array([1, 1, 0]) + np.array([0, 0, 0.1]),
             rng.uniform(-1.2, 1.2, (64, 3))]
    rest = m - sum(len(p) for p in parts)
    x = rng.permutation(np.concatenate(parts + [rng.uniform(-1, 1, (rest, 3))]))
    x = torch.from_numpy(x).to(dtype).cuda()
    ctx = G.Context(tau=1)
    ctx.build(torch.from_numpy(w.p).cuda(), torch.from_numpy(w.s).cuda())
    whole = ctx.query(x)
    alone = [ctx.query(x[i:i + 20000]) for i in range(0, m, 20000)]
    ctx.close()
    assert torch.equal(whole["s64"].view(torch.int64), torch.cat([o["s64"] for o in alone]).view(torch.int64))
    for key in ("argmin", "flags"):
        assert torch.equal(whole[key], torch.cat([o[key] for o in alone])), key
