"""Packets of the batched query, 16 points each, or 32 where the points are very
many for the samples, at their edges: equal to the single-shape results."""
import numpy as np
import pytest
import torch

from paper_2605_01919_gb300 import workloads as W

pytestmark = pytest.mark.gpu


# points per sample below and above 128 in all
@pytest.mark.parametrize("samples, points", [((200, 33, 900), (1, 15, 16, 17, 31, 33, 700)),
                                             ((3, 20, 40), (31, 32, 33, 47, 6000, 12289))])
def test_packets_match_single_shapes(samples, points):
    from paper_2605_01919_gb300 import gfs as G
    G.load()
    rng = np.random.default_rng(len(points))
    shapes = []
    for k, m in enumerate(points):
        p, s = W.tiny_random(samples[k % len(samples)], k)
        x = np.concatenate([p[:1], rng.uniform(-1, 1, (m - 1, 3))])   # a sample among the points
        shapes.append({"p": torch.from_numpy(p).cuda(), "s": torch.from_numpy(s).cuda(), "x": torch.from_numpy(x).cuda()})
    n = sum(t["p"].shape[0] for t in shapes)
    assert (sum(points) >= 128 * n) == (max(points) > 1000)
    ctx, single = G.Context(tau=2), G.Context(tau=2)
    outs = ctx.batch_build(shapes)
    ctx.batch_query()
    torch.cuda.synchronize()
    for o, t in zip(outs, shapes):
        single.build(t["p"], t["s"])
        ref = single.query(t["x"])
        assert torch.equal(o["argmin"], ref["argmin"]) and torch.equal(o["flags"], ref["flags"])
        assert torch.equal(o["s64"].view(torch.int64), ref["s64"].view(torch.int64))
    ctx.close()
    single.close()
