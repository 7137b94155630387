"""A captured batch keeps working while the context serves other calls."""
import numpy as np
import pytest
import torch

from paper_2605_01919_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tau", [1, 3])
def test_graph_replay_after_a_larger_single_shape(tau):
    """The graph of a batch rebuild and query, captured and replayed after a
    single shape with more samples, candidates, points and survivors than the
    batch went through the same context (every shared workspace would have
    grown): the replay gives the batch's results again, and the single
    shape's results do not change by it either."""
    from paper_2605_01919_gb300 import gfs as G
    G.load()
    rng = np.random.default_rng(3)
    shapes = []
    for n, m in ((33, 40), (700, 513)):
        p, s = W.tiny_random(n, n)
        shapes.append({"p": torch.from_numpy(p).cuda(), "s": torch.from_numpy(s).cuda(),
                       "x": torch.from_numpy(rng.uniform(-0.6, 0.6, (m, 3))).cuda()})
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        ctx = G.Context(tau=tau, stream=side)
        outs = ctx.batch_build(shapes)
        ctx.batch_rebuild()
        ctx.batch_query()
        side.synchronize()
        want = [{k: o[k].clone() for k in ("s64", "argmin", "flags")} for o in outs]
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side):
            ctx.batch_rebuild()
            ctx.batch_query()
        big = W.union_grid(N=24, tau=tau)
        x = torch.from_numpy(rng.uniform(-1, 1, (200000, 3))).cuda()
        ctx.build(torch.from_numpy(big.p).cuda(), torch.from_numpy(big.s).cuda())
        first = {k: v.clone() for k, v in ctx.query(x).items()}
        filler = torch.full((1 << 26,), 0x55, dtype=torch.uint8, device="cuda")  # over what was freed, if anything
        for o in outs:
            o["s64"].fill_(7.0)
            o["argmin"].fill_(-7)
        graph.replay()
        side.synchronize()
        assert ctx.batch_status() == 0
        for o, w in zip(outs, want):
            assert torch.equal(o["s64"].view(torch.int64), w["s64"].view(torch.int64))
            assert torch.equal(o["argmin"], w["argmin"]) and torch.equal(o["flags"], w["flags"])
        again = ctx.query(x)
        side.synchronize()
        for k in ("argmin", "flags"):
            assert torch.equal(again[k], first[k])
        assert torch.equal(again["s64"].view(torch.int64), first["s64"].view(torch.int64))
        assert int(filler[0]) == 0x55
        ctx.close()
