"""The circle search with few and with many pairs per warp, on the GPU."""
import numpy as np
import pytest
import torch

from paper_2605_01919_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("copies", [2, 3])
def test_far_copies_change_nothing(copies):
    """A copy of the samples far away cuts no sphere of the first one and holds
    none of its points, so the first copy's circles and points stay the same
    bit for bit, while the pairs grow past the number (2^18) from which a warp
    takes four of them (171k pairs a copy)."""
    from paper_2605_01919_gb300 import gfs as G
    G.load()
    w = W.union_grid(N=12, tau=1)

    def lists(p, s):
        ctx = G.Context(tau=1)
        ctx.build(torch.from_numpy(np.ascontiguousarray(p)).cuda(), torch.from_numpy(np.ascontiguousarray(s)).cuda())
        circ, quads, pts, status = ctx.uncovered_intersections()
        ctx.close()
        assert status == 0
        return circ.cpu().numpy(), quads.cpu().numpy(), pts.cpu().numpy()

    c0, q0, t0 = lists(w.p, w.s)
    p = np.concatenate([w.p + np.array([16.0 * k, 0, 0]) for k in range(copies)])
    c1, q1, t1 = lists(p, np.tile(w.s, copies))
    n = len(w.s)
    in_c, in_q = c1[:, 1] < n, q1[:, 2] < n
    assert len(c0) > 0 and len(q0) > 0 and len(c1) > len(c0)
    assert np.array_equal(c1[in_c], c0) and np.array_equal(q1[in_q], q0) and np.array_equal(t1[in_q], t0)
