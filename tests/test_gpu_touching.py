"""Exact coverage of exactly touching samples, pinned bit for bit on the GPU.

On grids of distance samples the spheres touch within rounding, and the ball
that the coverage walk meets first decides which of them a certificate keeps:
the uncovered circles and points and the witnesses depend on the centres of
the hierarchy's nodes.  The digests are those of the centres by 23 IEEE steps
(the numbers of circles beside them: with 12 fast steps the first two lists
had 11,084 and 30,585 circles); a change of the hierarchy that moves them
changes results."""
import hashlib

import numpy as np
import pytest
import torch

from paper_2605_01919_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def digest(t):
    return hashlib.sha1(np.ascontiguousarray(t.cpu().numpy()).tobytes()).hexdigest()[:12]


@pytest.mark.parametrize("grid, N, circles, points, lists, coverage", [
    ("csg", 16, 11085, 18247, ("6bb18785b8cf", "0d514bd0c826", "0c3ac2ed8996"), ("0ec7cdd5434c", "f14c44bc36a3")),
    ("union", 16, 30586, 593729, ("1cfab1321041", "0f79f079b3f6", "c42c540a9d9a"), ("0c7f2cbe5e40", "1387bccb86f4")),
    # (2.9M pairs: every lane of the circle search has one)
    ("csg", 24, 49417, 1685021, ("f792cae76e8f", "b2da4f6d11a8", "75ef16f4960b"), ("54650f2dd649", "866c685d9764")),
    ("csg", 32, 48132, 153279, ("218993a25b2e", "03aa1ad48930", "92ba1e3d76d5"), ("7f647172e673", "4a76ac9a6682")),
])
def test_touching_lists_and_witnesses(grid, N, circles, points, lists, coverage):
    from paper_2605_01919_gb300 import gfs as G
    G.load()
    w = {"csg": W.csg_pseudo_grid, "union": W.union_grid}[grid](N=N, tau=2)
    ctx = G.Context(tau=2)
    ctx.build(torch.from_numpy(w.p).cuda(), torch.from_numpy(w.s).cuda())
    circ, quads, pts, status = ctx.uncovered_intersections()
    state, witness = ctx.sphere_uncovered(witness=True)
    ctx.close()
    assert status == 0 and (len(circ), len(quads)) == (circles, points)
    assert (digest(circ), digest(quads), digest(pts)) == lists
    assert (digest(state), digest(witness)) == coverage
