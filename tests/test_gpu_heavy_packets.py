"""Packets that give up in the middle of a walk, past their limit of work, and go
point by point: the results of small calls, which take every point alone."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def same(a, b):
    for key in ("argmin", "flags"):
        assert torch.equal(a[key], torch.cat([o[key] for o in b])), key
    assert torch.equal(a["s64"].view(torch.int64), torch.cat([o["s64"] for o in b]).view(torch.int64))


@pytest.mark.parametrize("walk", ["spheres", "survivors"])
def test_heavy_packets(walk):
    from paper_2605_01919_gb300 import gfs as G
    G.load()
    rng = np.random.default_rng(4)
    if walk == "spheres":
        # 8,000 nearly concentric spheres of nearly the same radius: no packet
        # of 8 can leave one out (1,700 units of a limit of 640)
        p, s, tau, m = rng.normal(0, 1e-5, (8000, 3)), -0.5 + rng.normal(0, 1e-5, 8000), 0, 24576
        x = rng.uniform(-0.9, 0.9, (m, 3))
    else:
        # points beside the centre of one sphere: its 10,242 survivors are all
        # about as near (7,000 units of a limit of 1,600 for a packet of 16)
        p, s, tau, m = np.array([[0.1, 0.0, -0.1]]), np.array([-0.5]), 5, 131072
        x = p[0] + rng.normal(0, 1e-3, (m, 3))
    ctx = G.Context(tau=tau)
    ctx.build(torch.from_numpy(p).cuda(), torch.from_numpy(s).cuda())
    x = torch.from_numpy(x).cuda()
    whole = ctx.query(x)
    alone = [ctx.query(x[i:i + 24000]) for i in range(0, m, 24000)]
    ctx.close()
    same(whole, alone)
