"""Candidates that mostly survive: small spheres apart from one another, whose
open candidates walk together (many groups), one by one (few groups) or in one
pair of launches (few tiles), against the oracle."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def samples(n, kind, seed):
    rng = np.random.default_rng(seed)
    p = rng.uniform(-0.98, 0.98, (n, 3))
    s = {"apart": rng.uniform(-0.01, 0.01, n), "touching": rng.uniform(-0.12, 0.12, n), "zero": np.zeros(n),
         "one place": np.full(n, 0.2)}[kind]
    if kind == "apart":
        s[:: 9] = 0.3                    # some cover many of the others
    if kind == "one place":
        p[:] = p[0]
    return p, s


# 47 x 630 = 29,610 groups of tile and direction at most: more than the 4,864
# warps; 13 x 150 fewer; 64 spheres are the most without levels
@pytest.mark.parametrize("n, tau", [(1500, 3), (400, 2), (65, 3), (64, 3), (40, 4), (1, 3)])
@pytest.mark.parametrize("kind", ["apart", "touching", "zero", "one place"])
@pytest.mark.parametrize("box", [True, False])
def test_survivors_match_oracle(orc, n, tau, kind, box):
    from paper_2605_01919_gb300 import gfs as G
    G.load()
    p, s = samples(n, kind, n + tau)
    U = orc.icosphere(tau)
    want = orc.collect(p, s, U, orc.keep_all(p, s, U, box_cull=box))[0]
    ctx = G.Context(tau=tau, box_cull=box)
    pt, st = torch.from_numpy(p).cuda(), torch.from_numpy(s).cuda()
    ctx.build(pt, st)
    assert np.array_equal(ctx.survivors().cpu().numpy(), want)
    x = torch.zeros((1, 3), dtype=torch.float64, device="cuda")
    ctx.batch_build([{"p": pt, "s": st, "x": x}] * 2)
    for k in range(2):
        assert np.array_equal(ctx.batch_survivors(k).cpu().numpy(), want)
    ctx.close()
