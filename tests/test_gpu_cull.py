"""The cull's levels and tiles at their edges: icospheres below, at and above
the levels whose covering balls are kept, sphere counts around a 32-sphere
tile, spheres that share a place, zero samples, candidates outside the box --
the survivor set against the oracle's, and the batched cull against both."""
import numpy as np
import pytest
import torch

from paper_2605_01919_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2605_01919_gb300 import gfs
    gfs.load()
    return gfs


def _samples(n, seed, valid):
    p, s = W.tiny_random(n, seed, valid=valid, spread=0.9)
    if n > 8:
        s[3] = 0.0
        p[5], s[5] = p[4], s[4]          # the same sphere twice
        p[7] = p[6]                      # concentric
    return p, s


@pytest.mark.parametrize("tau", [0, 1, 2, 4, 5])
@pytest.mark.parametrize("n", [1, 31, 33, 97])
@pytest.mark.parametrize("valid", [True, False])
@pytest.mark.parametrize("box", [True, False])
def test_survivors_match_oracle(G, orc, tau, n, valid, box):
    p, s = _samples(n, 100 * tau + n, valid)
    U = orc.icosphere(tau)
    want = orc.collect(p, s, U, orc.keep_all(p, s, U, box_cull=box))[0]
    ctx = G.Context(tau=tau, box_cull=box)
    pt, st = torch.from_numpy(p).cuda(), torch.from_numpy(s).cuda()
    ctx.build(pt, st)
    assert np.array_equal(ctx.survivors().cpu().numpy(), want)
    x = torch.zeros((1, 3), dtype=torch.float64, device="cuda")
    p2, s2 = _samples(40, 7, valid)
    ctx.batch_build([{"p": pt, "s": st, "x": x},
                     {"p": torch.from_numpy(p2).cuda(), "s": torch.from_numpy(s2).cuda(), "x": x}])
    ctx.batch_rebuild()
    assert ctx.batch_status() == 0
    assert np.array_equal(ctx.batch_survivors(0).cpu().numpy(), want)
    want2 = orc.collect(p2, s2, U, orc.keep_all(p2, s2, U, box_cull=box))[0]
    assert np.array_equal(ctx.batch_survivors(1).cpu().numpy(), want2)
    ctx.close()
