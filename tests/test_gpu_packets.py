"""The query's packets of neighbouring points at their edges: point counts on
both sides of the size where packets begin, a last packet that is not full,
packets whose points lie far apart, points on samples and outside the box --
against the oracle, bit for bit."""
import numpy as np
import pytest
import torch

from paper_2605_01919_gb300 import workloads as W

pytestmark = pytest.mark.gpu

PACKET_MIN = 131072


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2605_01919_gb300 import gfs
    gfs.load()
    return gfs


def _points(m, p, seed):
    """Uniform points, tight clusters (near ties, small packets), two far
    corners, points outside the box and points on samples."""
    rng = np.random.default_rng(seed)
    x = rng.uniform(-1, 1, (m, 3))
    k = m // 4
    c = rng.uniform(-0.6, 0.6, (7, 3))
    x[:k] = c[rng.integers(0, 7, k)] + rng.normal(0, 1e-4, (k, 3))
    x[k:k + k // 8] = np.where(rng.random((k // 8, 1)) < 0.5, -1.0, 1.0)
    x[k + k // 8:k + k // 4] *= 1.7
    j = min(m // 16, p.shape[0])
    if j:
        x[-j:] = p[:j]
    return x[rng.permutation(m)]


@pytest.mark.parametrize("m", [1, 31, 33, 24575, 24579, PACKET_MIN - 1, PACKET_MIN, PACKET_MIN + 5])
@pytest.mark.parametrize("case", ["valid", "mixed", "single"])
@pytest.mark.parametrize("fp32", [False, True])
def test_packets_match_oracle(G, orc, m, case, fp32):
    tau = 1
    if case == "valid":
        w = W.sphere_grid(N=6, up=1, tau=tau)
        p, s = w.p, w.s
    elif case == "mixed":
        p, s = W.tiny_random(90, 5, valid=False)
        s[:4] = 0.0
    else:
        p, s = np.array([[0.1, -0.2, 0.3]]), np.array([0.4])
    x = _points(m, p, 17 + m)
    if fp32:
        x = x.astype(np.float32)
    U = orc.icosphere(tau)
    surv = orc.collect(p, s, U, orc.keep_all(p, s, U))
    val, arg, fl, _ = orc.query(p, s, surv, x.astype(np.float64))
    ctx = G.Context(tau=tau)
    ctx.build(torch.from_numpy(p).cuda(), torch.from_numpy(s).cuda())
    out = ctx.query(torch.from_numpy(x).cuda())
    assert np.array_equal(out["flags"].cpu().numpy().astype(np.int32) & 0xFFFF, fl)
    assert np.array_equal(out["argmin"].cpu().numpy(), arg)
    assert np.array_equal(out["s64"].cpu().numpy(), val, equal_nan=True)
    ctx.close()
