"""Single graphs whose edges stay near their source, yet not near enough for the
two-level evaluation (needs a GB300): policies hundreds of steps deep, which the
one-level evaluation takes by jump rounds without trying to walk, and the
smaller fraction of such edges at which it walks.  Cold and warm starts, exact
comparison with the oracle."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_1111_0627_gb300 as ocm


@pytest.mark.parametrize("spread", [300, 1100, 1700, 4000])
def test_local_graphs(spread):
    n = 270_001                     # (ranges of 1,777 vertices)
    rng = np.random.default_rng(spread)
    deg = rng.choice([3, 5], n)
    rp = np.zeros(n + 1, np.int32)
    rp[1:] = np.cumsum(deg)
    m = int(rp[-1])
    src = np.repeat(np.arange(n), deg)
    off = 1 + np.floor(np.abs(rng.normal(0, spread, m))).astype(np.int64)
    off[rp[:-1]] = 1
    col = ((src + off) % n).astype(np.int32)
    w = rng.integers(-1000, 1001, m).astype(np.int32)
    d = [torch.from_numpy(x).cuda() for x in (rp, col, w)]
    h = oracle.howard(rp, col, w, "min")
    s = ocm.solve(*d, "min", certificate=True)
    assert (s.num, s.den, s.stats["iterations"]) == (h.num, h.den, h.iterations)
    assert s.cycle.cpu().tolist() == h.cycle.tolist()
    assert (s.potential.cpu().numpy() == h.V).all()
    w2 = w.copy()
    k = rng.integers(0, m, m // 64)
    w2[k] = rng.integers(-1000, 1001, k.size)
    h2 = oracle.howard(rp, col, w2, "min", init_policy=s.policy.cpu().numpy())
    s2 = ocm.solve(d[0], d[1], torch.from_numpy(w2).cuda(), "min", init_policy=s.policy,
                   certificate=True)
    assert (s2.num, s2.den, s2.stats["iterations"]) == (h2.num, h2.den, h2.iterations)
    assert s2.cycle.cpu().tolist() == h2.cycle.tolist()
    assert (s2.potential.cpu().numpy() == h2.V).all()
