"""Policies of thousands of cycles on the whole grid (needs a GB300): at, below
and above the number whose roots are settled ahead of the walks, from the
second evaluation on as well as under a warm start.  The graphs are above the
size solved by one team and keep their cycles to the end: small terminal rings
with everything else leading into them.  Value, critical cycle, iteration count
and the certificate are the oracle's, for the mean and the cycle ratio."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_1111_0627_gb300 as ocm


def _terminal(n, K, size, seed):
    rng = np.random.default_rng(seed)
    c = K * size
    deg = np.full(n, 3)
    deg[:c] = 2
    rp = np.zeros(n + 1, np.int32)
    rp[1:] = np.cumsum(deg)
    col = rng.integers(0, n, int(rp[-1]))
    v = np.arange(c)
    base = v - v % size
    col[rp[:c]] = base + (v - base + 1) % size
    col[rp[:c] + 1] = base + rng.integers(0, size, c)
    # (rings anywhere in the vertex order)
    name = rng.permutation(n)
    order = np.argsort(name)
    src = np.repeat(np.arange(n), deg)
    w = rng.integers(0, 1000, col.shape[0])
    e = np.argsort(name[src], kind="stable")
    rp[1:] = np.cumsum(deg[order])
    return rp, name[col[e]].astype(np.int32), w[e].astype(np.int32), rng


@pytest.mark.parametrize("ratio", [False, True], ids=["mean", "ratio"])
@pytest.mark.parametrize("K,size", [(1023, 2), (1025, 3), (8191, 1), (8192, 2), (8193, 2), (15_000, 2)])
def test_terminal_rings(K, size, ratio):
    n = 40_000
    rp, col, w, rng = _terminal(n, K, size, 100 * K + size)
    t = rng.integers(1, 9, w.shape[0]).astype(np.int32) if ratio else None
    d = [torch.from_numpy(x).cuda() for x in (rp, col, w)]
    td = None if t is None else torch.from_numpy(t).cuda()
    starts = [None, (rp[:-1] + rng.integers(0, 2, n)).astype(np.int32)]
    for init in starts:
        h = oracle.howard(rp, col, w, "max", init_policy=init, transit=t)
        s = ocm.solve(*d, "max", init_policy=None if init is None else torch.from_numpy(init).cuda(),
                      transit=td, certificate=True)
        assert s.stats["cycles"] >= min(K, 8000)
        assert (s.num, s.den, s.stats["iterations"]) == (h.num, h.den, h.iterations)
        assert s.cycle.cpu().tolist() == h.cycle.tolist()
        assert (s.potential.cpu().numpy() == h.V).all()
        assert (s.eta_num.cpu().numpy() == h.eta_p).all()
        assert (s.eta_den.cpu().numpy() == h.eta_q).all()
