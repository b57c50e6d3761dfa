"""Small graphs with a vertex of more than 1,024 out-edges (needs a GB300): the
one-launch solve leaves them to the general path once it has checked row_ptr,
which is then not checked again.  Results, errors and the launches they cost."""
import numpy as np
import pytest
import torch

import oracle
from paper_1111_0627_gb300.ocm import OCM_FLAG_EVAL_GLOBAL

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_1111_0627_gb300 as ocm


def _hub(n, extra, seed):
    rng = np.random.default_rng(seed)
    deg = np.full(n, 3)
    deg[n // 2] += extra
    rp = np.zeros(n + 1, np.int32)
    rp[1:] = np.cumsum(deg)
    col = rng.integers(0, n, int(rp[-1])).astype(np.int32)
    col[rp[:-1]] = (np.arange(n) + 1) % n
    return rp, col, rng.integers(-1000, 1000, col.shape[0]).astype(np.int32)


@pytest.mark.parametrize("n,extra", [(1, 2000), (400, 1021), (400, 1022), (3000, 5000), (16_000, 90_000)])
def test_small_hubs(n, extra):
    rp, col, w = _hub(n, extra, n + extra)
    h = oracle.howard(rp, col, w, "max")
    d = [torch.from_numpy(x).cuda() for x in (rp, col, w)]
    s = ocm.solve(*d, "max", certificate=True)
    r = ocm.solve(*d, "max", certificate=True, flags=OCM_FLAG_EVAL_GLOBAL)
    assert (s.num, s.den, s.stats["iterations"]) == (h.num, h.den, h.iterations)
    assert s.cycle.cpu().tolist() == h.cycle.tolist() == r.cycle.cpu().tolist()
    assert (s.potential.cpu().numpy() == h.V).all()
    assert s.stats["launches"] <= r.stats["launches"]   # (never more than without the one-launch solve)


def test_errors_beside_a_hub():
    rp, col, w = _hub(500, 2000, 1)
    d = [torch.from_numpy(x).cuda() for x in (rp, col, w)]

    def status(rp=d[0], col=d[1], w=d[2], **kw):
        with pytest.raises(ocm.OCMError) as e:
            ocm.solve(rp, col, w, "max", **kw)
        return e.value.status

    bad = d[0].clone()
    bad[3] = bad[4]
    assert status(rp=bad) == -3          # a vertex without an out-edge
    bad = d[0].clone()
    bad[7] = bad[9] + 1
    assert status(rp=bad) == -2          # row_ptr decreases
    bad = d[1].clone()
    bad[11] = 500
    assert status(col=bad) == -2         # a target out of range
    bad = d[2].clone()
    bad[5] = -2**31
    assert status(w=bad) == -4
    init = d[0][:-1].clone()
    init[6] = d[0][7]
    assert status(init_policy=init) == -1
    assert status(max_iters=1) == -5
