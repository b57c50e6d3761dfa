"""The walks of the one-level evaluation (needs a GB300), started by a given
policy whose shape reaches each of their branches: cycles around the sizes at
which a walk looks for one (32 steps) and gives up (256 steps), chains that a
few vertices or most of them are too deep to walk (the jump rounds take those,
or everything), many cycles at once, and trees that pass new roots.  Value,
critical cycle, iteration count and the final values must be the oracle's,
for the mean and for the cycle ratio; all comparisons are exact."""
import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_1111_0627_gb300 as ocm


def _chain(n, length, cycle):
    """Everything points at one cycle except a chain of the given length."""
    to = np.arange(n) % cycle
    to[:cycle] = (np.arange(cycle) + 1) % cycle
    a = np.arange(cycle, cycle + length)
    to[a] = np.where(a + 1 < cycle + length, a + 1, 0)
    return to


def _cycles(n, size):
    v = np.arange(n)
    start = v - v % size
    return np.minimum(start + (v - start + 1) % size, n - 1)


SHAPES = {
    **{f"ring_{k}": (lambda k=k: (np.arange(k) + 1) % k)
       for k in (1, 2, 31, 32, 33, 64, 255, 256, 257, 513, 1500)},
    "chain_40": lambda: _chain(3000, 40, 3),
    "chain_300": lambda: _chain(3000, 300, 1),       # a few walks give up
    "chain_2000": lambda: _chain(2500, 2000, 5),     # nearly all do
    "pairs": lambda: _cycles(4001, 2),               # more than 1,024 cycles
    "cycles_50": lambda: _cycles(20_000, 50),
    "tree": lambda: np.maximum(np.arange(30_000) // 2, 0),
    "tree_cycle": lambda: np.where(np.arange(50_000) < 37, (np.arange(50_000) + 1) % 37,
                                   np.arange(50_000) // 3),
}


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("ratio", [False, True], ids=["mean", "ratio"])
def test_given_policies_follow_the_oracle(shape, ratio):
    rng = np.random.default_rng(20_011 + len(shape))
    to = SHAPES[shape]().astype(np.int32)
    n = to.shape[0]
    name = rng.permutation(n).astype(np.int32)       # roots anywhere in the vertex order
    succ = np.empty(n, np.int32)
    succ[name] = name[to]
    col = np.empty(2 * n, np.int32)
    col[0::2] = rng.integers(0, n, n)
    col[1::2] = succ                                  # the start policy: the second edge
    rp = (2 * np.arange(n + 1)).astype(np.int32)
    w = rng.integers(-1000, 1001, 2 * n).astype(np.int32)
    t = rng.integers(1, 9, 2 * n).astype(np.int32) if ratio else None
    init = (2 * np.arange(n) + 1).astype(np.int32)
    g = synth.Graph(rp, col, w, "max", shape)
    h = oracle.howard(rp, col, w, "max", init_policy=init, transit=t)
    d = [torch.from_numpy(x).cuda() for x in (rp, col, w, init)]
    s = ocm.solve(*d[:3], "max", init_policy=d[3], certificate=True,
                  transit=None if t is None else torch.from_numpy(t).cuda())
    assert (s.num, s.den) == (h.num, h.den)
    assert s.cycle.cpu().tolist() == h.cycle.tolist()
    assert s.stats["iterations"] == h.iterations
    rc, bad = oracle.certificate(g.row_ptr, g.col_idx, g.w, g.mode, s.eta_num.cpu().numpy(),
                                 s.eta_den.cpu().numpy(), s.potential.cpu().numpy(), s.num, s.den,
                                 s.cycle.cpu().numpy(), transit=t)
    assert rc == 0, (rc, bad)
