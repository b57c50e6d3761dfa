"""Deep policies on the whole grid (needs a GB300): walks that publish their
parts, samples that settle the roots of new cycles, and what both leave to the
jump rounds.  The graphs are above the size solved by one team; a given first
policy is deep, or full of cycles the samples miss, and the iterations after it
are too.  Exact comparison with the oracle's value, cycle and iteration count,
and the certificate."""
import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_1111_0627_gb300 as ocm


def _strands(n, depth):
    """Chains of the given length, side by side, into one cycle of 11."""
    v = np.arange(n)
    to = np.where(v < 11, (v + 1) % 11, v - 1)
    to[(v >= 11) & ((v - 11) % depth == 0)] = 3
    return to


def _pairs_and_strands(n, depth):
    """The same with a thousand cycles of two among the chains' ends."""
    to = _strands(n, depth)
    a = n - 2000 + 2 * np.arange(1000)
    to[a], to[a + 1] = a + 1, a
    return to


@pytest.mark.parametrize("make,depth", [(_strands, 40), (_strands, 129), (_strands, 1100),
                                        (_strands, 9000), (_pairs_and_strands, 300)])
@pytest.mark.parametrize("n", [16_385, 70_001])
def test_deep_first_policy(make, depth, n):
    rng = np.random.default_rng(n + depth)
    succ = np.empty(n, np.int32)
    name = rng.permutation(n)
    succ[name] = name[make(n, depth)]
    col = np.empty(3 * n, np.int32)
    col[0::3] = rng.integers(0, n, n)
    col[1::3] = succ
    col[2::3] = rng.integers(0, n, n)
    rp = (3 * np.arange(n + 1)).astype(np.int32)
    # (the policy's edges are good ones: it stays deep while single vertices leave it)
    w = rng.integers(0, 1000, 3 * n).astype(np.int32)
    w[1::3] = rng.integers(700, 1100, n)
    init = (3 * np.arange(n) + 1).astype(np.int32)
    h = oracle.howard(rp, col, w, "max", init_policy=init)
    d = [torch.from_numpy(x).cuda() for x in (rp, col, w, init)]
    s = ocm.solve(*d[:3], "max", init_policy=d[3], certificate=True)
    assert (s.num, s.den, s.stats["iterations"]) == (h.num, h.den, h.iterations)
    assert s.cycle.cpu().tolist() == h.cycle.tolist()
    rc, bad = oracle.certificate(rp, col, w, "max", s.eta_num.cpu().numpy(), s.eta_den.cpu().numpy(),
                                 s.potential.cpu().numpy(), s.num, s.den, s.cycle.cpu().numpy())
    assert rc == 0, (rc, bad)


@pytest.mark.parametrize("seed", range(4))
def test_random_graphs_with_wide_weights(seed):
    g = synth.ring_extra(60_000 + 7 * seed, 0, 7, 0, 1_000_000, seed=500 + seed, tag=3, mode="max")
    h = oracle.howard(g.row_ptr, g.col_idx, g.w, g.mode)
    d = [torch.from_numpy(x).cuda() for x in (g.row_ptr, g.col_idx, g.w)]
    s = ocm.solve(*d, g.mode)
    assert (s.num, s.den, s.stats["iterations"]) == (h.num, h.den, h.iterations)
    assert s.cycle.cpu().tolist() == [int(x) for x in h.cycle]
