"""Policies too deep to walk, over many iterations that change little (needs a
GB300): the jump rounds keep the values of vertices whose path saw no switch.
The optimum itself is deep, so that the iterations approach it by small steps;
alone, with transit times, in the single-lambda form and as the union of a
batch.  All comparisons with the oracle are exact."""
import numpy as np
import pytest
import torch

import oracle
import synth
from paper_1111_0627_gb300.ocm import OCM_FLAG_EVAL_GLOBAL, OCM_FLAG_HOST_LOOP

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_1111_0627_gb300 as ocm


def _dev(*arrays):
    return tuple(torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)).cuda() for a in arrays)


def _chains(n, depth, seed, cycles=1):
    """Chains of the given length, mostly of the best edges, into cycles of 11."""
    rng = np.random.default_rng(seed)
    v = np.arange(n)
    head = 11 * cycles
    to = np.where(v < head, v // 11 * 11 + (v % 11 + 1) % 11, v - 1)
    ends = np.nonzero((v >= head) & ((v - head) % depth == 0))[0]
    to[ends] = 11 * (np.arange(ends.size) % cycles) + 3
    name = rng.permutation(n)
    succ = np.empty(n, np.int64)
    succ[name] = name[to]
    col = np.empty(3 * n, np.int64)
    col[0::3], col[1::3], col[2::3] = rng.integers(0, n, n), succ, rng.integers(0, n, n)
    w = rng.integers(0, 1000, 3 * n)
    w[1::3] = np.where(rng.random(n) < 0.9, 3000, 900)
    w[3 * name[:head] + 1] = 2500
    rp = 3 * np.arange(n + 1)
    g = synth.Graph(rp.astype(np.int32), col.astype(np.int32), w.astype(np.int32), "max", "chains")
    return g, (rp[:-1] + 1).astype(np.int32), rng


def _check(g, s, h):
    assert (s.num, s.den, s.stats["iterations"]) == (h.num, h.den, h.iterations)
    assert s.cycle.cpu().tolist() == h.cycle.tolist()
    assert (s.eta_num.cpu().numpy() == h.eta_p).all()
    assert (s.eta_den.cpu().numpy() == h.eta_q).all()
    assert (s.potential.cpu().numpy() == h.V).all()


@pytest.mark.parametrize("ratio", [False, True], ids=["mean", "ratio"])
@pytest.mark.parametrize("n,depth,cycles", [(20_000, 20_000, 1), (20_000, 5000, 3), (50_000, 3000, 7),
                                            (3000, 3000, 2)])
def test_deep_optimum(n, depth, cycles, ratio):
    g, init, rng = _chains(n, depth, n + depth, cycles)
    t = rng.integers(1, 4, g.m).astype(np.int32) if ratio else None
    d = _dev(g.row_ptr, g.col_idx, g.w)
    kw = {} if t is None else {"transit": _dev(t)[0]}
    for start in (None, init):
        h = oracle.howard(g.row_ptr, g.col_idx, g.w, g.mode, init_policy=start, transit=t)
        ini = None if start is None else _dev(start)[0]
        for flags in (OCM_FLAG_EVAL_GLOBAL, OCM_FLAG_EVAL_GLOBAL | OCM_FLAG_HOST_LOOP):
            _check(g, ocm.solve(*d, g.mode, init_policy=ini, certificate=True, flags=flags, **kw), h)


@pytest.mark.parametrize("ratio", [False, True], ids=["mean", "ratio"])
def test_deep_single_lambda(ratio):
    g, init, rng = _chains(6000, 3000, 5, 2)
    w = g.w.copy()
    w[2::3] -= 5000
    col = g.col_idx.copy()
    col[2::3] = (np.arange(g.n) + 1) % g.n      # strongly connected
    t = rng.integers(1, 4, g.m).astype(np.int32) if ratio else None
    h = oracle.howard_single(g.row_ptr, col, w, "max", transit=t, init_policy=init)
    d = _dev(g.row_ptr, col, w, init)
    s = ocm.solve(*d[:3], "max", single_lambda=True, init_policy=d[3],
                  transit=None if t is None else _dev(t)[0])
    assert (s.num, s.den, s.stats["iterations"]) == (h.num, h.den, h.iterations)
    assert s.cycle.cpu().tolist() == h.cycle.tolist()


@pytest.mark.parametrize("ratio", [False, True], ids=["mean", "ratio"])
def test_deep_union_batch(ratio):
    rng = np.random.default_rng(3)
    parts = [_chains(n, n, n, 1) for n in (500, 3000, 9000, 20_000)]
    graphs = [p[0] for p in parts]
    graphs += [synth.tiny_random(rng, 30, max_extra=3, wlo=-9, whi=9, ring=True) for _ in range(40)]
    times = [rng.integers(1, 4, g.m).astype(np.int32) if ratio else None for g in graphs]
    b = synth.concat(graphs)
    vp, rp, col, w = _dev(b.graph_vptr, b.row_ptr, b.col_idx, b.w)
    tt = _dev(np.concatenate(times))[0] if ratio else None
    s = ocm.solve_batch(vp, rp, col, w, "max", transit=tt, small_vertices=-1)
    for k, g in enumerate(graphs):
        h = oracle.howard(g.row_ptr, g.col_idx, g.w, "max", transit=times[k])
        e0 = int(b.row_ptr[int(b.graph_vptr[k])])
        assert (int(s.num[k]), int(s.den[k])) == (h.num, h.den), k
        assert (s.cycle(k).cpu() - e0).tolist() == h.cycle.tolist(), k
