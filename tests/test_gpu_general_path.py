"""The launch-per-step path on small graphs (needs a GB300).  By default they
are solved in one launch by one team; the flag that forbids the two-level
evaluation also keeps the general path: the graph loop and its exits, the
initial pass, the walks and jump rounds and the extraction, on the shapes and
sizes at which they can go wrong.  All comparisons with the oracle are exact."""
import numpy as np
import pytest
import torch

import oracle
import synth
from paper_1111_0627_gb300.ocm import OCM_FLAG_EVAL_GLOBAL as GENERAL
from paper_1111_0627_gb300.ocm import OCM_FLAG_HOST_LOOP
from test_gpu_walk import SHAPES

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_1111_0627_gb300 as ocm


def _dev(*arrays):
    return [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in arrays]


def _check(g, s, h):
    assert s.stats["launches"] > 2
    assert (s.num, s.den, s.stats["iterations"]) == (h.num, h.den, h.iterations), g.name
    assert s.cycle.cpu().tolist() == [int(x) for x in h.cycle], g.name


@pytest.mark.parametrize("mode", ["max", "min"])
def test_graph_loop_equals_host_loop_and_team(mode):
    rng = np.random.default_rng(77_101 + (mode == "min"))
    for trial in range(60):
        n = int(rng.integers(1, 40))
        g = synth.tiny_random(rng, n, max_extra=4, wlo=-25, whi=25, ring=bool(trial % 2), mode=mode)
        init = synth.random_policy(rng, g.row_ptr) if trial % 3 == 0 else None
        h = oracle.howard(g.row_ptr, g.col_idx, g.w, mode, init_policy=init)
        d = _dev(g.row_ptr, g.col_idx, g.w)
        ini = None if init is None else _dev(init)[0]
        a = ocm.solve(*d, mode, init_policy=ini, flags=GENERAL, certificate=True)
        b = ocm.solve(*d, mode, init_policy=ini, flags=GENERAL | OCM_FLAG_HOST_LOOP, certificate=True)
        c = ocm.solve(*d, mode, init_policy=ini, certificate=True)
        assert (a.stats["graph_loop"], b.stats["graph_loop"]) == (1, 0) and c.stats["launches"] == 2
        _check(g, a, h)
        _check(g, b, h)
        for k in ("iterations", "switched", "cycles"):
            assert a.stats[k] == b.stats[k] == c.stats[k], k
        for k in ("eta_num", "eta_den", "potential", "policy"):
            assert torch.equal(getattr(a, k), getattr(b, k)), k
            assert torch.equal(getattr(a, k), getattr(c, k)), k


def test_graph_loop_iteration_cap_and_stream():
    g = synth.ring10k()
    h = oracle.howard(g.row_ptr, g.col_idx, g.w, g.mode)
    d = _dev(g.row_ptr, g.col_idx, g.w)
    for cap in (1, 2, h.iterations):
        with pytest.raises(ocm.OCMError) as ei:
            ocm.solve(*d, g.mode, max_iters=cap, flags=GENERAL)
        assert ei.value.status == -5
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        sol = ocm.solve(*d, g.mode, max_iters=h.iterations + 1, flags=GENERAL)
    assert sol.stats["graph_loop"] == 1
    _check(g, sol, h)


def test_resolve_on_the_general_path():
    g = synth.ring10k()
    d = _dev(g.row_ptr, g.col_idx, g.w)
    first = ocm.solve(*d, g.mode, certificate=True, flags=GENERAL)
    rng = np.random.default_rng(12)
    w2 = g.w.copy()
    w2[rng.integers(0, g.m, 64)] += rng.integers(-30, 31, 64).astype(np.int32)
    (w2d,) = _dev(w2)
    h = oracle.howard(g.row_ptr, g.col_idx, w2, g.mode, init_policy=first.policy.cpu().numpy())
    _check(g, ocm.solve(d[0], d[1], w2d, g.mode, init_policy=first.policy, flags=GENERAL), h)


@pytest.mark.parametrize("shape", SHAPES)
def test_given_policies_follow_the_oracle(shape):
    """The mean instance of the walks (test_gpu_walk: the ratio's, and teams)."""
    rng = np.random.default_rng(30_011 + len(shape))
    to = SHAPES[shape]().astype(np.int32)
    n = to.shape[0]
    name = rng.permutation(n).astype(np.int32)
    succ = np.empty(n, np.int32)
    succ[name] = name[to]
    col = np.empty(2 * n, np.int32)
    col[0::2] = rng.integers(0, n, n)
    col[1::2] = succ
    rp = (2 * np.arange(n + 1)).astype(np.int32)
    w = rng.integers(-1000, 1001, 2 * n).astype(np.int32)
    init = (2 * np.arange(n) + 1).astype(np.int32)
    g = synth.Graph(rp, col, w, "max", shape)
    h = oracle.howard(rp, col, w, "max", init_policy=init)
    d = _dev(rp, col, w, init)
    s = ocm.solve(*d[:3], "max", init_policy=d[3], certificate=True, flags=GENERAL)
    _check(g, s, h)
    assert (s.potential.cpu().numpy() == h.V).all()
    assert (s.eta_num.cpu().numpy() == h.eta_p).all()
    assert (s.eta_den.cpu().numpy() == h.eta_q).all()


def test_errors_on_the_general_path():
    g = synth.ring10k()
    d = _dev(g.row_ptr, g.col_idx, g.w)

    def status(rp=d[0], col=d[1], w=d[2], **kw):
        with pytest.raises(ocm.OCMError) as e:
            ocm.solve(rp, col, w, g.mode, **kw)
        return e.value.status

    cases = []
    x = d[0].clone()
    x[5] = x[6]
    cases.append((dict(rp=x), -3))
    x = d[0].clone()
    x[5] = x[7] + 1
    cases.append((dict(rp=x), -2))
    x = d[1].clone()
    x[99] = g.n
    cases.append((dict(col=x), -2))
    x = d[1].clone()
    x[99] = -1
    cases.append((dict(col=x), -2))
    x = d[2].clone()
    x[g.m - 1] = -2**31
    cases.append((dict(w=x), -4))
    x = d[0][:-1].clone()
    x[8] = d[0][9]
    cases.append((dict(init_policy=x), -1))
    for kw, code in cases:
        assert status(**kw) == code == status(flags=GENERAL, **kw)
