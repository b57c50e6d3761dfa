"""The union path of the batched solve (needs a GB300): every graph in one
disjoint union, walked and jumped together, with thousands of policy cycles in
an evaluation, so that the cycle table is built by more than one block.  All
results are exact integers, compared with the oracle's graph by graph."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_1111_0627_gb300 as ocm
    from paper_1111_0627_gb300 import _native


def _dev(*arrays):
    return tuple(torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)).cuda() for a in arrays)


def _check_batch(b, graphs, sol, oracles):
    num, den = sol.num.cpu().tolist(), sol.den.cpu().tolist()
    length, cyc = sol.cycle_len.cpu().tolist(), sol.cycle_out.cpu().numpy()
    for k, (g, h) in enumerate(zip(graphs, oracles)):
        assert (num[k], den[k]) == (h.num, h.den), k
        v0 = int(b.graph_vptr[k])
        e0 = int(b.row_ptr[v0])
        assert length[k] == len(h.cycle), k
        assert (cyc[v0:v0 + length[k]] - e0).tolist() == h.cycle.tolist(), k


@pytest.mark.parametrize("G", [1024, 1025, 5000])
def test_ratio_batch_of_many_graphs(G):
    """Ratios with large denominators, close together, in every block's part of
    the cycle table: the order keys need the largest denominator of them all."""
    rng = np.random.default_rng(4_100 + G)
    graphs = [synth.tiny_random(rng, int(rng.integers(2, 30)), max_extra=4, wlo=-40, whi=40, ring=True)
              for _ in range(G)]
    times = [rng.integers(1, 4000, g.m).astype(np.int32) for g in graphs]
    b = synth.concat(graphs)
    vp, rp, col, w, tt = _dev(b.graph_vptr, b.row_ptr, b.col_idx, b.w, np.concatenate(times))
    oracles = [oracle.howard(g.row_ptr, g.col_idx, g.w, "max", transit=t)
               for g, t in zip(graphs, times)]
    for rep in range(3):
        _check_batch(b, graphs, ocm.solve_batch(vp, rp, col, w, "max", transit=tt), oracles)


@pytest.mark.parametrize("seed", range(3))
def test_ratio_roots_settled_by_others(seed):
    """Pairs that become cycles at the third evaluation, 16 to a warp, most of
    which a warp gives up on; walks that come by from elsewhere settle some of
    their roots all the same.  A root's value is 0 whoever settled it."""
    rng = np.random.default_rng(9_200 + seed)
    n, pairs, feeders = 120_000, 1000, 3000
    a = 64 + 2 * np.arange(pairs)         # pairs (a, a + 1), neighbours in the vertex order
    edges = [np.stack([np.arange(n), np.arange(n) // 3, rng.integers(-6, -1, n)], 1)]   # a tree
    edges[0][0] = (0, 0, 0)               # ... to a loop of mean 0
    high, low = n - 1, n - 2
    edges[0][high], edges[0][low] = (high, 0, 500), (low, 0, -500)
    edges[0][a] = np.stack([a, np.full(pairs, high), rng.integers(0, 50, pairs)], 1)
    edges[0][a + 1] = np.stack([a + 1, np.full(pairs, low), rng.integers(0, 50, pairs)], 1)
    c = n - 10 - feeders + np.arange(feeders)
    edges[0][c] = np.stack([c, a[rng.permutation(feeders) % pairs], rng.integers(-9, 9, feeders)], 1)
    edges.append(np.stack([a, a + 1, rng.integers(1, 9, pairs)], 1))
    edges.append(np.stack([a + 1, a, rng.integers(1, 9, pairs)], 1))
    e = np.concatenate(edges)
    # (nothing of the tree leads through the pairs or the feeders)
    inner = np.isin(e[:, 1], np.concatenate([a, a + 1, c])) & ~np.isin(e[:, 0], np.concatenate(
        [a, a + 1, c]))
    e[inner, 1] = 1
    order = np.argsort(e[:, 0], kind="stable")
    e = e[order].astype(np.int32)
    rp = np.zeros(n + 1, np.int32)
    rp[1:] = np.cumsum(np.bincount(e[:, 0], minlength=n))
    col, w = np.ascontiguousarray(e[:, 1]), np.ascontiguousarray(e[:, 2])
    t = rng.integers(1, 9, col.shape[0]).astype(np.int32)
    init = rp[:-1].copy()
    h = oracle.howard(rp, col, w, "max", init_policy=init, transit=t)
    assert h.iterations >= 2
    d = _dev(rp, col, w, init, t)
    s = ocm.solve(*d[:3], "max", init_policy=d[3], transit=d[4], certificate=True)
    assert (s.num, s.den, s.stats["iterations"]) == (h.num, h.den, h.iterations)
    assert s.cycle.cpu().tolist() == h.cycle.tolist()
    V = s.potential.cpu().numpy()
    assert (V[a] == 0).all() and (V == h.V).all()


@pytest.mark.parametrize("ratio", [False, True], ids=["mean", "ratio"])
def test_per_vertex_outputs_of_a_batch(ratio):
    """Graphs that converge in different steps, among them some with several
    cycles in the final policy: every vertex's value, cycle mean and policy
    edge, through the C interface, are those of its graph solved alone."""
    rng = np.random.default_rng(77 + ratio)
    graphs = [synth.tiny_random(rng, int(rng.integers(1, 60)), max_extra=3, wlo=-30, whi=30,
                                ring=k % 3 == 0) for k in range(150)]
    graphs += [synth.ring_extra(3000, 0, 5, -100, 100, seed=8, tag=k, mode="max") for k in range(3)]
    times = [rng.integers(1, 9, g.m).astype(np.int32) for g in graphs]
    b = synth.concat(graphs)
    N, M, G = b.row_ptr.shape[0] - 1, b.col_idx.shape[0], len(graphs)
    vp, rp, col, w, tt = _dev(b.graph_vptr, b.row_ptr, b.col_idx, b.w, np.concatenate(times))
    lib = _native.load()
    out = {"eta_num": torch.zeros(N, dtype=torch.int64, device="cuda"),
           "eta_den": torch.zeros(N, dtype=torch.int32, device="cuda"),
           "potential": torch.zeros(N, dtype=torch.int64, device="cuda"),
           "policy": torch.zeros(N, dtype=torch.int32, device="cuda")}
    opt = _native.OcmOptions()
    for k, x in out.items():
        setattr(opt, k, x.data_ptr())
    if ratio:
        opt.transit = tt.data_ptr()
    num = torch.zeros(G, dtype=torch.int64, device="cuda")
    den, clen = (torch.zeros(G, dtype=torch.int32, device="cuda") for _ in range(2))
    cyc = torch.zeros(N, dtype=torch.int32, device="cuda")
    ws = torch.empty(lib.ocm_workspace_size_batch(G, N, M), dtype=torch.uint8, device="cuda")
    rc = lib.ocm_solve_batch(vp.data_ptr(), rp.data_ptr(), col.data_ptr(), w.data_ptr(), G, N, M, 0,
                             num.data_ptr(), den.data_ptr(), clen.data_ptr(), cyc.data_ptr(),
                             ws.data_ptr(), ws.numel(), torch.cuda.current_stream().cuda_stream,
                             ctypes.byref(opt), None)
    assert rc == 0
    got = {k: x.cpu().numpy() for k, x in out.items()}
    for k, g in enumerate(graphs):
        h = oracle.howard(g.row_ptr, g.col_idx, g.w, "max", transit=times[k] if ratio else None)
        v0, v1 = int(b.graph_vptr[k]), int(b.graph_vptr[k + 1])
        assert (int(num[k]), int(den[k])) == (h.num, h.den), k
        assert (got["eta_num"][v0:v1] == h.eta_p).all(), k
        assert (got["eta_den"][v0:v1] == h.eta_q).all(), k
        assert (got["potential"][v0:v1] == h.V).all(), k
        assert (got["policy"][v0:v1] - int(b.row_ptr[v0]) == h.policy).all(), k
