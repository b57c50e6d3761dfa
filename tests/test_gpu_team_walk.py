"""The walks of a block or a cluster on its own graph (needs a GB300), started
by given policies: small cycles that the samples miss, found while others
already walk, none or few of them settled before; thousands of cycles at once;
long cycles.  Solved alone (one launch) and as a batch with warm starts, in
blocks and in clusters.  All comparisons are exact."""
import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_1111_0627_gb300 as ocm


def _dev(*arrays):
    return tuple(torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)).cuda() for a in arrays)


def _loops(n):
    return np.arange(n)


def _small_cycles(n, size):
    """Cycles of the given size and nothing else."""
    v = np.arange(n)
    start = v - v % size
    return np.minimum(start + (v - start + 1) % size, n - 1)


def _chains_and_cycles(n, size, every):
    """One cycle with everything behind it, in chains of 40, and small cycles
    with nothing behind them: samples meet few of those."""
    v = np.arange(n)
    to = np.where(v < 5, (v + 1) % 5, v - 1)
    to[(v >= 5) & ((v - 5) % 40 == 0)] = 2
    for a in range(7, n - size - 1, every):
        to[a:a + size] = np.arange(a + 1, a + size + 1)
        to[a + size - 1] = a
    return to


SHAPES = {
    "loops": _loops,
    "pairs": lambda n: _small_cycles(n, 2),
    "cycles_37": lambda n: _small_cycles(n, 37),
    "cycles_300": lambda n: _small_cycles(n, 300),
    "missed_2": lambda n: _chains_and_cycles(n, 2, 331),
    "missed_9": lambda n: _chains_and_cycles(n, 9, 977),
}


def _graph(shape, n, seed):
    """Random edges beside the policy's; some of the policy's are good ones."""
    rng = np.random.default_rng(seed)
    name = rng.permutation(n)
    succ = np.empty(n, np.int32)
    succ[name] = name[SHAPES[shape](n)]
    col = np.empty(3 * n, np.int32)
    col[0::3] = rng.integers(0, n, n)
    col[1::3] = succ
    col[2::3] = (np.arange(n) + 1) % n
    w = rng.integers(0, 1000, 3 * n).astype(np.int32)
    w[1::3] = rng.integers(500, 1100, n)
    rp = (3 * np.arange(n + 1)).astype(np.int32)
    return synth.Graph(rp, col, w, "max", shape), (3 * np.arange(n) + 1).astype(np.int32)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("n", [500, 1021, 4001, 16_384])
def test_given_policies_alone(shape, n):
    g, init = _graph(shape, n, 31 * n + len(shape))
    h = oracle.howard(g.row_ptr, g.col_idx, g.w, g.mode, init_policy=init)
    d = _dev(g.row_ptr, g.col_idx, g.w, init)
    for rep in range(3):
        s = ocm.solve(*d[:3], g.mode, init_policy=d[3], certificate=True)
        assert (s.num, s.den, s.stats["iterations"]) == (h.num, h.den, h.iterations), rep
        assert s.cycle.cpu().tolist() == h.cycle.tolist(), rep
        rc, bad = oracle.certificate(g.row_ptr, g.col_idx, g.w, g.mode, s.eta_num.cpu().numpy(),
                                     s.eta_den.cpu().numpy(), s.potential.cpu().numpy(), s.num,
                                     s.den, s.cycle.cpu().numpy())
        assert rc == 0, (rc, bad)


@pytest.mark.parametrize("shape", SHAPES)
def test_given_policies_as_a_batch(shape):
    sizes = [100, 1500, 4000, 4100, 9000, 12_500, 30_000]
    pairs = [_graph(shape, n, 7 * n + len(shape)) for n in sizes]
    graphs = [g for g, _ in pairs]
    b = synth.concat(graphs)
    e0 = [int(b.row_ptr[int(v)]) for v in b.graph_vptr[:-1]]
    init = np.concatenate([i + e for (_, i), e in zip(pairs, e0)])
    vp, rp, col, w, ini = _dev(b.graph_vptr, b.row_ptr, b.col_idx, b.w, init)
    oracles = [oracle.howard(g.row_ptr, g.col_idx, g.w, g.mode, init_policy=i) for g, i in pairs]
    for rep in range(3):
        s = ocm.solve_batch(vp, rp, col, w, b.mode, init_policy=ini, small_vertices=40_000)
        for k, h in enumerate(oracles):
            assert (int(s.num[k]), int(s.den[k])) == (h.num, h.den), (rep, k)
            assert (s.cycle(k).cpu() - e0[k]).tolist() == h.cycle.tolist(), (rep, k)
        assert s.stats["iterations"] == max(h.iterations for h in oracles)


@pytest.mark.parametrize("n,K", [(512, 256), (1024, 511), (1024, 512), (4096, 510), (4096, 511),
                                 (1024, 513), (1024, 1024), (4096, 2048), (4096, 2049), (9000, 4100)])
def test_best_of_many_cycles(n, K):
    """K loops with many equal weights and a few better cycles, in blocks and in
    clusters, whose blocks find the best of them together; K on both sides of
    the numbers at which one thread ranks a cycle, or several do."""
    rng = np.random.default_rng(n + K)
    name = rng.permutation(n)
    edges = []
    for v in range(n):
        if v < K:
            edges.append((int(name[v]), int(name[v]), int(rng.integers(0, 40))))
        else:
            edges += [(int(name[v]), int(name[t]), int(rng.integers(0, 100)))
                      for t in rng.integers(0, n, 3)] + [(int(name[v]), int(name[v - 1]), 0)]
    g = synth.from_edges(n, edges, "max", "loops")
    h = oracle.howard(g.row_ptr, g.col_idx, g.w, g.mode)
    s = ocm.solve(*_dev(g.row_ptr, g.col_idx, g.w), g.mode, certificate=True)
    assert s.stats["launches"] <= 2 and s.stats["cycles"] >= K
    assert (s.num, s.den, s.stats["iterations"]) == (h.num, h.den, h.iterations)
    assert s.cycle.cpu().tolist() == h.cycle.tolist()
    assert (s.potential.cpu().numpy() == h.V).all()
    assert (s.eta_num.cpu().numpy() == h.eta_p).all()
