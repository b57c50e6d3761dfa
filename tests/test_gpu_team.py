"""Graphs solved by one block or one cluster (needs a GB300): the whole solve of
a small graph in one launch, and the batch's teams.  Sizes lie at the edges of
the dispatch (blocks and clusters, states in shared or global memory, threads
and warps per vertex, cycles walked or lifted).  All results are exact integers:
the oracle's value, cycle, iteration count and, for the certificate, values."""
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


def _check(g, **kw):
    h = oracle.howard(g.row_ptr, g.col_idx, g.w, g.mode, **kw)
    init = {k: _dev(v)[0] for k, v in kw.items()}
    s = ocm.solve(*_dev(g.row_ptr, g.col_idx, g.w), g.mode, certificate=True, **init)
    assert (s.num, s.den, s.stats["iterations"]) == (h.num, h.den, h.iterations), g.name
    assert s.cycle.cpu().tolist() == [int(x) for x in h.cycle], g.name
    rc, bad = oracle.certificate(g.row_ptr, g.col_idx, g.w, g.mode, s.eta_num.cpu().numpy(),
                                 s.eta_den.cpu().numpy(), s.potential.cpu().numpy(), s.num, s.den,
                                 s.cycle.cpu().numpy())
    assert rc == 0, (g.name, rc, bad)
    return s


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 512, 513, 1024, 1025, 4096, 4097, 8192, 8193,
                               12190, 12191, 16384, 16385])
@pytest.mark.parametrize("mode", ["max", "min"])
def test_solve_sizes(n, mode):
    s = _check(synth.ring_extra(n, 0, 5, -1000, 1000, seed=91 + n, tag=1, mode=mode))
    if n <= 16384:
        assert s.stats["launches"] <= 2   # (the solve and the certificate)


@pytest.mark.parametrize("n", [300, 1500, 9000])
@pytest.mark.parametrize("deg", [32, 33, 200, 1024, 1025])
def test_solve_wide_vertices(n, deg):
    rng = np.random.default_rng(n + deg)
    edges = [(v, (v + 1) % n, int(rng.integers(-50, 50))) for v in range(n)]
    for v in rng.integers(0, n, 2):
        edges += [(int(v), int(t), int(rng.integers(-50, 60))) for t in rng.integers(0, n, deg)]
    _check(synth.from_edges(n, edges, "max", "wide"))


@pytest.mark.parametrize("n,cycle", [(400, 48), (400, 49), (1000, 300), (3000, 2999), (10_000, 257),
                                     (16_000, 16_000), (20_000, 48), (20_000, 49)])
def test_solve_long_cycles_and_chains(n, cycle):
    """The heaviest cycle has the given length; the first policy leads into it
    by a chain of all other vertices, every one of which has a loop as well."""
    to = np.arange(1, n + 1) % n
    to[cycle - 1] = 0
    if cycle < n:
        to[n - 1] = 0
    edges = []
    for v in range(n):
        edges += [(v, int(to[v]), 5), (v, v, 4)]
    g = synth.from_edges(n, edges, "max", "chain")
    _check(g)
    _check(g, init_policy=np.asarray(g.row_ptr[:-1], dtype=np.int32))       # the chain
    _check(g, init_policy=np.asarray(g.row_ptr[:-1] + 1, dtype=np.int32))   # the loops


@pytest.mark.parametrize("extra", [0, 60])
def test_batch_teams(extra):
    """Graphs around the sizes at which a block, a cluster and its shared memory
    change, among small ones; the largest is far above the average per block."""
    sizes = [1, 40, 4095, 4096, 4097, 12_189, 12_190, 12_191, 16_384, 50_000] + [300] * extra
    graphs = [synth.ring_extra(n, 0, 7, 1, 10_000, seed=17, tag=k, mode="max")
              for k, n in enumerate(sizes)]
    b = synth.concat(graphs)
    args = _dev(b.graph_vptr, b.row_ptr, b.col_idx, b.w)
    for small in (0, 60_000):
        s = ocm.solve_batch(*args, b.mode, small_vertices=small)
        for k, g in enumerate(graphs):
            h = oracle.howard(g.row_ptr, g.col_idx, g.w, g.mode)
            assert (int(s.num[k]), int(s.den[k])) == (h.num, h.den), (small, k)
            e0 = int(b.row_ptr[int(b.graph_vptr[k])])
            assert (s.cycle(k).cpu() - e0).tolist() == [int(x) for x in h.cycle], (small, k)
