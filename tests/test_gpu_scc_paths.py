"""Components of graphs with long acyclic parts (needs a GB300): the trimming
rounds shorten every path at once, where a search splits one path of a class
per iteration.  Labels are exact; the iterations are counted by the launches."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_1111_0627_gb300 as ocm


def _solve(count, length, seed):
    """Vertex-disjoint paths in random vertex order, one end with a loop."""
    n = count * length
    name = np.random.default_rng(seed).permutation(n)
    v = np.arange(n)
    edges = [(int(name[a]), int(name[a + 1]), 1) for a in v[v % length != length - 1]]
    edges.append((int(name[n - 1]), int(name[n - 1]), 7))
    g = synth.from_edges(n, edges, "max", f"paths({count},{length})")
    s = ocm.solve_scc(*(torch.from_numpy(x).cuda() for x in (g.row_ptr, g.col_idx, g.w)), "max")
    assert s.labels.cpu().tolist() == list(range(n))
    assert (s.root.tolist(), s.num.tolist(), s.den.tolist()) == ([int(name[n - 1])], [7], [1])
    return s.stats["launches"]


@pytest.mark.parametrize("length", [2, 25, 64, 200])
def test_bundles_of_paths_take_few_iterations(length):
    """An iteration has 12 trimming rounds, each of which takes both ends of
    every path: 24 vertices of a path at least, and one launch."""
    assert _solve(200, length, length) - _solve(200, 1, 0) <= length // 24 + 3


@pytest.mark.parametrize("n,K,size", [(20_000, 300, 1), (20_000, 300, 7), (5000, 4990, 1), (3000, 2, 1400)])
def test_many_components_of_one_class(n, K, size):
    """K rings with trees leading into them and no other edge: every split leaves
    the rings that its pivot does not reach in one class, scattered over all
    threads, beside the classes split off."""
    rng = np.random.default_rng(n + K + size)
    v = np.arange(n)
    head = K * size
    to = np.where(v < head, v // size * size + (v % size + 1) % size, rng.integers(0, n, n))
    to[head:] = np.minimum(to[head:], np.maximum(v[head:] - 1, 0))   # (no other ring)
    name = rng.permutation(n)
    col = np.empty(n, np.int64)
    col[name] = name[to]
    labels, count = ocm.scc(*(torch.from_numpy(x.astype(np.int32)).cuda()
                              for x in (np.arange(n + 1), col)))
    want = v.copy()
    for k in range(K):
        ring = name[k * size:(k + 1) * size]
        want[ring] = ring.min()
    assert (labels.cpu().numpy() == want).all()
    assert count == n - head + K
