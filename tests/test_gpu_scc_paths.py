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
