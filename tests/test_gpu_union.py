"""The union path of the batched solve (needs a GB300): every graph in one
disjoint union, walked and jumped together, with thousands of policy cycles in
an evaluation, so that the cycle table is built by more than one block.  All
results are exact integers, compared with the oracle's graph by graph."""
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
