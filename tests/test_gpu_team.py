"""Graphs solved by one block or one cluster each (needs a GB300), at the sizes
where the batch changes between them.  All results are exact integers."""
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
