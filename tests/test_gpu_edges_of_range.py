"""Sizes and weights at the edges of what a form holds (needs a GB300): the
largest graph whose states fit in one block's shared memory, in a batch large
enough that it is solved by a block and not by a cluster; and path times just
below the limit of the cycle ratio.  Exact comparison with the oracle."""
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


def test_states_that_just_fit_in_shared_memory():
    """8.2 million vertices: a graph of less than 16,384 is no sixth of a
    block's share, so each is solved by one block."""
    graphs = [synth.ring_extra(n, 0, 4, 1, 10_000, seed=3, tag=n, mode="max")
              for n in (12_191, 12_192, 12_193, 12_224)]
    b = synth.concat(graphs)
    copies = 168
    N, M = int(b.row_ptr.shape[0] - 1), int(b.col_idx.shape[0])
    assert copies * N > 6 * 152 * 8192
    vp, rp, col, w = _dev(b.graph_vptr, b.row_ptr, b.col_idx, b.w)
    k = torch.arange(copies, dtype=torch.int32, device="cuda")[:, None]
    one = torch.ones(1, dtype=torch.int32, device="cuda")
    vps = torch.cat([(vp[None, :-1] + k * N).reshape(-1), one * (copies * N)])
    rps = torch.cat([(rp[None, :-1] + k * M).reshape(-1), one * (copies * M)])
    cols, ws = (col[None, :] + k * N).reshape(-1), w.repeat(copies)
    s = ocm.solve_batch(vps, rps, cols, ws, "max")
    assert s.stats["batch_small_graphs"] == 4 * copies
    hs = [oracle.howard(g.row_ptr, g.col_idx, g.w, "max") for g in graphs]
    num, den = s.num.reshape(copies, 4).cpu(), s.den.reshape(copies, 4).cpu()
    cyc = s.cycle_out.reshape(copies, N).cpu().numpy()
    for j, h in enumerate(hs):
        assert (num[:, j] == h.num).all() and (den[:, j] == h.den).all(), j
        v0, e0 = int(b.graph_vptr[j]), int(b.row_ptr[int(b.graph_vptr[j])])
        L = len(h.cycle)
        want = h.cycle[None, :] + e0 + M * np.arange(copies)[:, None]
        assert (cyc[:, v0:v0 + L] == want).all(), j


@pytest.mark.parametrize("n", [300, 20_000, 70_000])
def test_path_times_up_to_the_limit(n):
    """n max t = 2^31 - 1 less a remainder, on a policy whose paths have nearly
    n steps: times, values and the optimum are exact; one more is refused."""
    top = (2**31 - 1) // n
    rng = np.random.default_rng(n)
    rp = (2 * np.arange(n + 1)).astype(np.int32)
    col = np.empty(2 * n, np.int32)
    col[0::2] = np.minimum(np.arange(n) + 1, n - 1)   # one chain into a loop
    col[1::2] = np.maximum(np.arange(n) - rng.integers(0, 40, n), 0)
    w = rng.integers(-3, 4, 2 * n).astype(np.int32)
    t = rng.integers(top - 5, top + 1, 2 * n).astype(np.int32)
    t[7] = top
    assert 4 * n * n * int(np.abs(w).max()) * top < 2**62
    init = rp[:-1].copy()
    h = oracle.howard(rp, col, w, "max", init_policy=init, transit=t)
    d = _dev(rp, col, w, init, t)
    s = ocm.solve(*d[:3], "max", init_policy=d[3], transit=d[4], certificate=True)
    assert (s.num, s.den, s.stats["iterations"]) == (h.num, h.den, h.iterations)
    assert s.cycle.cpu().tolist() == h.cycle.tolist()
    assert (s.potential.cpu().numpy() == h.V).all()
    d[4][7] = top + 1
    if n * (top + 1) > 2**31 - 1:
        with pytest.raises(ocm.OCMError) as e:
            ocm.solve(*d[:3], "max", init_policy=d[3], transit=d[4])
        assert e.value.status == -4
