"""The autotuner on graphs that the library solves in one launch (needs a
GB300): the recorded choice must not take that away where it is faster, whoever
wrote the table."""
import json

import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_1111_0627_gb300 as ocm


@pytest.mark.parametrize("n", [257, 9000])
def test_tuned_small_graphs_stay_in_one_launch(n, tmp_path, monkeypatch):
    path = tmp_path / "tune.json"
    monkeypatch.setenv("OCM_TUNE_FILE", str(path))
    g = synth.ring_extra(n, 0, 4, 1, 100, seed=3, tag=1, mode="max")
    d = [torch.from_numpy(x).cuda() for x in (g.row_ptr, g.col_idx, g.w)]
    h = oracle.howard(g.row_ptr, g.col_idx, g.w, g.mode)
    res = ocm.autotune.tune(*d, g.mode, candidates=[(1, 8, 512), (2, 4, 128)])
    # (1.3 to 3 times as fast at these sizes)
    assert (res["sweep_kind"], res["edges_per_lane"], res["sweep_threads"]) == (0, 0, 0)
    assert ocm.autotune.lookup(d[0]) == (0, 0, 0)
    s = ocm.solve(*d, g.mode, tune=True)
    assert (s.num, s.den, s.stats["iterations"]) == (h.num, h.den, h.iterations)
    assert s.stats["launches"] == 1
    # a table from before there was a one-launch solve
    path.write_text(json.dumps({res["signature"]: {"sweep_kind": 1, "edges_per_lane": 8,
                                                   "sweep_threads": 512, "sweep_ms": 0.004}}))
    assert ocm.autotune.lookup(d[0]) is None
    assert ocm.solve(*d, g.mode, tune=True).stats["launches"] == 1


def test_tuned_small_hub_keeps_a_candidate(tmp_path, monkeypatch):
    """More than 1,024 out-edges: the default is no single launch."""
    monkeypatch.setenv("OCM_TUNE_FILE", str(tmp_path / "tune.json"))
    rng = np.random.default_rng(4)
    n = 2000
    deg = np.full(n, 2)
    deg[7] = 3000
    rp = np.zeros(n + 1, np.int32)
    rp[1:] = np.cumsum(deg)
    col = rng.integers(0, n, int(rp[-1])).astype(np.int32)
    w = rng.integers(0, 99, col.shape[0]).astype(np.int32)
    d = [torch.from_numpy(x).cuda() for x in (rp, col, w)]
    cands = [(1, 8, 512), (1, 4, 256)]
    res = ocm.autotune.tune(*d, "max", candidates=cands)
    picked = (res["sweep_kind"], res["edges_per_lane"], res["sweep_threads"])
    assert picked in cands and ocm.autotune.lookup(d[0]) == picked
    h = oracle.howard(rp, col, w, "max")
    s = ocm.solve(*d, "max", tune=True)
    assert (s.num, s.den) == (h.num, h.den)
