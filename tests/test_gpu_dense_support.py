"""The dense support schedule's sweeps (GPU only): deletions re-checked with the
vertex rule alongside, on rows whose class-major copy is kept up to date; and
runs of one handle launched directly, then as a graph.  Bit-exact against the
plain bitset sweep."""
import numpy as np
import pytest

import paper_2212_00574_gb300 as kz
from paper_2212_00574_gb300 import synth
from tests.test_gpu_parity import gpu_run

pytestmark = pytest.mark.gpu


# classes of 1 to 55 words (below and above a warp's width), long cascades in
# which vertices fail in most sweeps, k = 2 (no edge rule: vertices only)
@pytest.mark.parametrize("n,k,p", [(90, 4, 0.3), (700, 9, 0.28), (1300, 3, 0.02), (2500, 2, 0.0004), (2500, 12, 0.17),
                                   (5200, 12, 0.11), (6200, 4, 0.036), (7000, 4, 0.036), (3100, 30, 0.33)])
def test_support_sweeps_match_the_plain_ones(n, k, p):
    g = synth.kpartite(n, k, p, 9600 + n, planted=True)
    want = gpu_run(g, dense=True, path="bitset")
    for path in ("auto", "bitset"):
        got = gpu_run(g, dense=True, path=path, schedule="support")
        for f in ("alive", "edges", "dv", "de", "v_sweep"):
            assert np.array_equal(got[f], want[f]), f
        for f in ("sweeps", "n_live", "m_live", "status"):
            assert got["stats"][f] == want["stats"][f], f
    lim = max(1, want["stats"]["sweeps"] // 2)
    got = gpu_run(g, dense=True, schedule="support", max_sweeps=lim)
    part = gpu_run(g, dense=True, path="bitset", max_sweeps=lim)
    assert np.array_equal(got["edges"], part["edges"]) and got["stats"]["sweeps"] == part["stats"]["sweeps"]
    assert got["stats"]["status"] == part["stats"]["status"]


@pytest.mark.parametrize("n,k,p", [(2600, 6, 0.4), (300, 10, 0.7)])
def test_runs_of_one_handle(n, k, p):
    g = synth.kpartite(n, k, p, 9700 + n, planted=True)
    want = gpu_run(g, dense=True, path="bitset", use_graph=0)
    with kz.KernelGraph.from_synth(g, dense=True) as kg:
        for lim in (0, 0, 0, 1, 0):  # direct, graph, graph, another limit, back
            kg.reset().kernelize(path="bitset", max_sweeps=lim)
            alive, edges, st = kg.fetch(allow=(kz.KZ_OK, kz.KZ_ERR_LIMIT))
            if lim == 0:
                assert np.array_equal(alive, want["alive"]) and np.array_equal(edges, want["edges"])
                assert st["sweeps"] == want["stats"]["sweeps"] and st["edge_tests"] == want["stats"]["edge_tests"]
            else:
                assert st["sweeps"] <= 1
