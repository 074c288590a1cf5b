"""CSR passes on graphs of short rows, whose vertices share a warp (GPU only):
isolated vertices, rows around eight entries, hubs among them with rows beyond
the hash table, clique sizes, limits and the support schedule.  Bit-exact
against the oracle."""
import numpy as np
import pytest

import oracle
import paper_2212_00574_gb300 as kz
from paper_2212_00574_gb300 import synth
from tests.test_gpu_parity import assert_parity, gpu_run

pytestmark = pytest.mark.gpu


def _hubs(n, k, mean, hubs, seed):
    # short rows, and `hubs` vertices joined to one another and to 600 of the rest
    rng = np.random.default_rng(seed)
    colour = rng.integers(0, k, n).astype(np.int32)
    e = rng.integers(0, n, (int(mean * n / 2), 2))
    h = np.repeat(np.arange(hubs), 600)
    w = rng.integers(0, min(n, 1500), len(h))
    iu = np.stack(np.triu_indices(hubs, 1), axis=1)
    e = np.concatenate([e, np.stack([h, w], 1), iu])
    e = e[colour[e[:, 0]] != colour[e[:, 1]]]
    return synth.Graph(n=n, k=k, colour=colour, edges=synth.canonical_edges(e), planted=[])


@pytest.mark.parametrize("n,k,mean,hubs", [(9000, 3, 2.0, 0), (12000, 4, 7.5, 0), (30000, 3, 5.0, 400),
                                           (40000, 5, 1.0, 500), (37, 3, 6.0, 0), (30011, 12, 3.0, 330)])
def test_short_rows_and_hubs(n, k, mean, hubs):
    g = _hubs(n, k, mean, hubs, 9900 + n)
    edges = g.get_edges()
    assert 2 * len(edges) < 16 * n
    assert_parity(g, gpu_run(g, path="sparse"))
    for q in sorted({k - 1, 2}):
        res = gpu_run(g, path="sparse", clique_k=q)
        orc = oracle.fixpoint(g.colour, edges, k, clique_k=q)
        assert np.array_equal(res["alive"], orc["vlive"])
        assert np.array_equal(res["edges"], edges[orc["elive"].astype(bool)])
        assert res["stats"]["sweeps"] == orc["sweeps"] and res["stats"]["edge_tests"] == orc["tests"]
    full = oracle.fixpoint(g.colour, edges, k)
    with kz.KernelGraph.from_synth(g, dense=False) as kg:
        for opts, lim in (({"schedule": "support"}, 0), ({}, 1), ({"schedule": "support"}, 1)):
            kg.reset().kernelize(path="sparse", max_sweeps=lim, **opts)
            alive, kept, _ = kg.fetch(allow=(kz.KZ_OK, kz.KZ_ERR_LIMIT))
            orc = oracle.fixpoint(g.colour, edges, k, max_sweeps=lim, raise_on_limit=False) if lim else full
            assert np.array_equal(alive, orc["vlive"]) and np.array_equal(kept, edges[orc["elive"].astype(bool)])
