"""The support schedule's counts on the CSR state (GPU only): graphs beyond
4096 vertices or 32 colours whose first sweeps are light, so that the counts are
built at once and kept up to date over many sweeps, recounted when a sweep is
heavy, cut off by sweep limits, taken up again and left for other paths.  Against
the oracle, sweep by sweep."""
import numpy as np
import pytest

import oracle
import paper_2212_00574_gb300 as kz
from paper_2212_00574_gb300 import synth

pytestmark = pytest.mark.gpu

SUPPORT = {"path": "sparse", "schedule": "support"}
# sweeps: 50 (light all along), 8 (some heavy: recounts), 10; and a first sweep
# that is heavy (counts after a plain pass)
GRAPHS = [(4200, 4, 0.045), (4300, 5, 0.055), (4500, 8, 0.1), (4200, 4, 0.04)]


def _state(g, orc):
    return orc["vlive"], g.get_edges()[orc["elive"].astype(bool)]


@pytest.mark.parametrize("n,k,p", GRAPHS)
def test_counts_follow_the_sweeps(n, k, p):
    g = synth.tiny_random(9700 + n, n, k, p, planted=True)
    orc = oracle.fixpoint(g.colour, g.get_edges(), k)
    want_alive, want = _state(g, orc)
    with kz.KernelGraph.from_synth(g, dense=False) as kg:
        for _ in range(2):
            kg.reset().kernelize(**SUPPORT)
            alive, kept, st = kg.fetch()
            dv, de, vs = kg.trace()
            assert np.array_equal(alive, want_alive) and np.array_equal(kept, want)
            assert st["sweeps"] == orc["sweeps"] and st["passes"] == orc["passes"] and st["m_live"] == len(want)
            assert np.array_equal(vs, orc["v_sweep"])
            for a, b in ((dv, orc["dv"]), (de, orc["de"])):
                assert list(a[:orc["sweeps"]]) == list(b[:orc["sweeps"]])
            # every live edge once, then only what lost a witness
            assert len(g.get_edges()) <= st["edge_tests"] < orc["tests"]


@pytest.mark.parametrize("n,k,p", GRAPHS[1:])
def test_counts_limits_reruns_and_other_paths(n, k, p):
    g = synth.tiny_random(9700 + n, n, k, p, planted=True)
    edges = g.get_edges()
    full = oracle.fixpoint(g.colour, edges, k)
    assert full["sweeps"] >= 6
    with kz.KernelGraph.from_synth(g, dense=False) as kg:
        for lim in (1, 2, 5):
            kg.reset().kernelize(max_sweeps=lim, **SUPPORT)
            alive, kept, st = kg.fetch(allow=(kz.KZ_OK, kz.KZ_ERR_LIMIT))
            orc = oracle.fixpoint(g.colour, edges, k, max_sweeps=lim, raise_on_limit=False)
            want_alive, want = _state(g, orc)
            assert st["sweeps"] == lim and st["status"] == kz.KZ_ERR_LIMIT
            assert np.array_equal(alive, want_alive) and np.array_equal(kept, want)
            # on from there, by counts or by another path, and by counts again
            for then in ((SUPPORT, SUPPORT), ({"path": "sparse"}, SUPPORT), ({"path": "bitset"}, SUPPORT),
                         ({"path": "bitset", "max_sweeps": 1}, SUPPORT)):
                kg.reset().kernelize(max_sweeps=lim, **SUPPORT)
                for opts in then:
                    kg.kernelize(**opts)
                alive, kept, _ = kg.fetch()
                assert np.array_equal(alive, full["vlive"])
                assert np.array_equal(kept, edges[full["elive"].astype(bool)])


@pytest.mark.parametrize("n,k,p", [(200, 4, 0.3), (2000, 6, 0.1), (4050, 5, 0.055)])
def test_sweeps_without_counts_test_what_plain_sweeps_test(n, k, p):
    # graphs within the bitset remnant: a plain pass, then the remnant
    g = synth.tiny_random(9700 + n, n, k, p, planted=True)
    orc = oracle.fixpoint(g.colour, g.get_edges(), k)
    assert orc["sweeps"] >= 2
    with kz.KernelGraph.from_synth(g, dense=False) as kg:
        kg.kernelize(**SUPPORT)
        alive, kept, st = kg.fetch()
    want_alive, want = _state(g, orc)
    assert np.array_equal(alive, want_alive) and np.array_equal(kept, want)
    assert [st["sweeps"], st["passes"], st["edge_tests"]] == [orc["sweeps"], orc["passes"], orc["tests"]]
