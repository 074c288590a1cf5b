"""The CSR path's passes at the places where they change form (GPU only):
oriented rows around the hash table's length, remnants that move to bitset
rows and remnants that cannot, sweep limits on either side of that move, and
reruns.  Bit-exact against the oracle."""
import numpy as np
import pytest

import oracle
import paper_2212_00574_gb300 as kz
from paper_2212_00574_gb300 import synth
from tests.test_gpu_parity import assert_parity, gpu_run

pytestmark = pytest.mark.gpu


# n above 4096 keeps the first passes off the bitset remnant; dense rows reach
# beyond 256 oriented neighbours; k = 33 never leaves the CSR passes
@pytest.mark.parametrize("n,k,p", [(4200, 4, 0.004), (4300, 6, 0.03), (4500, 9, 0.06), (5000, 33, 0.2), (900, 5, 0.75),
                                   (1100, 3, 0.5), (4097, 2, 0.002), (4400, 8, 0.13)])
@pytest.mark.parametrize("schedule", ["plain", "support"])
def test_random_graphs(n, k, p, schedule):
    g = synth.tiny_random(9300 + n, n, k, p, planted=True)
    res = gpu_run(g, path="sparse", schedule=schedule)
    if schedule == "support":
        res["stats"]["edge_tests"] = oracle.fixpoint(g.colour, g.get_edges(), k)["tests"]  # tests made, at most these
    assert_parity(g, res)


@pytest.mark.parametrize("k", [5, 12])
def test_power_law_graphs_through_every_limit(k):
    g = synth.chung_lu(30000, k, 24.0, 9400 + k)
    edges = g.get_edges()
    full = oracle.fixpoint(g.colour, edges, k)
    assert full["sweeps"] >= 3
    with kz.KernelGraph.from_synth(g, dense=False) as kg:
        for lim in range(1, min(full["sweeps"], 6) + 1):
            kg.reset().kernelize(path="sparse", max_sweeps=lim)
            alive, kept, st = kg.fetch(allow=(kz.KZ_OK, kz.KZ_ERR_LIMIT))
            dv, de, vs = kg.trace()
            orc = oracle.fixpoint(g.colour, edges, k, max_sweeps=lim, raise_on_limit=False)
            assert np.array_equal(alive, orc["vlive"]) and np.array_equal(kept, edges[orc["elive"].astype(bool)])
            assert np.array_equal(vs, orc["v_sweep"]) and list(de[:lim]) == list(orc["de"][:lim])
        for opts in ({"path": "sparse"}, {"path": "sparse"}, {"schedule": "support", "path": "sparse"}):
            kg.kernelize(**opts)  # on from the limited state, then from the fixpoint
            alive, kept, _ = kg.fetch()
            assert np.array_equal(alive, full["vlive"]) and np.array_equal(kept, edges[full["elive"].astype(bool)])
        for q in (k - 1, k - 2):  # a clique size below k stays on the CSR passes
            kg.reset().kernelize(path="sparse", clique_k=q)
            alive, kept, st = kg.fetch()
            orc = oracle.fixpoint(g.colour, edges, k, clique_k=q)
            assert np.array_equal(alive, orc["vlive"]) and np.array_equal(kept, edges[orc["elive"].astype(bool)])
            assert st["sweeps"] == orc["sweeps"] and st["edge_tests"] == orc["tests"]


def test_remnant_too_uneven_for_bitset_rows():
    # 3500 live vertices, one class of 3000 and 31 of sixteen: rows of 94 x 32
    # words exceed the scratch, so every pass stays on the CSR
    rng = np.random.default_rng(95)
    n, k = 3500, 32
    colour = np.where(np.arange(n) < 3000, 0, 1 + np.arange(n) % (k - 1)).astype(np.int32)
    iu = rng.integers(0, 3000, 60000)
    iv = rng.integers(3000, n, 60000)
    a = rng.integers(3000, n, 60000)
    e = np.concatenate([np.stack([iu, iv], 1), np.stack([iv, a], 1)])
    e = synth.canonical_edges(e[colour[e[:, 0]] != colour[e[:, 1]]])
    g = synth.Graph(n=n, k=k, colour=colour, edges=e, planted=[])
    assert_parity(g, gpu_run(g, path="sparse"))


def test_fetch_reports_the_size_and_fills_what_fits():
    g = synth.chung_lu(6000, 4, 20.0, 96)
    with kz.KernelGraph.from_synth(g, dense=False) as kg:
        kg.kernelize(path="sparse")
        alive, kept, st = kg.fetch()
        assert st["m_live"] == len(kept) > 8
        with pytest.raises(kz.KzError) as err:
            kz.kz_fetch_kernel(kg.h, g.n, cap=len(kept) - 3)
        assert err.value.status == kz.KZ_ERR_BUFFER
        _, part, _ = kz.kz_fetch_kernel(kg.h, g.n, cap=len(kept) - 3, allow=(kz.KZ_OK, kz.KZ_ERR_BUFFER))
        assert np.array_equal(part[:len(kept) - 3], kept[:-3])
