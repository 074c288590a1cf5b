"""The pair form of the passes (what AUTO runs in the tensor form's region)
against the bitset sweep and the oracle (GPU only).  Bit-exact: survivors,
sweeps, passes, tests and per-sweep counts."""
import numpy as np
import pytest

import oracle
import paper_2212_00574_gb300 as kz
from paper_2212_00574_gb300 import synth
from tests.test_gpu_parity import assert_parity, gpu_run

pytestmark = pytest.mark.gpu


def _same(a, b):
    assert np.array_equal(a["alive"], b["alive"]) and np.array_equal(a["edges"], b["edges"])
    for f in ("sweeps", "passes", "edge_tests", "n_live", "m_live", "status"):
        assert a["stats"][f] == b["stats"][f], f
    for f in ("dv", "de", "v_sweep"):
        assert np.array_equal(a[f], b[f]), f


# widths of the staged words (4, 8, 16, 32), class counts that leave a last
# group part empty, one to many tiles, blocks of a few members
@pytest.mark.parametrize("n,k,p", [(3073, 5, 0.08), (3100, 17, 0.1), (3333, 12, 0.2), (4500, 18, 0.16), (6150, 3, 0.02),
                                   (6145, 4, 0.05), (6200, 33, 0.2), (7001, 64, 0.24), (9001, 17, 0.112),
                                   (12289, 7, 0.04)])
def test_pairs_match_the_bitset_sweep(n, k, p):
    g = synth.kpartite(n, k, p, 9100 + n, planted=True)
    a = gpu_run(g, dense=True)
    assert a["stats"]["path"] == 4
    _same(a, gpu_run(g, dense=True, path="bitset"))


# long cascades, whose passes from the third on keep witnesses: classes of 14 to
# 55 words (both block widths), lists rebuilt as edges go, twice on one handle,
# and a run cut off among those passes and continued
@pytest.mark.parametrize("n,k,p", [(5200, 12, 0.11), (7001, 11, 0.09), (6200, 4, 0.038), (7000, 4, 0.036),
                                   (9300, 6, 0.055)])
def test_long_cascades_match_the_bitset_sweep(n, k, p):
    g = synth.kpartite(n, k, p, 9400 + n, planted=True)
    want = gpu_run(g, dense=True, path="bitset")
    assert want["stats"]["sweeps"] >= 6
    with kz.KernelGraph.from_synth(g, dense=True) as kg:
        for _ in range(2):
            kg.reset().kernelize()
            alive, edges, st = kg.fetch()
            assert st["path"] == 4 and np.array_equal(alive, want["alive"]) and np.array_equal(edges, want["edges"])
            for f in ("sweeps", "passes", "edge_tests", "n_live", "m_live"):
                assert st[f] == want["stats"][f], f
        kg.reset().kernelize(max_sweeps=4)
        assert kg.stats(allow=(kz.KZ_ERR_LIMIT,))["sweeps"] == 4
        kg.kernelize()
        alive, edges, _ = kg.fetch()
        assert np.array_equal(alive, want["alive"]) and np.array_equal(edges, want["edges"])
    _same(gpu_run(g, dense=True), want)


@pytest.mark.parametrize("n,k,p", [(3080, 9, 0.09), (3300, 13, 0.11)])
def test_pairs_match_the_oracle(n, k, p):
    g = synth.kpartite(n, k, p, 9200 + n, planted=True)
    a = gpu_run(g, dense=True)
    assert a["stats"]["path"] == 4
    assert_parity(g, a)


def test_pairs_with_uneven_classes():
    # Zipf classes: one of many planes, several of a few members
    rng = np.random.default_rng(93)
    n, k = 3400, 9
    colour = synth.colours_zipf(rng, n, k, 1.6)
    iu, iv = np.triu_indices(n, 1)
    keep = (colour[iu] != colour[iv]) & (rng.random(len(iu)) < 0.13)
    edges = np.stack([iu[keep], iv[keep]], axis=1).astype(np.int32)
    g = synth.Graph(n=n, k=k, colour=colour, edges=edges, planted=[])
    a = gpu_run(g)
    assert a["stats"]["path"] == 4
    _same(a, gpu_run(g, path="bitset"))


def test_pairs_limits_continuation_and_other_options():
    g = synth.kpartite(4600, 12, 0.1, 94, planted=True)
    full = gpu_run(g, dense=True, path="bitset")
    assert full["stats"]["sweeps"] > 2
    with kz.KernelGraph.from_synth(g, dense=True) as kg:
        for lim in (1, 2):
            kg.reset().kernelize(max_sweeps=lim)
            st = kg.stats(allow=(kz.KZ_ERR_LIMIT,))
            assert st["path"] == 4 and st["sweeps"] == lim and st["status"] == kz.KZ_ERR_LIMIT
        # from the limited state to the fixpoint, there once more, and on the
        # other paths of the same handle
        for opts in ({}, {}, {"path": "bitset"}, {"path": "tensor"}, {"schedule": "support"}):
            kg.kernelize(**opts)
            alive, edges, _ = kg.fetch()
            assert np.array_equal(alive, full["alive"]) and np.array_equal(edges, full["edges"])
        kg.reset().kernelize(schedule="support")
        alive, edges, st = kg.fetch()
        assert np.array_equal(edges, full["edges"]) and st["sweeps"] == full["stats"]["sweeps"]
        # a clique size below k counts classes, not one: the tensor form
        for q in (11, 9):
            want = gpu_run(g, dense=True, path="bitset", clique_k=q)
            kg.reset().kernelize(clique_k=q)
            alive, edges, st = kg.fetch()
            assert np.array_equal(edges, want["edges"]) and st["sweeps"] == want["stats"]["sweeps"]
