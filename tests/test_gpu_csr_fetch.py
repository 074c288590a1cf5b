"""The fetch of a CSR state on either side of the line between the host's scan
and the device's gathering of the survivors (32,768 edges), with all edges, some
and none alive (GPU only)."""
import numpy as np
import pytest

import oracle
import paper_2212_00574_gb300 as kz
from paper_2212_00574_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [0, 1, 32767, 32768, 32769])
@pytest.mark.parametrize("k,keep", [(2, "all"), (3, "some"), (4, "none")])
def test_fetch_around_the_scan_line(m, k, keep):
    # a bipartite graph of m edges: k = 2 keeps every edge, k = 4 none; k = 3
    # keeps the edges between the two classes' vertices that share a neighbour of
    # the third, one vertex joined to the first 50 of each
    n = 401
    u, v = np.divmod(np.arange(m), 200)
    edges = np.stack([u, 200 + v], axis=1).astype(np.int32)
    colour = np.where(np.arange(n) < 200, 0, 1).astype(np.int32)
    if keep == "some":
        colour[400] = 2
        edges = edges[:max(m - 100, 0)]
        hub = np.stack([np.r_[0:50, 200:250], np.full(100, 400)], axis=1).astype(np.int32)
        edges = synth.canonical_edges(np.concatenate([edges, hub[:m - len(edges)]]))
    assert len(edges) == m
    g = synth.Graph(n=n, k=k, colour=colour, edges=edges, planted=[])
    orc = oracle.fixpoint(colour, edges, k)
    want = edges[orc["elive"].astype(bool)]
    assert len(want) == {"all": m, "none": 0}.get(keep, len(want))
    with kz.KernelGraph.from_synth(g, dense=False) as kg:
        kg.kernelize(path="sparse")
        alive, kept, st = kg.fetch()
        assert np.array_equal(alive, orc["vlive"]) and np.array_equal(kept, want) and st["m_live"] == len(want)
        part = kz.kz_fetch_kernel(kg.h, n, cap=7, allow=(kz.KZ_OK, kz.KZ_ERR_BUFFER))
        assert part[2]["m_live"] == len(want) and np.array_equal(part[1][:7], want[:7])
