"""The device CSR build at the edges of its sort (GPU only): edge counts around
a tile of 4096 keys, vertex counts on either side of a digit and of the edge
count, edges in any order and direction, merged duplicates.  Bit-exact against
the oracle."""
import numpy as np
import pytest

import paper_2212_00574_gb300 as kz
from paper_2212_00574_gb300 import synth
from tests.test_gpu_parity import assert_parity

pytestmark = pytest.mark.gpu


def _graph(n, k, m, hubs, seed):
    """m edges: a clique over the classes, one end of the rest among `hubs` vertices."""
    rng = np.random.default_rng(seed)
    colour = (np.arange(n) % k).astype(np.int32)
    pairs = set()
    for a in range(k):
        for b in range(a + 1, k):
            pairs.add((n - k + a, n - k + b))
    pairs = set(list(sorted(pairs))[:m])
    while len(pairs) < m:
        a, b = sorted((int(rng.integers(0, hubs)), int(rng.integers(0, n))))
        if a != b and colour[a] != colour[b]:
            pairs.add((a, b))
    return synth.Graph(n=n, k=k, colour=colour, edges=np.array(sorted(pairs), np.int32).reshape(-1, 2), planted=[])


@pytest.mark.parametrize("n,k,m,hubs", [(5, 3, 1, 5), (257, 4, 2, 257), (256, 4, 4095, 256), (257, 4, 4096, 257),
                                        (300, 5, 4097, 300), (20000, 6, 8192, 3), (9000, 3, 4097, 9000),
                                        (65536, 5, 40000, 400), (65537, 5, 12289, 65537)])
@pytest.mark.parametrize("repeats", [False, True])
def test_build_matches_the_oracle(n, k, m, hubs, repeats):
    g = _graph(n, k, m, hubs, 9500 + m)
    rng = np.random.default_rng(m)
    edges = g.edges[rng.permutation(m)]
    if repeats:
        edges = np.concatenate([edges, edges[rng.integers(0, m, m // 3 + 1)]])[:, ::1]
    edges = np.where(rng.random(len(edges))[:, None] < 0.5, edges, edges[:, ::-1]).astype(np.int32)
    if repeats:
        with pytest.raises(kz.KzError) as e:
            kz.KernelGraph(n, k, g.colour, edges=edges)
        assert e.value.status == kz.KZ_ERR_DUPLICATE_EDGE
    with kz.KernelGraph(n, k, g.colour, edges=edges, flags=kz.KZ_DEDUP if repeats else 0) as kg:
        kg.kernelize(path="sparse")
        alive, kept, stats = kg.fetch()
        dv, de, vs = kg.trace()
    assert stats["m"] == m
    assert_parity(g, dict(alive=alive, edges=kept, stats=stats, dv=dv[:stats["sweeps"]], de=de[:stats["sweeps"]],
                          v_sweep=vs))
