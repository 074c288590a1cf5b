"""The host check of a caller's edge list: the first wrong edge in list order
decides, wherever it lies in the threads' runs."""
import numpy as np
import pytest

import paper_2212_00574_gb300 as kz

BAD = {"range_high": ((0, 1000), kz.KZ_ERR_VERTEX_RANGE), "range_low": ((-1, 5), kz.KZ_ERR_VERTEX_RANGE),
       "loop": ((7, 7), kz.KZ_ERR_SELF_LOOP), "colour": ((3, 6), kz.KZ_ERR_ILLEGAL_COLOURING)}


def _status(colour, edges):
    with pytest.raises(kz.KzError) as e:
        kz.kz_free_graph(kz.kz_load_graph(len(colour), 3, colour, edges))
        raise kz.KzError(kz.KZ_OK, "accepted")
    return e.value.status


@pytest.mark.parametrize("m", [1, 2, 2 * 262144 - 1, 2 * 262144, 3 * 262144 + 5, 9 * 262144])
def test_first_wrong_edge_decides(m):
    rng = np.random.default_rng(m)
    n = 1000
    colour = (np.arange(n) % 3).astype(np.int32)
    u = rng.integers(0, n - 2, m)
    edges = np.stack([u, u + 1 + rng.integers(0, 2, m)], axis=1).astype(np.int32)  # legal (duplicates come later)
    spots = sorted({0, m - 1, m // 2, m // 2 - 1, m // 3, m // 3 - 1, min(m - 1, 262143), min(m - 1, 262144)} - {-1})
    kinds = list(BAD)
    for i, at in enumerate(spots):
        (bad, want), (other, _) = BAD[kinds[i % 4]], BAD[kinds[(i + 1) % 4]]
        e = edges.copy()
        e[at] = bad
        assert _status(colour, e) == want
        if at + 1 < m:  # a later wrong edge of another kind changes nothing
            e[at + 1 + int(rng.integers(0, m - at - 1))] = other
            e[m - 1] = other
            assert _status(colour, e) == want
