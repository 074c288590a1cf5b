"""Which form AUTO takes in the tensor form's region, seen in the memory the
first run asks for (GPU only): the tensor form's operand matrix holds a byte a
pair of vertices, the pair form's rows and lists a quarter of that at most."""
import ctypes as C

import numpy as np
import pytest

import paper_2212_00574_gb300 as kz
from paper_2212_00574_gb300 import synth

pytestmark = pytest.mark.gpu


# either side of the lines: n = 4200 and 4400, an expected 7 or 30 common
# neighbours a class
@pytest.mark.parametrize("n,k,p,pairs", [(3100, 12, 0.2, False), (3100, 12, 0.1, True), (3080, 3, 0.2, False),
                                         (4150, 17, 0.21, False), (4250, 17, 0.21, True), (4250, 3, 0.2, False),
                                         (4450, 3, 0.2, True), (6200, 6, 0.2, True)])
def test_form_by_size_and_density(n, k, p, pairs):
    import torch
    g = synth.kpartite(n, k, p, 9500 + n, planted=True)
    asked = []

    def alloc(nbytes, stream, ctx):
        asked.append(nbytes)
        return int(torch.cuda.caching_allocator_alloc(int(nbytes), 0, int(stream or 0)))

    def free(ptr, nbytes, stream, ctx):
        torch.cuda.caching_allocator_delete(int(ptr))

    table = kz.kz_allocator(kz._ALLOC_FN(alloc), kz._FREE_FN(free), None)
    assert kz._lib().kz_set_allocator(C.byref(table)) == kz.KZ_OK
    try:
        with kz.KernelGraph.from_synth(g, dense=True) as kg:
            asked.clear()
            kg.kernelize()
            assert (max(asked) < n * n // 2) == pairs
            alive, edges, st = kg.fetch()
            assert st["path"] == 4
            kg.reset().kernelize(path="bitset")
            want_alive, want, want_st = kg.fetch()
    finally:
        kz.use_default_allocator()
    assert np.array_equal(alive, want_alive) and np.array_equal(edges, want)
    for f in ("sweeps", "passes", "edge_tests"):
        assert st[f] == want_st[f], f
