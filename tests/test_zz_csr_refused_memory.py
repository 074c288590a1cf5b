"""Device memory refused while a CSR handle is at work (GPU only).  The lists
and the bitset remnant that the CSR path asks for make it faster and change
nothing else: a fetch, and a run, without them give the same kernel."""
import ctypes as C

import numpy as np
import pytest

import oracle
import paper_2212_00574_gb300 as kz
from paper_2212_00574_gb300 import synth
from tests.test_zz_allocator_failure import _install

pytestmark = pytest.mark.gpu


def _graph():
    # 59,000 edges, of which a few thousand survive
    return synth.chung_lu(6000, 4, 20.0, 96)


# requests the fetch may make: none, the first (the counts; not the survivors)
@pytest.mark.parametrize("granted", [0, 1])
def test_fetch_without_device_memory(granted):
    g = _graph()
    orc = oracle.fixpoint(g.colour, g.get_edges(), g.k)
    want = g.get_edges()[orc["elive"].astype(bool)]
    assert len(want) > 8
    kz.use_default_allocator()
    with kz.KernelGraph.from_synth(g, dense=False) as kg:
        kg.kernelize(path="sparse")
        try:
            for fetch in ("edges", "part", "dense"):
                a, state = _install(granted)
                if fetch == "edges":
                    alive, kept, st = kg.fetch()
                    assert np.array_equal(kept, want) and st["m_live"] == len(want)
                elif fetch == "part":
                    alive, kept, st = kz.kz_fetch_kernel(kg.h, g.n, cap=5, allow=(kz.KZ_OK, kz.KZ_ERR_BUFFER))
                    assert np.array_equal(kept[:5], want[:5]) and st["m_live"] == len(want)
                else:
                    alive, bits, st = kg.fetch_dense()
                    assert np.array_equal(synth.bits_to_edges(bits, g.n), want)
                assert np.array_equal(alive, orc["vlive"])
                assert not state["live"]
        finally:
            kz.use_default_allocator()


@pytest.mark.parametrize("schedule", ["plain", "support"])
def test_run_without_the_remnants_memory(schedule):
    import torch
    g = _graph()
    orc = oracle.fixpoint(g.colour, g.get_edges(), g.k)
    running, refused = [], []

    def alloc(nbytes, stream, ctx):
        if running and nbytes > 8 << 20:  # the remnant's rows; nothing else of this run is as large
            refused.append(nbytes)
            return None
        return int(torch.cuda.caching_allocator_alloc(int(nbytes), 0, int(stream or 0)))

    def free(ptr, nbytes, stream, ctx):
        torch.cuda.caching_allocator_delete(int(ptr))

    table = kz.kz_allocator(kz._ALLOC_FN(alloc), kz._FREE_FN(free), None)
    assert kz._lib().kz_set_allocator(C.byref(table)) == kz.KZ_OK
    try:
        with kz.KernelGraph.from_synth(g, dense=False) as kg:
            running.append(1)
            kg.kernelize(path="sparse", schedule=schedule)
            running.clear()
            alive, kept, st = kg.fetch()
            dv, de, vs = kg.trace()
    finally:
        kz.use_default_allocator()
    assert refused  # asked for and refused
    assert np.array_equal(alive, orc["vlive"]) and np.array_equal(kept, g.get_edges()[orc["elive"].astype(bool)])
    assert st["sweeps"] == orc["sweeps"] and np.array_equal(vs, orc["v_sweep"])
    assert list(de[:st["sweeps"]]) == list(orc["de"][:st["sweeps"]])
