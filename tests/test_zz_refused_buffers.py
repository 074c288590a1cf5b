"""Requests refused one after another while a schedule makes its buffers (GPU
only): the run returns KZ_ERR_OOM and gives back what it took, and the next run
of the handle finds nothing half made."""
import ctypes as C

import numpy as np
import pytest

import oracle
import paper_2212_00574_gb300 as kz
from paper_2212_00574_gb300 import synth

pytestmark = pytest.mark.gpu


class Refusing:
    """Serves requests through torch's caching allocator; from the last `start`
    on, the first `refuse` of them only (None: all)."""

    def __init__(self):
        import torch
        self.refuse, self.count, self.live = None, 0, {}

        def alloc(nbytes, stream, ctx):
            self.count += 1
            if self.refuse is not None and self.count > self.refuse:
                return None
            p = int(torch.cuda.caching_allocator_alloc(int(nbytes), 0, int(stream or 0)))
            self.live[p] = int(nbytes)
            return p

        def free(ptr, nbytes, stream, ctx):
            assert self.live.pop(int(ptr)) == nbytes
            torch.cuda.caching_allocator_delete(int(ptr))

        self.table = kz.kz_allocator(kz._ALLOC_FN(alloc), kz._FREE_FN(free), None)
        assert kz._lib().kz_set_allocator(C.byref(self.table)) == kz.KZ_OK

    def start(self, refuse):
        self.refuse, self.count = refuse, 0


@pytest.mark.parametrize("opts,dense", [({"path": "sparse", "schedule": "support"}, False),
                                        ({"dominance": 2, "path": "bitset"}, True)])
def test_every_request_refused_in_turn(opts, dense):
    # beyond the bitset remnant (33 colours), so that the support counts are built
    g = synth.tiny_random(9801, 1500, 33, 0.55, planted=True)
    want = oracle.fixpoint(g.colour, g.get_edges(), g.k)
    mem = Refusing()
    try:
        with kz.KernelGraph.from_synth(g, dense=dense) as kg:
            mem.start(None)
            kg.kernelize(**opts)
            total = mem.count
            ref_alive, ref_edges, _ = kg.fetch()
        assert total >= 2 and not mem.live
        if "dominance" not in opts:
            assert np.array_equal(ref_alive, want["vlive"])
            assert np.array_equal(ref_edges, g.get_edges()[want["elive"].astype(bool)])
        for refuse in range(total):
            mem.start(None)
            with kz.KernelGraph.from_synth(g, dense=dense) as kg:
                for _ in range(2):
                    held = dict(mem.live)
                    mem.start(refuse)
                    with pytest.raises(kz.KzError) as e:
                        kg.kernelize(**opts)
                    assert e.value.status == kz.KZ_ERR_OOM and mem.count >= refuse + 1
                    assert mem.live == held
                    mem.start(None)
                    kg.reset()
                kg.kernelize(**opts)
                alive, edges, _ = kg.fetch()
                assert np.array_equal(alive, ref_alive) and np.array_equal(edges, ref_edges)
            assert not mem.live
    finally:
        kz.use_default_allocator()


@pytest.mark.parametrize("opts", [{}, {"schedule": "support"}])
def test_pair_form_refused_leaves_the_tensor_form(opts):
    import torch
    g = synth.kpartite(3100, 17, 0.1, 9802, planted=True)
    with kz.KernelGraph.from_synth(g, dense=True) as kg:
        kg.kernelize(path="bitset")
        want_alive, want, want_st = kg.fetch()
    once = [None]
    asked = []

    def alloc(nbytes, stream, ctx):
        asked.append(nbytes)
        if once[0] is not None and len(asked) == once[0] + 1:
            return None  # this one only
        return int(torch.cuda.caching_allocator_alloc(int(nbytes), 0, int(stream or 0)))

    def free(ptr, nbytes, stream, ctx):
        torch.cuda.caching_allocator_delete(int(ptr))

    table = kz.kz_allocator(kz._ALLOC_FN(alloc), kz._FREE_FN(free), None)
    assert kz._lib().kz_set_allocator(C.byref(table)) == kz.KZ_OK
    operand = g.n * g.n // 2  # the tensor form's operands take more, the pair form's buffers less
    try:
        with kz.KernelGraph.from_synth(g, dense=True) as kg:
            asked.clear()
            kg.kernelize()
            total = len(asked)
            assert total >= 2 and max(asked) < operand
        for refuse in range(total):
            with kz.KernelGraph.from_synth(g, dense=True) as kg:
                asked.clear()
                once[0] = refuse
                kg.kernelize(**opts)
                once[0] = None
                assert max(asked) >= operand
                alive, edges, st = kg.fetch()
                assert np.array_equal(alive, want_alive) and np.array_equal(edges, want)
                assert st["sweeps"] == want_st["sweeps"] and st["path"] == 4
                asked.clear()
                kg.reset().kernelize()  # and once memory is there again, the pair form
                assert asked and max(asked) < operand
                alive, edges, st = kg.fetch()
                assert np.array_equal(edges, want) and st["edge_tests"] == want_st["edge_tests"]
    finally:
        kz.use_default_allocator()


# from the third pass on the runs of the pair form keep witnesses, in memory that
# they ask for once a run and do without when it is refused
@pytest.mark.parametrize("n,k,p", [(5200, 12, 0.11), (7001, 11, 0.09)])
def test_long_cascade_without_the_witnesses_memory(n, k, p):
    g = synth.kpartite(n, k, p, 9400 + n, planted=True)
    kz.use_default_allocator()
    mem = Refusing()
    try:
        with kz.KernelGraph.from_synth(g, dense=True) as kg:
            kg.kernelize(path="bitset")
            want_alive, want, want_st = kg.fetch()
            assert want_st["passes"] >= 4
            kg.reset().kernelize()
            mem.start(None)
            kg.reset().kernelize()
            assert mem.count == 1  # the witnesses; everything else is there
            held = dict(mem.live)
            mem.start(0)
            kg.reset().kernelize()
            assert mem.count == 1 and mem.live == held  # refused
            mem.start(None)
            alive, edges, st = kg.fetch()
        assert np.array_equal(alive, want_alive) and np.array_equal(edges, want)
        for f in ("sweeps", "passes", "edge_tests", "m_live"):
            assert st[f] == want_st[f], f
        assert not mem.live
    finally:
        kz.use_default_allocator()


@pytest.mark.parametrize("opts", [{"path": "tensor"}, {"path": "tensor", "tensor_precision": 1}])
def test_refused_runs_keep_no_memory(opts):
    g = synth.tiny_random(9803, 2500, 9, 0.2, planted=True)
    want = oracle.fixpoint(g.colour, g.get_edges(), g.k)
    mem = Refusing()
    try:
        with kz.KernelGraph.from_synth(g, dense=True) as kg:
            mem.start(None)
            kg.kernelize(**opts)
            total = mem.count
        assert total >= 1 and not mem.live
        with kz.KernelGraph.from_synth(g, dense=True) as kg:
            for refuse in range(total):
                before = dict(mem.live)
                mem.start(refuse)
                with pytest.raises(kz.KzError) as e:
                    kg.kernelize(**opts)
                assert e.value.status == kz.KZ_ERR_OOM and mem.live == before
            mem.start(None)
            kg.reset().kernelize(**opts)
            alive, edges, _ = kg.fetch()
        assert np.array_equal(alive, want["vlive"]) and np.array_equal(edges, g.get_edges()[want["elive"].astype(bool)])
        assert not mem.live
    finally:
        kz.use_default_allocator()
