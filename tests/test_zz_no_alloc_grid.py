"""The grid form of kz_kernelize_dense_noalloc and its packer at the sizes
where they can go wrong (GPU only): around the one-CTA limit, ragged last row
groups, every class-word width, classes of several planes, a wider row pitch,
and garbage where the packer must not look."""
import numpy as np
import pytest

import paper_2212_00574_gb300 as kz
from paper_2212_00574_gb300 import synth

pytestmark = pytest.mark.gpu


def _run(n, k, colour, bits, max_sweeps=0):
    import torch
    dev = torch.device("cuda", 0)
    c = torch.from_numpy(np.ascontiguousarray(colour, np.int32)).to(dev)
    b = torch.from_numpy(np.ascontiguousarray(bits).view(np.int64)).to(dev)
    alive = torch.full((n,), 7, dtype=torch.uint8, device=dev)
    out = torch.full_like(b, -1)
    counts = torch.full((4,), -5, dtype=torch.int64, device=dev)
    st = kz.kz_kernelize_dense_noalloc(n, k, c.data_ptr(), b.data_ptr(), b.shape[1], max_sweeps, alive.data_ptr(),
                                       out.data_ptr(), counts.data_ptr())
    return st, alive.cpu().numpy(), out.cpu().numpy().view(np.uint64), counts.cpu().numpy()


@pytest.mark.parametrize("n,k,p", [(63, 5, 0.6), (64, 6, 0.6), (65, 6, 0.6), (95, 8, 0.55), (97, 9, 0.6), (129, 3, 0.2),
                                   (255, 16, 0.6), (257, 17, 0.6), (700, 24, 0.5), (1023, 25, 0.5), (1025, 7, 0.1),
                                   (2049, 32, 0.5), (4095, 4, 0.03), (4096, 20, 0.9)])
@pytest.mark.parametrize("limit", [0, 1])
def test_grid_matches_the_bitset_sweep(n, k, p, limit):
    g = synth.kpartite(n, k, p, 9700 + n, planted=True)
    bits = g.get_bits()
    with kz.KernelGraph(n, k, g.colour, bits=bits) as kg:
        kg.kernelize(path="bitset", max_sweeps=limit)
        alive, kept, st = kg.fetch_dense(allow=(kz.KZ_OK, kz.KZ_ERR_LIMIT))
    # two words of padding a row; the lower triangle, the diagonal and the
    # bits past n hold garbage
    rng = np.random.default_rng(n)
    wide = rng.integers(0, 1 << 63, size=(n, bits.shape[1] + 2), dtype=np.uint64)
    cols = np.arange(64 * bits.shape[1])
    upper = (cols[None, :] > np.arange(n)[:, None]) & (cols < n)
    mask = synth.bool_to_bits(upper)
    wide[:, :bits.shape[1]] = (wide[:, :bits.shape[1]] & ~mask) | (bits & mask)
    status, a, b, counts = _run(n, k, g.colour, wide, limit)
    assert status == st["status"] == int(counts[3])
    assert np.array_equal(a, alive)
    assert np.array_equal(b[:, :bits.shape[1]], kept) and not b[:, bits.shape[1]:].any()
    assert list(counts[:3]) == [st["sweeps"], st["passes"], st["edge_tests"]]
