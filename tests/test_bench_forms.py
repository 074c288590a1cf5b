"""What the benchmark says of the pair form's runs (CPU only)."""
import os
import sys
from types import SimpleNamespace

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import bench  # noqa: E402
import paper_2212_00574_gb300 as kz  # noqa: E402


def _run(n, k, density, **over):
    g = SimpleNamespace(n=n, k=k, colour=np.arange(n) % k)
    sizes = np.bincount(g.colour, minlength=k).astype(float)
    st = {"path": 4, "k": k, "clique_k": k, "m": int(density * (n * n - (sizes ** 2).sum()) / 2)}
    args = SimpleNamespace(path="auto", tensor_precision="fp8")
    st.update({f: v for f, v in over.items() if f in st})
    for f, v in over.items():
        if f not in st:
            setattr(args, f, v)
    return g, st, args


@pytest.mark.parametrize("run,name", [(_run(32768, 24, 0.07), "pairs"), (_run(32768, 24, 0.07, clique_k=23), "tensor"),
                                      (_run(32768, 24, 0.07, tensor_precision="bf16"), "tensor"),
                                      (_run(3100, 12, 0.2), "tensor"), (_run(3100, 12, 0.1), "pairs")])
def test_form_name(run, name):
    g, st, args = run
    assert bench.form_name(kz, g, st, args) == name
    st["path"] = 1
    assert bench.form_name(kz, g, st, args) == "bitset"


def test_pair_launches():
    # rows, lists, pairs, commit, finish; then lists counted and built, and no more
    assert [bench.pair_launches(p) for p in (1, 2, 3, 4)] == [6, 11, 17, 21]
