"""The network's entry points take any device fp32 buffers: views at every
offset of a larger buffer (GPU only).  The same operands in the same order, so
the logits are the same bits wherever the features lie."""
import numpy as np
import pytest

import paper_2212_00574_gb300 as kz
from paper_2212_00574_gb300 import learned

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [1, 31, 33, 1000, 70001])
def test_forward_takes_features_at_any_offset(rows):
    import torch
    rng = np.random.default_rng(rows)
    w = learned.init_weights(21) + rng.normal(0, 0.05, kz.KZ_MLP_PARAMS).astype(np.float32)
    x = torch.from_numpy(rng.normal(size=rows * 16).astype(np.float32)).cuda()
    m = kz.kz_model_create(w)
    try:
        got = []
        for offset in range(4):
            buf = torch.full((rows * 16 + 8,), float("nan"), device="cuda")
            buf[offset:offset + rows * 16] = x
            out = torch.full((rows + 8,), float("nan"), device="cuda")
            view = buf[offset:]
            assert view.data_ptr() % 16 == 4 * offset
            kz.kz_mlp_forward(m, view.data_ptr(), rows, out[offset:].data_ptr())
            out = out.cpu().numpy()
            assert np.isnan(out[:offset]).all() and np.isnan(out[offset + rows:]).all()
            got.append(out[offset:offset + rows])
    finally:
        kz.kz_model_free(m)
    assert np.isfinite(got[0]).all()
    for g in got[1:]:
        assert np.array_equal(g.view(np.int32), got[0].view(np.int32))
