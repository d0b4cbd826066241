"""Rows wider than the front's centroid can be in shared memory: modes that rank without it take any width, whatever other
handles the process has used; the others say so."""
import gc

import numpy as np
import pytest
import torch

from paper_2603_05959_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def collected():
    yield
    gc.collect()                                         # (a raised error's frames hold a handle's workspace)


def _run(heads, dtype, mode, frames=5):
    cache = B.OvggtCache(n_layers=1, n_heads=heads, n_special=1, grid_h=2, grid_w=2, budget=12, anchor_tokens=0, k_max=0,
                         protect_first_frame=0, dtype=dtype, score_mode=mode, alpha=0.0)
    g = torch.Generator(device="cuda").manual_seed(heads)
    held = np.zeros(0)
    for t in range(frames):
        q, k, v, resid = torch.randn((4, 5, heads * 64), generator=g, device="cuda").to(B.torch_dtype(dtype))
        resid *= torch.rand((5, 1), generator=g, device="cuda").to(resid.dtype)
        cache.layer_step(0, t, q, k, v, resid)
        held = np.concatenate([held, resid.double().norm(dim=1).cpu().numpy()])
        sel = cache.last_selection(0)
        if mode == B.SCORE_RESIDUAL_STORED:
            np.testing.assert_allclose(sel["r"], held, rtol=1e-5)
        keep = np.sort(np.argsort(-sel["r"], kind="stable")[:12])
        np.testing.assert_array_equal(sel["survivors"], keep)
        held = held[keep]
    assert cache.stats(0)["device_status"] == 0
    cache.destroy()


@pytest.mark.parametrize("dtype", [B.DTYPE_BF16, B.DTYPE_F32], ids=["bf16", "f32"])
def test_wide_rows_beside_narrow_ones(dtype):
    for heads in (4, 193, 908, 1000):                    # 1, 48, 227 and 250 KB of centroid
        _run(heads, dtype, B.SCORE_RESIDUAL_STORED)
    for heads in (4, 193, 908):
        _run(heads, dtype, B.SCORE_HYBRID)
    with pytest.raises(B.OvggtError):
        _run(1000, dtype, B.SCORE_HYBRID)
    torch.cuda.synchronize()
