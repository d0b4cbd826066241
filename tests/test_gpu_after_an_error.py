"""A call that fails on the host side of CUDA says so, and leaves nothing behind for the next one."""
import gc

import pytest
import torch

from paper_2603_05959_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def collected():
    yield
    gc.collect()                                         # (a raised error's frames hold a handle's workspace)


def test_a_failed_call_does_not_fail_the_next():
    wide = B.OvggtCache(n_layers=1, n_heads=1000, n_special=1, grid_h=2, grid_w=2, budget=12, anchor_tokens=0, k_max=0,
                        protect_first_frame=0)
    x = torch.randn((5, 64000), device="cuda").bfloat16()
    with pytest.raises(B.OvggtError):                    # 250 KB of key sums do not fit a CTA's shared memory
        for t in range(2):
            wide.layer_step(0, t, x, x, x, x)
    cache = B.OvggtCache(n_layers=1, n_heads=1, n_special=1, grid_h=9, grid_w=9, budget=200, anchor_tokens=0, k_max=0,
                         protect_first_frame=0)
    y = torch.randn((82, 64), device="cuda").bfloat16()
    assert B.k_row_norms(y).shape == (82,)
    for t in range(4):
        cache.layer_attend(0, t, y, y, y)
        cache.layer_compress(0, t, y)
    assert cache.stats(0)["n_cached"] == 200
    cache.destroy()
    wide.destroy()
