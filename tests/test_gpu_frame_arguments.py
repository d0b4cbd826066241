"""Frame arguments as C converts them: a coverage ratio beyond fp32 is infinite (no anchor), an id beyond 64 bits wraps and is
refused as out of order, numbers as text or as tensors are numbers."""
import gc

import pytest
import torch

from paper_2603_05959_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def collected():
    yield
    gc.collect()                                         # (a raised error's frames hold tensors)


def test_conversions():
    cache = B.OvggtCache(n_layers=1, n_heads=1, n_special=1, grid_h=3, grid_w=3, budget=40, anchor_tokens=2, k_max=2,
                         min_anchor_interval=1, tau=0.5)
    x, conf = torch.randn((10, 64), device="cuda").bfloat16(), torch.rand(9, device="cuda")
    host = [torch.zeros(10, 64, dtype=torch.bfloat16) for _ in range(2)]
    for t, (rho, anchors) in enumerate([(0.1, 0), (1e39, 0), ("0.9", 0), (torch.tensor(0.1), 1), ("0.1", 2), (-1e39, 2)]):
        if t % 2:
            cache.layer_step(0, t, x, x, x, x, conf, rho)
        else:
            cache.layer_attend(0, t, x, x, x)
            cache.layer_compress(0, t, x, conf, rho)
        assert cache.stats(0)["n_active_anchors"] == anchors, rho
    calls = [lambda f: cache.layer_attend(0, f, x, x, x), lambda f: cache.layer_compress(0, f, x),
             lambda f: cache.layer_step(0, f, x, x, x, x),
             lambda f: cache.layer_step_host(0, f, host[0], host[0], host[0], host[0], None, 1e39, host[1])]
    for call in calls:
        for frame in (2 ** 63, 2 ** 64 + 1, -1):
            with pytest.raises(B.OvggtError):
                call(frame)
    cache.destroy()
