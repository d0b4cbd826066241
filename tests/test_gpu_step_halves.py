"""The fused step and its two halves are the same arithmetic: outputs bit for bit, frame by frame, from the first frame through
the one that fills the cache into the steady state."""
import numpy as np
import pytest
import torch

from paper_2603_05959_b200 import binding as B
from paper_2603_05959_b200 import inputs as gen

pytestmark = pytest.mark.gpu


# KV ranges that several rules of splitting cut differently: 1041 to 9566 rows under 16 heads, and a few of fewer heads
@pytest.mark.parametrize("grid,heads,budget,frames", [((37, 37), 16, 8192, 8), ((28, 37), 16, 3000, 4), ((23, 31), 5, 2200, 5)],
                         ids=["1374x16", "1041x16", "718x5"])
@pytest.mark.parametrize("compaction", [B.COMPACT_FILL_HOLES, B.COMPACT_STABLE_GATHER], ids=["holes", "stable"])
def test_step_equals_its_halves(grid, heads, budget, frames, compaction):
    cfg = gen.StreamConfig(name="halves", n_heads=heads, grid_h=grid[0], grid_w=grid[1], budget=budget, anchor_tokens=16,
                           min_anchor_interval=3)
    step, halves = (B.OvggtCache.from_stream(cfg, compaction=compaction) for _ in range(2))
    g = torch.Generator(device="cuda").manual_seed(heads)
    for t in range(frames):
        q, k, v, resid = torch.randn((4, cfg.tokens_per_frame, cfg.dim), generator=g, device="cuda").bfloat16()
        conf, rho = torch.rand(grid[0] * grid[1], generator=g, device="cuda"), 0.1
        got = step.layer_step(0, t, q, k, v, resid, conf, rho)
        want = halves.layer_attend(0, t, q, k, v)
        halves.layer_compress(0, t, resid, conf, rho)
        assert torch.equal(got, want), t
        assert np.array_equal(step.last_selection(0)["survivors"], halves.last_selection(0)["survivors"]), t
    for cache in (step, halves):
        cache.stats(0)                                   # (raises if a kernel has left a status)
        cache.destroy()
