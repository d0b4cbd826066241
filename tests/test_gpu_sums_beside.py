"""The key sums that a fused step's selection leaves for the attention beside it, against the same stream in halves (bit for bit)
and against fp64: through the priorities of the cached rows, on every frame, over attentions of one wave of CTAs and of
several, narrow rows and rows of more columns than a launch has warps for, the filling of the cache, an export's moves, an
import, and the refresh of the sums."""
import numpy as np
import pytest
import torch

from paper_2603_05959_b200 import binding as B
from paper_2603_05959_b200 import inputs as gen

pytestmark = pytest.mark.gpu


def _cached_priorities(keys, ids, beta):
    """Eq. 7's priorities of the cached rows (none of them protected) in fp64, from their keys."""
    k = keys[ids].astype(np.float64)
    c = k.sum(0)
    d = 1.0 - k @ c / (np.linalg.norm(k, axis=1) * np.linalg.norm(c))
    return (1.0 - beta) * (d - d.min()) / (d.max() - d.min())


@pytest.mark.parametrize("grid,heads,budget,frames", [((37, 37), 16, 6000, 9),     # three waves of CTAs
                                                      ((37, 37), 8, 9000, 10),     # two
                                                      ((23, 31), 12, 2500, 8),     # one, joined inside
                                                      ((28, 37), 20, 4200, 8),     # 320 groups of four columns
                                                      ((31, 33), 1, 5000, 10),     # sixteen groups of four columns
                                                      ((13, 11), 2, 1100, 72)],    # the sums afresh on the way
                         ids=lambda x: str(x).replace(" ", ""))
def test_sums_beside_the_attention(grid, heads, budget, frames):
    cfg = gen.StreamConfig(name="beside", n_heads=heads, grid_h=grid[0], grid_w=grid[1], budget=budget, anchor_tokens=0,
                           protect_first_frame=0)
    step, halves = (B.OvggtCache.from_stream(cfg) for _ in range(2))
    M = cfg.tokens_per_frame
    g = torch.Generator(device="cuda").manual_seed(budget)
    keys = np.zeros((frames * M, cfg.dim), np.float32)
    for t in range(frames):
        q, k, v, resid = torch.randn((4, M, cfg.dim), generator=g, device="cuda").bfloat16()
        keys[t * M:(t + 1) * M] = k.float().cpu().numpy()
        ids = step.export(0, with_kv=t == 5)["ids"] if t in (3, 5) or t > 6 else None      # (an export carries out the pending moves)
        if t == 6:                                       # what an import leaves has no sums
            ex = step.export(0)
            for cache in (step, halves):
                cache.import_(0, ex["ids"], ex["flags"], ex["stored"], ex["k"], ex["v"], t, 0)
        got = step.layer_step(0, t, q, k, v, resid)
        want = halves.layer_attend(0, t, q, k, v)
        halves.layer_compress(0, t, resid)
        assert torch.equal(got, want), t
        a, b = step.last_selection(0), halves.last_selection(0)
        assert np.array_equal(a["survivors"], b["survivors"]), t
        assert np.array_equal(a["r"].view(np.uint32), b["r"].view(np.uint32)), t
        if ids is not None:
            np.testing.assert_allclose(a["r"][:len(ids)], _cached_priorities(keys, ids, 0.5), rtol=0, atol=2e-5, err_msg=str(t))
    for cache in (step, halves):
        cache.stats(0)                                   # (raises if a kernel has left a status)
        cache.destroy()
