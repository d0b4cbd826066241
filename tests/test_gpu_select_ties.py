"""The selection where its threshold bin is crowded: ties, near-ties and dense ranges, on one CTA and on a cluster, against a
stable sort.  (Survivors only: what the same launch leaves of the key sums is checked in test_gpu_key_sums.py.)"""
import numpy as np
import pytest
import torch

from paper_2603_05959_b200 import binding as B

pytestmark = pytest.mark.gpu


def _priorities(rng, n):
    few = rng.integers(0, 6, n).astype(np.float32)
    dense = (1 + 1e-3 * rng.random(n)).astype(np.float32)
    pair = np.where(rng.random(n) < 0.4, np.float32(1), np.nextafter(np.float32(1), np.float32(2)))
    far = rng.random(n) < 0.05                               # outliers, which stretch the range that the bins share
    spread = (rng.standard_normal(n) * 1e3).astype(np.float32)
    yield "all equal", np.ones(n, np.float32)
    yield "few values", few
    yield "few values and others near", np.where(far, few + np.float32(1e-4) * rng.random(n).astype(np.float32), few)
    yield "dense", np.where(far, spread, dense)
    yield "two neighbours", np.where(far, spread, pair)
    yield "copies", rng.permutation(np.repeat(rng.standard_normal(n // 3 + 1).astype(np.float32), 3)[:n])
    yield "no ties", spread


@pytest.mark.parametrize("grid", [(4, 25), (8, 50), (23, 31)], ids=["single", "cluster", "cluster-crowded"])
@pytest.mark.parametrize("compaction", [B.COMPACT_FILL_HOLES, B.COMPACT_STABLE_GATHER], ids=["holes", "stable"])
def test_crowded_threshold(grid, compaction):
    M, C = 1 + grid[0] * grid[1], 64
    budget = 4 * M
    cache = B.OvggtCache(n_layers=1, n_heads=1, n_special=1, grid_h=grid[0], grid_w=grid[1], budget=budget, anchor_tokens=0, k_max=0,
                         protect_first_frame=0, compaction=compaction)
    rng = np.random.default_rng(M)
    x = torch.from_numpy(rng.standard_normal((M, C)).astype(np.float32)).bfloat16().cuda()
    for t in range(4):
        cache.layer_step(0, t, x, x, x, x)
    for name, r in _priorities(rng, budget + M):
        t += 1
        cache.layer_step(0, t, x, x, x, x, score_override=torch.from_numpy(r).cuda())
        want = np.sort(np.argsort(-r, kind="stable")[:budget])
        assert np.array_equal(cache.last_selection(0)["survivors"], want), name
    cache.stats(0)                                           # (raises if a kernel has left a status)
    cache.destroy()
