"""The attention of the fused step, which starts behind the selection and reads rows that the front has just written over evicted
ones: many moves a step, every output against fp64 over the rows that the survivor lists name."""
import numpy as np
import pytest
import torch

from paper_2603_05959_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [B.DTYPE_F32, B.DTYPE_BF16], ids=["f32", "bf16"])
@pytest.mark.parametrize("grid,budget", [((8, 8), 256), ((23, 31), 2200)], ids=["one CTA selects", "a cluster selects"])
def test_outputs_while_rows_move(grid, budget, dtype):
    heads, M = 3, 5 + grid[0] * grid[1]
    cache = B.OvggtCache(n_layers=1, n_heads=heads, n_special=5, grid_h=grid[0], grid_w=grid[1], budget=budget, anchor_tokens=0, k_max=0,
                         protect_first_frame=0, dtype=dtype, score_mode=B.SCORE_RANDOM, random_seed=3)
    g = torch.Generator(device="cuda").manual_seed(budget)
    K = V = torch.empty((0, heads * 64), device="cuda", dtype=torch.float64)
    split = lambda x: x.view(-1, heads, 64).transpose(0, 1)
    got, want = [], []
    for t in range(16):
        q, k, v, resid = torch.randn((4, M, heads * 64), generator=g, device="cuda").to(B.torch_dtype(dtype))
        got.append(cache.layer_step(0, t, q, k, v, resid))
        K, V = torch.cat([K, k.double()]), torch.cat([V, v.double()])
        p = torch.softmax(split(q.double()) @ split(K).transpose(1, 2) / 8, -1)
        want.append((p @ split(V)).transpose(0, 1).reshape(M, -1))
        keep = torch.from_numpy(cache.last_selection(0)["survivors"].astype(np.int64)).cuda()
        K, V = K[keep], V[keep]
    # bf16: weights and outputs are rounded to 2^-8 of themselves, independently of each other; fp32: a score of up to 6 sigma
    # carries a few roundings of 2^-24, weights, sums and outputs a few more
    tol = 2.0 ** -8 if dtype == B.DTYPE_BF16 else 2.0 ** -22 * (8 + 6)
    for t, (a, b) in enumerate(zip(got, want)):
        assert torch.linalg.norm(a.double() - b) <= tol * torch.linalg.norm(b), t
    cache.stats(0)                                       # (raises if a kernel has left a status)
    cache.destroy()
