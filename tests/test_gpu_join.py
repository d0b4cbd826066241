"""Parts of a split KV range joined inside the attention: edges of the 128-row query tile, of the KV tiles and of the number of
parts, and the ticket counters over several launches, against the fp64 oracle.  (fp32: every shape is joined by "attend", those of one
query tile also by "step".)"""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_2603_05959_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid,cached,heads", [((1, 1), 700, 16),      # one row
                                               ((1, 127), 1025, 3),    # a whole tile
                                               ((3, 43), 2049, 2),     # one row more; 11 and 12 parts
                                               ((3, 43), 2860, 2),     # the largest number of parts, 16, of one KV tile (fp32: of three)
                                               ((11, 35), 260, 5),     # few parts
                                               ((1, 126), 127, 1)],    # two KV tiles in one part: nothing to join (fp32: 4, then 6 parts)
                         ids=lambda x: str(x).replace(" ", ""))
@pytest.mark.parametrize("dtype", [B.DTYPE_BF16, B.DTYPE_F32], ids=["bf16", "f32"])
@pytest.mark.parametrize("fused", [False, True], ids=["attend", "step"])
def test_joined_parts(grid, cached, heads, dtype, fused):
    orc.set_threads(8)
    rng = np.random.default_rng(cached)
    n_special = 1 if grid != (1, 1) else 0
    M, C = n_special + grid[0] * grid[1], heads * 64
    cache = B.OvggtCache(n_layers=1, n_heads=heads, n_special=n_special, grid_h=grid[0], grid_w=grid[1], budget=cached + 2 * M,
                         anchor_tokens=0, k_max=0, protect_first_frame=0, dtype=dtype)
    td = torch.bfloat16 if dtype == B.DTYPE_BF16 else torch.float32
    draw = lambda rows: torch.from_numpy(rng.standard_normal((rows, C)).astype(np.float32)).to(td).cuda()
    f32 = lambda x: x.float().cpu().numpy()
    bits = lambda x: x.cpu().numpy() if td == torch.float32 else x.view(torch.int16).cpu().numpy().view(np.uint16)
    n0 = cached // M * M                                # whole frames
    k0, v0 = draw(n0), draw(n0)
    cache.import_(0, np.arange(n0), np.zeros(n0, np.uint8), np.zeros(n0, np.float32), bits(k0), bits(v0), n0 // M, 0)
    K, V = f32(k0), f32(v0)
    for t in range(2):                                  # the second launch finds the tickets as the first one left them
        q, k, v, resid = (draw(M) for _ in range(4))
        if fused:                                       # the attention beside the selection of the same step
            got = f32(cache.layer_step(0, n0 // M + t, q, k, v, resid)).astype(np.float64)
        else:
            got = f32(cache.layer_attend(0, n0 // M + t, q, k, v)).astype(np.float64)
            cache.layer_compress(0, n0 // M + t, resid)
        K, V = np.concatenate([K, f32(k)]), np.concatenate([V, f32(v)])
        ref = orc.attention(f32(q), K, V, heads, 64).astype(np.float64)
        # bf16: outputs are rounded to within 2^-8 of themselves, weights too, but independently of each other; fp32: a score
        # of up to 6 sigma carries a few roundings of 2^-24, weights, sums and outputs a few more
        tol = 2.0 ** -8 if dtype == B.DTYPE_BF16 else 2.0 ** -22 * (8 + 6)
        assert np.linalg.norm(got - ref) <= tol * np.linalg.norm(ref)
    cache.stats(0)                                      # (raises if a kernel has left a status)
    cache.destroy()
