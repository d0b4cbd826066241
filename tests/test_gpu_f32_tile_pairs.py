"""The fp32 attention with one and with two query tiles a CTA: frames of one tile, of pairs, of pairs and a half, KV ranges whole and
in parts that a kernel of its own merges (the parts joined inside: test_gpu_join.py), one to several KV tiles a part, against fp64."""
import pytest
import torch

from paper_2603_05959_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,H", [(256, 64, 1), (257, 128, 1), (255, 129, 2), (384, 700, 3), (385, 192, 16), (1374, 1374, 16),
                                   (1374, 5470, 2), (69, 325, 4), (640, 3000, 12), (1041, 1200, 16), (518, 64, 16)])
def test_tile_pairs(M, N, H):
    g = torch.Generator(device="cuda").manual_seed(M + N)
    q, k, v = (torch.randn((r, H * 64), generator=g, device="cuda") for r in (M, N, N))
    got = B.k_attention(q, k, v, H)
    s = torch.einsum("mhd,nhd->hmn", q.double().view(M, H, 64), k.double().view(N, H, 64)) / 8
    ref = torch.einsum("hmn,nhd->mhd", torch.softmax(s, 2), v.double().view(N, H, 64)).reshape(M, H * 64)
    # scores of up to about 6 carry a few roundings of 2^-24, weights, sums and outputs a few more
    assert (got.double() - ref).norm() <= 2.0 ** -22 * (8 + 6) * ref.norm()


# (frames whose halves and whose steps take different CTAs, or one of them joins its parts and the other merges them)
@pytest.mark.parametrize("grid,budget,heads", [((3, 43), 2049, 2), ((11, 35), 386, 5), ((14, 37), 1100, 12), ((28, 37), 2500, 4)])
@pytest.mark.parametrize("compaction", [B.COMPACT_FILL_HOLES, B.COMPACT_STABLE_GATHER], ids=["holes", "stable"])
def test_step_equals_its_halves(grid, budget, heads, compaction):
    M = 1 + grid[0] * grid[1]
    step, halves = (B.OvggtCache(n_layers=1, n_heads=heads, n_special=1, grid_h=grid[0], grid_w=grid[1], budget=budget, anchor_tokens=0,
                                 k_max=0, protect_first_frame=0, dtype=B.DTYPE_F32, compaction=compaction) for _ in range(2))
    g = torch.Generator(device="cuda").manual_seed(M)
    for t in range(-(-budget // M) + 2):
        q, k, v, resid = torch.randn((4, M, heads * 64), generator=g, device="cuda")
        got = step.layer_step(0, t, q, k, v, resid)
        want = halves.layer_attend(0, t, q, k, v)
        halves.layer_compress(0, t, resid)
        assert torch.equal(got, want), t
    for cache in (step, halves):
        cache.stats(0)                                   # (raises if a kernel has left a status)
        cache.destroy()
