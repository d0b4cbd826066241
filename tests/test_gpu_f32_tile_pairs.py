"""The fp32 attention, two query tiles a CTA: one tile, a pair, a pair and a half, with the parts merged, joined and whole, and
KV ranges of one to several tiles a part, against fp64."""
import pytest
import torch

from paper_2603_05959_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,H", [(256, 64, 1), (257, 128, 1), (255, 129, 2), (384, 700, 3), (385, 192, 16), (1374, 1374, 16),
                                   (1374, 5470, 2), (69, 325, 4), (640, 3000, 12)])
def test_tile_pairs(M, N, H):
    g = torch.Generator(device="cuda").manual_seed(M + N)
    q, k, v = (torch.randn((r, H * 64), generator=g, device="cuda") for r in (M, N, N))
    got = B.k_attention(q, k, v, H)
    s = torch.einsum("mhd,nhd->hmn", q.double().view(M, H, 64), k.double().view(N, H, 64)) / 8
    ref = torch.einsum("hmn,nhd->mhd", torch.softmax(s, 2), v.double().view(N, H, 64)).reshape(M, H * 64)
    # scores of up to about 6 carry a few roundings of 2^-24, weights, sums and outputs a few more
    assert (got.double() - ref).norm() <= 2.0 ** -22 * (8 + 6) * ref.norm()
