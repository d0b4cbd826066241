"""The attention under the key-norm bound where the bound decides whether the exponentials' cubic needs its clamp: query norms
that put the lowest possible exponent on either side of the cubic's range and the bound on either side of being taken at all,
and the columns past the last row, against fp64."""
import pytest
import torch

from paper_2603_05959_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [96, 97, 192, 500, 575, 576, 4000])
@pytest.mark.parametrize("scale", [0.0, 1.0, 3.0, 4.5, 5.0, 5.5, 6.0, 8.0])
def test_bounded_attention_over_query_norms(scale, N):
    M, H = 130, 2
    g = torch.Generator(device="cuda").manual_seed(N)
    q, k, v = (torch.randn((r, H * 64), generator=g, device="cuda") for r in (M, N, N))
    q = (q / q.view(M, H, 64).norm(dim=2).repeat_interleave(64, 1) * 8 * scale).bfloat16()
    k = (k / k.view(N, H, 64).norm(dim=2).repeat_interleave(64, 1) * 8).bfloat16()
    k[N // 2] = k[N // 2] * 0                            # a key of no length: score 0 under any bound
    k[N // 3, :64] = -q[5, :64] / max(scale, 1.0)        # the lowest score there can be, for one row
    v = v.bfloat16()
    got = B.k_attention(q, k, v, H, bounded=True).double()
    s = torch.einsum("mhd,nhd->hmn", q.double().view(M, H, 64), k.double().view(N, H, 64)) / 8
    ref = torch.einsum("hmn,nhd->mhd", torch.softmax(s, 2), v.double().view(N, H, 64)).reshape(M, H * 64)
    # probabilities and outputs are rounded to within 2^-9 of themselves, the cubic to within 1e-4
    assert (got - ref).norm() <= 2.0 ** -8 * ref.norm()
