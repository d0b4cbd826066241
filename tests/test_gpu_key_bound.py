"""bf16 attention and the key-norm bound.  A key that is not a number, in every kind of column of a tile (exponentials of either unit,
a tile's halves, the first half, which fixes the reference, and the last row): under the bound the same bits as without it.  The
bound switched off and on."""
import pytest
import torch

from paper_2603_05959_b200 import binding as B

pytestmark = pytest.mark.gpu


def _draw(rows, C, g):
    return torch.randn((rows, C), generator=g, device="cuda").bfloat16()


@pytest.mark.parametrize("row", [0, 5, 95, 96, 191, 192, 300, 301, 302, 303, 304, 305, 699])
def test_bounded_attention(row):
    M, N, H = 130, 700, 2
    g = torch.Generator(device="cuda").manual_seed(row)
    q, k, v = (_draw(r, H * 64, g) for r in (M, N, N))
    assert float(B.k_key_norm_bound(k, H).max()) < float("inf")
    k[row, 7] = float("nan")
    assert B.k_key_norm_bound(k, H).tolist()[0] == float("inf")
    got, want = (B.k_attention(q, k, v, H, bounded=b) for b in (True, False))
    assert torch.equal(got[:, :64].view(torch.int16), want[:, :64].view(torch.int16))
    assert bool(torch.isfinite(got[:, 64:]).all())       # (the other head)


@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_step(sign):
    """Through a cache: the key comes with a frame, attended to in that step and the next."""
    H, g = 2, torch.Generator(device="cuda").manual_seed(1)
    frames = [[_draw(66, H * 64, g) for _ in range(4)] for _ in range(14)]
    frames[11][1][37, 7] = sign * float("nan")
    outs = []
    for bound in (True, False):
        cache = B.OvggtCache(n_layers=1, n_heads=H, n_special=1, grid_h=5, grid_w=13, budget=1024, anchor_tokens=0, k_max=0)
        cache.set_key_bound(bound)
        outs.append([cache.layer_step(0, t, *x) for t, x in enumerate(frames)])
        cache.stats(0)
        cache.destroy()
    bits = lambda x: x[:, :64].contiguous().view(torch.int16)
    for t in (11, 12, 13):
        assert torch.equal(bits(outs[0][t]), bits(outs[1][t])), t
        assert bool(torch.isfinite(outs[0][t][:, 64:]).all())


def test_bound_off_and_on():
    """Keys that come while the bound is off are under it when it is on again."""
    H, g = 2, torch.Generator(device="cuda").manual_seed(2)
    frames = [[_draw(66, H * 64, g) for _ in range(4)] for _ in range(5)]
    frames[2][1][30:] *= 40                              # scores of some hundreds, behind the first half of a tile
    outs = []
    for on in ([True, True, False, True, True], [False] * 5):
        cache = B.OvggtCache(n_layers=1, n_heads=H, n_special=1, grid_h=5, grid_w=13, budget=1024, anchor_tokens=0, k_max=0)
        for t, x in enumerate(frames):
            cache.set_key_bound(on[t])
            out = cache.layer_step(0, t, *x)
        outs.append(out.double())
        cache.stats(0)
        cache.destroy()
    # probabilities and outputs are rounded to within 2^-9 of themselves on either side
    assert (outs[0] - outs[1]).norm() <= 2.0 ** -7 * outs[1].norm()
