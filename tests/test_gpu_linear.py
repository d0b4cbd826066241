"""The scaffold's dense products: tile edges, every tile width, the fused epilogues."""
import pytest
import torch

from paper_2603_05959_b200 import binding as B

pytestmark = pytest.mark.gpu

# rows, columns, K: single partial tiles, ragged edges, few tiles (64 wide), one wave of 128
# and of 256 wide
SHAPES = [(1, 8, 64), (127, 72, 64), (129, 264, 192), (333, 512, 2048), (130, 768, 3072), (1041, 1024, 1024), (700, 2304, 768),
          (1041, 4096, 64)]


def _ab(M, N, K):
    g = torch.Generator(device="cuda")
    g.manual_seed(M + N + K)
    a = torch.randn((M, K), generator=g, device="cuda").bfloat16()
    w = (torch.randn((K, N), generator=g, device="cuda") * 0.05).bfloat16()
    return a, w, torch.randn((M, N), generator=g, device="cuda").bfloat16(), torch.zeros(16, dtype=torch.int32, device="cuda")


def _close(got, ref, terms):
    # the unit roundoff of bf16 (8 significant bits: 2^-8) per rounding, and the rounding of the fp32 accumulation
    torch.testing.assert_close(got.double(), ref, rtol=terms * 2.0 ** -8, atol=1e-3 * float(ref.abs().max()))


@pytest.mark.parametrize("M,N,K", SHAPES)
def test_linear_epilogues(M, N, K):
    a, w, x, st = _ab(M, N, K)
    ref = a.double() @ w.double()
    t, s = torch.empty_like(x), torch.empty_like(x)
    B.k_linear_bf16(a, w, (t,), residual=x, sum_out=s, status=st)
    _close(t, ref, 1)
    assert torch.equal(s, x + t)                       # the sum is taken of the rounded product
    B.k_linear_bf16(a, w, (t,), gelu=True, status=st)
    _close(t, torch.nn.functional.gelu((a.double() @ w.double()).bfloat16().double()), 3)
    if N % 24 == 0:
        parts = [torch.empty((M, N // 3), dtype=torch.bfloat16, device="cuda") for _ in range(3)]
        B.k_linear_bf16(a, w, parts, status=st)
        _close(torch.cat(parts, 1), ref, 1)
    assert int(st[0]) == 0


def test_gelu_over_its_range():
    """Every finite bf16 value through an identity product: the bf16 rounding of torch's GELU, tails included."""
    v = torch.arange(0, 0x7F80, dtype=torch.int16, device="cuda").view(torch.bfloat16)
    a = torch.cat([v, -v]).view(-1, 64)
    out = torch.empty_like(a)
    st = torch.zeros(16, dtype=torch.int32, device="cuda")
    B.k_linear_bf16(a, torch.eye(64, device="cuda").bfloat16(), (out,), gelu=True, status=st)
    assert torch.equal(out, torch.nn.functional.gelu(a))


def test_gelu_where_no_value_is_below_its_polynomial():
    """Every finite bf16 value from -3 on, without the others beside them that send a warp to the error functions."""
    v = torch.arange(0, 0x7F80, dtype=torch.int16, device="cuda").view(torch.bfloat16)
    v = torch.cat([v, -v[v <= 3]])
    a = torch.cat([v, v.new_zeros(-v.numel() % 64)]).view(-1, 64)
    out = torch.empty_like(a)
    st = torch.zeros(16, dtype=torch.int32, device="cuda")
    B.k_linear_bf16(a, torch.eye(64, device="cuda").bfloat16(), (out,), gelu=True, status=st)
    assert torch.equal(out, torch.nn.functional.gelu(a))
