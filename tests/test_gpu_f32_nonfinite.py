"""fp32 attention where numbers are infinite, not numbers, or beyond the largest bf16: what plain fp32 arithmetic gives, in one
part, in parts merged by a kernel and in parts joined inside."""
import numpy as np
import pytest
import torch

from paper_2603_05959_b200 import binding as B

pytestmark = pytest.mark.gpu

INF, BIG = float("inf"), 3.4e38                          # BIG: finite in fp32, above the largest bf16


def _spoil(kind, q, k, v, h):
    c = h * 64 + 5
    if kind == "infinite values":
        v[3, c], v[-1, c + 1] = INF, -INF
    elif kind == "large values":
        v[3, c] = BIG
    elif kind == "keys of weight 0":                     # scores of -inf for every query; one KV tile of 64 has no others
        q[:, c] = q[:, c].abs() + 0.1
        k[2, c] = k[-1, c] = -INF
        k[64:128, c] = -INF
    elif kind == "a query that is not a number":
        q[1, c] = float("nan")
    elif kind == "a score of +inf":
        q[:, c], k[2, c] = q[:, c].abs() + 0.1, INF


def _reference(q, k, v, heads):
    split = lambda x: x.double().view(-1, heads, 64).transpose(0, 1)
    p = torch.softmax(split(q) @ split(k).transpose(1, 2) / 8, -1)
    out = []                                             # (a matrix product may skip what it multiplies by 0: sum by rows)
    for ph, vh in zip(p, split(v)):
        out.append((ph[:, :, None] * vh[None]).sum(1))
    return torch.stack(out, 1).reshape(q.shape)


KINDS = pytest.mark.parametrize("kind", ["infinite values", "large values", "keys of weight 0", "a query that is not a number",
                                         "a score of +inf"])


@KINDS
@pytest.mark.parametrize("route", ["one part", "merged", "joined", "joined, one query tile"])
def test_nonfinite(kind, route):
    heads, M, n0 = 3, 130, 650                           # 780 rows: 13 tiles of 64, the last one ragged
    if route == "joined, one query tile":                # (which a CTA of two takes)
        M = 117
    g = torch.Generator(device="cuda").manual_seed(len(kind))
    q, k, v = (torch.randn((r, heads * 64), generator=g, device="cuda") for r in (M, n0 + M, n0 + M))
    _spoil(kind, q, k, v, 1)
    before = B.kernel_launches()
    if route.startswith("joined"):
        cache = B.OvggtCache(n_layers=1, n_heads=heads, n_special=0, grid_h=M // 13, grid_w=13, budget=n0 + M, anchor_tokens=0, k_max=0,
                             protect_first_frame=0, dtype=B.DTYPE_F32, score_mode=B.SCORE_RESIDUAL_STORED)
        rows = lambda x: x[:n0].cpu().numpy()
        cache.import_(0, np.arange(n0), np.zeros(n0, np.uint8), np.zeros(n0, np.float32), rows(k), rows(v), n0 // M, 0)
        before = B.kernel_launches() + 1                 # (of the frame's append)
        got = cache.layer_attend(0, n0 // M, q, k[n0:], v[n0:])
        launches = B.kernel_launches() - before
        cache.stats(0)
        cache.destroy()
    elif route == "merged":
        got = B.k_attention(q, k, v, heads)
        launches = B.kernel_launches() - before
    else:
        got = torch.empty_like(q)
        assert B.lib().ovggt_k_attention(q.data_ptr(), k.data_ptr(), v.data_ptr(), M, n0 + M, heads, B.DTYPE_F32, got.data_ptr(), None,
                                         None, torch.cuda.current_stream().cuda_stream) == 0
        launches = B.kernel_launches() - before
    assert launches == (2 if route == "merged" else 1)   # a merge is a launch of its own, so is nothing else
    want = _reference(q, k, v, heads)
    assert bool(torch.isfinite(want).all()) == (kind in ("large values", "keys of weight 0"))
    # entries of the size of 1, a few roundings of 2^-24 of up to 6-sigma scores; BIG weighs 1 / 780 and swamps its column
    scale = want.abs().nan_to_num(0, 0, 0).amax(0, keepdim=True).clamp(min=1)
    torch.testing.assert_close((got.double() / scale), want / scale, rtol=0, atol=1e-5, equal_nan=True)
