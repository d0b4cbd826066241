"""The camera head's attend half in one launch, its move and its selection of the one row that leaves: edges of the batches of
rows a CTA takes (32 or 16 rows at a time, eight of those in flight) and of the one-CTA selection, against fp64."""
import numpy as np
import pytest
import torch

from paper_2603_05959_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [B.DTYPE_BF16, B.DTYPE_F32], ids=["bf16", "f32"])
@pytest.mark.parametrize("compaction", [B.COMPACT_FILL_HOLES, B.COMPACT_STABLE_GATHER], ids=["holes", "stable"])
@pytest.mark.parametrize("budget,heads", [(4, 1), (15, 3), (31, 16), (32, 5), (255, 2), (256, 16), (511, 3), (1023, 1), (1024, 2),
                                          (5, 160), (5, 161), (5, 192)])    # (the most heads of one launch, more)
@pytest.mark.parametrize("mode", [B.SCORE_HYBRID, B.SCORE_RESIDUAL_STORED], ids=["hybrid", "stored"])   # (stored: nothing scored beside)
def test_token_stream(budget, heads, compaction, dtype, mode):
    cache = B.OvggtCache.camera(n_heads=heads, budget=budget, dtype=dtype, compaction=compaction, score_mode=mode)
    C, td = heads * 64, B.torch_dtype(dtype)
    g = torch.Generator(device="cuda").manual_seed(budget)
    draw = lambda *shape: torch.randn(shape, generator=g, device="cuda").to(td)
    if budget > 40:                                      # the cache as it is a few rows below its budget
        n0 = budget - 3
        k0, v0 = draw(n0, C), draw(n0, C)
        bits = lambda x: x.cpu().numpy() if td == torch.float32 else x.view(torch.int16).cpu().numpy().view(np.uint16)
        flags = np.zeros(n0, np.uint8)
        flags[0] = 1
        cache.import_(0, np.arange(n0), flags, np.zeros(n0, np.float32), bits(k0), bits(v0), n0, 0)
    else:
        n0 = 0
        k0, v0 = draw(0, C), draw(0, C)
    K, V, ids, flags = k0.double(), v0.double(), list(range(n0)), [1] + [0] * (n0 - 1) if n0 else []
    for t in range(n0, n0 + (9 if n0 else 2 * budget + 3)):
        q, k, v, r = (draw(1, C) for _ in range(4))
        out = cache.layer_attend(0, t, q, k, v)
        K, V, ids = torch.cat([K, k.double()]), torch.cat([V, v.double()]), ids + [t]
        s = torch.einsum("hd,nhd->hn", q.double().view(heads, 64), K.view(-1, heads, 64)) / 8
        ref = torch.einsum("hn,nhd->hd", torch.softmax(s, 1), V.view(-1, heads, 64)).reshape(1, C)
        # fp32 arithmetic on the inputs as they are: a few roundings of the scores (up to about 6), of weights, sums and outputs
        tol = 2.0 ** -8 if dtype == B.DTYPE_BF16 else 2.0 ** -22 * (8 + 6)
        assert (out.double() - ref).norm() <= tol * ref.norm(), t
        registered = t % 4 == 2 and t > 0 and flags.count(2) < 2
        cache.camera_compress(0, t, r, registered, -1)
        flags.append(1 if t == 0 else 2 if registered else 0)
        sel = cache.last_selection(0)
        if mode == B.SCORE_HYBRID and len(ids) > 1 and len(ids) - 1 > flags[:-1].count(1) + flags[:-1].count(2) + 1:
            c = K[:-1].sum(0)
            d = (1 - K[:-1] @ c / (K[:-1].norm(dim=1) * c.norm())).cpu().numpy()
            free = np.array(flags[:-1]) == 0
            want = 0.5 * (d - d[free].min()) / (d[free].max() - d[free].min())
            np.testing.assert_allclose(sel["r"][:-1][free], want[free], rtol=0, atol=2e-5, err_msg=str(t))
        if len(ids) > budget:                            # the row that leaves: the lowest priority as ranked here, of equal ones the last
            pr = np.where(np.array(flags) == 0, sel["r"], np.inf)
            gone = len(pr) - 1 - int(np.argmin(pr[::-1]))
            assert sel["survivors"].tolist() == [i for i in range(len(ids)) if i != gone], t
            stay = [i for i in range(len(ids)) if i != gone]
            K, V, ids, flags = K[stay], V[stay], [ids[i] for i in stay], [flags[i] for i in stay]
    ex = cache.export(0)
    assert ex["ids"].tolist() == ids and ex["flags"].tolist() == flags
    if td == torch.float32:
        assert np.array_equal(ex["k"], K.float().cpu().numpy()) and np.array_equal(ex["v"], V.float().cpu().numpy())
    cache.stats(0)                                       # (raises if a kernel has left a status)
    cache.destroy()
