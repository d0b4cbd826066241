"""Steps at the largest budgets a handle accepts, where the selection's arrays share their shared memory: small frames, whose
key sums are then taken afresh, and frames that make up a seventh of the cache.  Everything is recomputed on the host from
the keys that the survivor lists name."""
import numpy as np
import pytest
import torch

from paper_2603_05959_b200 import binding as B
from paper_2603_05959_b200 import inputs as gen

from test_gpu_stream import R_ATOL

pytestmark = pytest.mark.gpu


def _minmax(x):
    return (x - x.min()) / (x.max() - x.min())


def _smoothed(s, n_special, h, w, alpha=0.5):
    e = np.exp(-0.5 * np.array([1.0, 0.0, 1.0]))
    g, p = np.outer(e, e), np.pad(s[n_special:].reshape(h, w), 1, mode="edge")
    conv = sum(g[y, x] / g.sum() * p[y:y + h, x:x + w] for y in range(3) for x in range(3))
    return np.concatenate([s[:n_special], (alpha * conv + (1 - alpha) * s[n_special:].reshape(h, w)).ravel()])


@pytest.mark.parametrize("grid,candidates", [((8, 8), 82912), ((37, 37), 78624), ((64, 128), 56320)], ids=["69", "1374", "8197"])
@pytest.mark.parametrize("compaction", [B.COMPACT_FILL_HOLES, B.COMPACT_STABLE_GATHER], ids=["holes", "stable"])
def test_steps_at_the_largest_budget(grid, candidates, compaction):
    n_special, C, A = 5, 64, 7
    M = n_special + grid[0] * grid[1]
    n = budget = candidates - M
    cache = B.OvggtCache(n_layers=1, n_heads=1, n_special=n_special, grid_h=grid[0], grid_w=grid[1], budget=budget, anchor_tokens=A,
                         k_max=2, min_anchor_interval=1, tau=0.5, protect_first_frame=0, compaction=compaction)
    rng = np.random.default_rng(M)
    draw = lambda rows: gen.round_to_dtype(rng.standard_normal((rows, C), dtype=np.float32), gen.DTYPE_BF16)
    dev = lambda x: torch.from_numpy(x).bfloat16().cuda()
    keys, held = draw(n), np.zeros(n, np.int64)          # held: the frame whose anchor a row is, or 0
    bits = gen.bf16_round_bits(keys)
    cache.import_(0, np.arange(n), np.zeros(n, np.uint8), np.zeros(n, np.float32), bits, bits, n // M + 1, 0)
    active = []
    for i in range(5):
        t = n // M + 1 + i
        k, resid, conf = draw(M), draw(M), rng.random(grid[0] * grid[1], dtype=np.float32)
        rho = 0.1 if i != 2 else 0.9                     # every frame but one becomes an anchor; the third demotes the first
        cache.layer_step(0, t, dev(k), dev(k), dev(k), dev(resid), torch.from_numpy(conf).cuda(), rho)
        new = np.zeros(M, np.int64)
        if rho < 0.5:
            new[n_special + np.argsort(-conf, kind="stable")[:A]] = t
            active = (active + [t])[-2:]
        held = np.concatenate([held, new])
        protected = np.isin(held, active)
        s = keys.astype(np.float64).sum(0)
        d = 1 - keys @ s / (np.linalg.norm(keys.astype(np.float64), axis=1) * np.linalg.norm(s))
        x = _smoothed(np.linalg.norm(resid.astype(np.float64), axis=1), n_special, *grid)
        r = np.full(n + M, np.inf)
        old, fresh = ~protected[:n], ~protected[n:]
        r[:n][old] = 0.5 * _minmax(d[old])
        r[n:][fresh] = 0.5 * _minmax(x[fresh])
        sel = cache.last_selection(0)
        assert np.array_equal(np.isinf(sel["r"]), protected)
        np.testing.assert_allclose(sel["r"][~protected], r[~protected], rtol=0, atol=R_ATOL)
        want = np.sort(np.argsort(-sel["r"], kind="stable")[:budget])
        np.testing.assert_array_equal(sel["survivors"], want)
        keys, held = np.concatenate([keys, k])[want], held[want]
    ex = cache.export(0)
    assert np.array_equal(gen.bf16_bits_to_f32(ex["k"]), keys)
    assert cache.stats(0)["device_status"] == 0
    cache.destroy()
