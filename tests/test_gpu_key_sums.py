"""The key column sums that the selection continues from step to step (+ admitted - evicted keys), on the cluster kernel: they are
seen through the diversity of the cached rows, so through the library's own priorities, on every frame.  Long streams across
the refreshes, and streams whose selection ends in ties, where which tied rows stay is settled CTA by CTA."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_2603_05959_b200 import binding as B
from paper_2603_05959_b200 import inputs as gen
from paper_2603_05959_b200.stream import DeviceFrame

from test_gpu_stream import R_ATOL, run_teacher_forced

pytestmark = pytest.mark.gpu

LAYOUTS = pytest.mark.parametrize("compaction", [B.COMPACT_FILL_HOLES, B.COMPACT_STABLE_GATHER], ids=["holes", "stable"])
# 748 candidates, 94 a CTA: the frame's 148 rows lie in the last two CTAs, and 94 tied ones crowd a CTA's list of 64
MID = gen.StreamConfig(name="sums", n_heads=2, grid_h=13, grid_w=11, budget=600, anchor_tokens=7, min_anchor_interval=20, tau=0.5)


def _flat_residuals(monkeypatch):
    """Residual rows of zero norm: Eq. 7's zero range, so all new rows tie at priority 0.  (Zero, not just equal: the 3x3 sums
    of other equal norms differ from those by a rounding, about 1e-7 of them, which Eq. 7 stretches over its whole range.)"""
    draw = gen.frame_inputs

    def flat(cfg, frame, layer=0, fields=None):
        fi = draw(cfg, frame, layer, fields)
        fi.resid = np.zeros_like(fi.resid)
        return fi

    monkeypatch.setattr(gen, "frame_inputs", flat)


@LAYOUTS
def test_sums_follow_a_long_stream_across_refreshes(compaction):
    cfg = MID.replace(n_frames=150)
    layer = run_teacher_forced(cfg, cfg.n_frames, attn_frames=set(), export_every=50, compaction=compaction)
    assert layer.evicted_total > 100 * cfg.tokens_per_frame


@LAYOUTS
@pytest.mark.parametrize("ties", ["beta 0", "zero norms"])
def test_sums_where_all_new_rows_tie(ties, compaction, monkeypatch):
    cfg = MID.replace(n_frames=70, beta=0.0) if ties == "beta 0" else MID.replace(n_frames=70)
    if ties == "zero norms":
        _flat_residuals(monkeypatch)
    run_teacher_forced(cfg, cfg.n_frames, attn_frames=set(), export_every=35, compaction=compaction)


@LAYOUTS
def test_sums_of_a_free_run_whose_threshold_is_a_tie(compaction):
    """beta = 0 without given priorities: every evictable row of the frame and the least diverse cached row are at 0, which is
    the threshold from the first eviction on; the lowest positions among them stay."""
    cfg = MID.replace(n_frames=40, beta=0.0)
    layer, cache = orc.OracleLayer.from_stream(cfg), B.OvggtCache.from_stream(cfg, compaction=compaction)
    for t in range(cfg.n_frames):
        fi = gen.frame_inputs(cfg, t)
        df = DeviceFrame(cfg, fi, "cuda")
        layer.attend(t, fi.q, fi.k, fi.v, compute=False)
        ref = layer.compress(fi.resid, fi.conf, fi.rho)
        cache.layer_step(0, t, df.q, df.k, df.v, df.resid, df.conf, df.rho)
        sel = cache.last_selection(0)
        np.testing.assert_array_equal(sel["survivors"], ref["survivors"], err_msg=f"frame {t}")
        fin = np.isfinite(ref["r"])
        np.testing.assert_allclose(sel["r"][fin], ref["r"][fin], rtol=0, atol=R_ATOL, err_msg=f"frame {t}")
    assert cache.stats(0)["device_status"] == 0
    cache.destroy()


@LAYOUTS
@pytest.mark.parametrize("values", [1, 2, 6], ids=["all equal", "two values", "six values"])
def test_sums_after_given_priorities_with_ties(values, compaction):
    """Tied overrides every other step; the cache's keys are followed on the host through the survivors."""
    grid, budget, C, beta = (23, 31), 2860, 128, 0.5
    M = 2 + grid[0] * grid[1]
    cache = B.OvggtCache(n_layers=1, n_heads=2, n_special=2, grid_h=grid[0], grid_w=grid[1], budget=budget, anchor_tokens=0, k_max=0,
                         protect_first_frame=0, beta=beta, compaction=compaction)
    rng = np.random.default_rng(values)
    keys = np.zeros((0, C), np.float32)
    for t in range(16):
        x = [gen.round_to_dtype(rng.standard_normal((M, C), dtype=np.float32), gen.DTYPE_BF16) for _ in range(2)]
        k, resid = (torch.from_numpy(y).bfloat16().cuda() for y in x)
        n = len(keys)
        ov = rng.integers(0, values, n + M).astype(np.float32) if t % 2 else None
        cache.layer_step(0, t, k, k, k, resid, score_override=None if ov is None else torch.from_numpy(ov).cuda())
        sel = cache.last_selection(0)
        if n:
            s = keys.astype(np.float64).sum(0)
            d = 1 - keys @ s / (np.linalg.norm(keys.astype(np.float64), axis=1) * np.linalg.norm(s))
            np.testing.assert_allclose(sel["r"][:n], (1 - beta) * (d - d.min()) / (d.max() - d.min()), rtol=0, atol=R_ATOL,
                                       err_msg=f"frame {t}")
        if ov is not None:
            want = np.sort(np.argsort(-ov, kind="stable")[:budget])
            np.testing.assert_array_equal(sel["survivors"], want, err_msg=f"frame {t}")
        keys = np.concatenate([keys, x[0]])[sel["survivors"]]
    assert cache.stats(0)["device_status"] == 0
    cache.destroy()
