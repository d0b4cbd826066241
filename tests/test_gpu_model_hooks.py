"""What a model's hook is given of a layer stays the hook's: it may be kept over later layers and frames."""
import gc

import pytest
import torch

from paper_2603_05959_b200 import harness as H
from paper_2603_05959_b200 import inputs as gen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("model", [H.ProjectionStack, H.Aggregator], ids=["stack", "aggregator"])
@pytest.mark.parametrize("matmul", ["library", "torch"])
def test_tapped_tensors_are_kept(model, matmul):
    cfg = gen.StreamConfig(name="hooks", n_layers=3, n_heads=2, grid_h=9, grid_w=15, budget=400, anchor_tokens=0)
    m = model(cfg, torch.device("cuda"), matmul=matmul)
    kept, seen = [], []

    def tap(t, l, *tensors):
        kept.append(tensors)
        seen.append([x.clone() for x in tensors])

    m.tap = tap
    g = torch.Generator(device="cuda").manual_seed(1)
    M = cfg.tokens_per_frame
    x, conf = torch.randn((2, M, cfg.dim), generator=g, device="cuda").bfloat16(), torch.rand(135, device="cuda")
    resid = [torch.randn((M, cfg.dim), generator=g, device="cuda").bfloat16() for _ in range(3)]
    for t in range(2):
        args = (x[t], conf, 0.9) if model is H.Aggregator else (x[t], resid, conf, 0.9)
        m.frame(t, *args, torch.cuda.current_stream())
    assert len(kept) == 6
    for a, b in zip(kept, seen):
        assert all(torch.equal(p, q) for p, q in zip(a, b))
    m.destroy()
    del m, tap, args
    gc.collect()                                         # (the hook and the model hold one another)
