"""What the scaffold's product refuses: other types than bf16 and sizes that do not fit, also through the models that use it."""
import gc

import pytest
import torch

from paper_2603_05959_b200 import binding as B
from paper_2603_05959_b200 import harness as H
from paper_2603_05959_b200 import inputs as gen

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def collected():
    yield
    gc.collect()                                         # (a raised error's frames hold tensors)


def _t(*shape, dtype=torch.bfloat16):
    return torch.zeros(shape, dtype=dtype, device="cuda")


@pytest.mark.parametrize("name", ["a", "w", "outs", "residual", "sum_out"])
@pytest.mark.parametrize("how", ["type", "size"])
def test_arguments(name, how):
    shapes = dict(a=(16, 64), w=(64, 32), outs=(16, 32), residual=(16, 32), sum_out=(16, 32))
    args = {k: _t(*s) for k, s in shapes.items()}
    st = torch.zeros(16, dtype=torch.int32, device="cuda")
    B.k_linear_bf16(args["a"], args["w"], (args["outs"],), residual=args["residual"], sum_out=args["sum_out"], status=st)
    r, c = shapes[name]
    args[name] = _t(r, c, dtype=torch.float32) if how == "type" else (_t(r, c + 8) if name == "a" else _t(r - 8, c))
    with pytest.raises(AssertionError):
        B.k_linear_bf16(args["a"], args["w"], (args["outs"],), residual=args["residual"], sum_out=args["sum_out"], status=st)


def test_models_refuse_other_types():
    cfg = gen.StreamConfig(name="types", n_layers=1, n_heads=2, grid_h=4, grid_w=5, budget=60, anchor_tokens=0)
    for model in (H.ProjectionStack(cfg, torch.device("cuda")), H.Aggregator(cfg, torch.device("cuda"))):
        x, conf = torch.zeros((cfg.tokens_per_frame, cfg.dim), device="cuda"), torch.zeros(20, device="cuda")
        with pytest.raises(AssertionError):
            if isinstance(model, H.Aggregator):
                model.frame(0, x, conf, 0.5, torch.cuda.current_stream())
            else:
                model.frame(0, x, [x.bfloat16()], conf, 0.5, torch.cuda.current_stream())
        model.destroy()
