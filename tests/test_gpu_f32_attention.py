"""The fp32 attention on split bf16 operands: edges of its 128 x 64 tiles and of its KV splits, against the fp64 oracle."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_2603_05959_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,H,qscale", [(1, 1, 1, 1.0), (128, 64, 2, 1.0), (127, 63, 3, 1.0), (129, 65, 1, 4.0),
                                          (5, 128, 16, 1.0), (300, 2049, 2, 4.0), (64, 5000, 1, 1.0)])
@pytest.mark.parametrize("scratch", [True, False], ids=["split", "no-scratch"])
def test_fp32_attention_at_tile_edges(M, N, H, qscale, scratch):
    orc.set_threads(8)
    rng = np.random.default_rng(M * 7 + N)
    q, k, v = ((rng.standard_normal((r, H * 64)) * s).astype(np.float32) for r, s in ((M, qscale), (N, 1.0), (N, 1.0)))
    dq, dk, dv = (torch.from_numpy(x).cuda() for x in (q, k, v))
    if scratch:
        got = B.k_attention(dq, dk, dv, H)
    else:                                   # the C call takes fp32 without scratch and without a status word
        got = torch.empty_like(dq)
        assert B.lib().ovggt_k_attention(dq.data_ptr(), dk.data_ptr(), dv.data_ptr(), M, N, H, B.DTYPE_F32, got.data_ptr(),
                                         None, None, torch.cuda.current_stream().cuda_stream) == 0
    got = got.cpu().numpy().astype(np.float64)
    ref = orc.attention(q, k, v, H, 64).astype(np.float64)
    # a score s carries a few fp32 roundings (2^-24 |s| each), which reach its weight as they are; weights, sums and
    # outputs add a few more
    smax = max(1.0, float(np.abs(q).max() * np.abs(k).max()))
    tol = 2.0 ** -22 * (8 + min(smax, 6 * qscale))
    assert np.linalg.norm(got - ref) <= tol * np.linalg.norm(ref)
