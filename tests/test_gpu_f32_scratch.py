"""fp32 attention with a scratch pointer that 16-byte accesses could not use: taken, as it was when fp32 needed no scratch."""
import pytest
import torch

from paper_2603_05959_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("offset", [4, 8])
def test_scratch_of_any_alignment(offset):
    M, N, H = 130, 900, 2
    g = torch.Generator(device="cuda").manual_seed(offset)
    q, k, v = (torch.randn((r, H * 64), generator=g, device="cuda") for r in (M, N, N))
    scratch = torch.empty(B.lib().ovggt_k_attention_scratch_bytes(M, N, H) + 16, dtype=torch.uint8, device="cuda")
    status = torch.zeros(16, dtype=torch.int32, device="cuda")
    outs = [torch.empty_like(q) for _ in range(2)]
    for out, s in zip(outs, (scratch.data_ptr() + offset, None)):
        assert B.lib().ovggt_k_attention(q.data_ptr(), k.data_ptr(), v.data_ptr(), M, N, H, B.DTYPE_F32, out.data_ptr(), s,
                                         status.data_ptr(), torch.cuda.current_stream().cuda_stream) == 0
    assert torch.equal(*outs) and int(status[0]) == 0
