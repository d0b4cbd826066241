"""Two copies of the library in one process (an application's and a plug-in's, say) do not share state: each launches its kernels."""
import ctypes as C
import shutil

import pytest
import torch

from paper_2603_05959_b200 import binding as B

pytestmark = pytest.mark.gpu


def test_each_copy_launches_its_kernels(tmp_path):
    copies = []
    for i in range(2):
        path = str(tmp_path / ("copy%d.so" % i))
        shutil.copy(B.LIB_PATH, path)
        copies.append(C.CDLL(path))
    M, N, H = 130, 700, 2
    stream = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    p = lambda t: C.c_void_p(t.data_ptr())
    scratch = torch.empty(B.lib().ovggt_k_attention_scratch_bytes(M, N, H), dtype=torch.uint8, device="cuda")
    status = torch.zeros(16, dtype=torch.int32, device="cuda")
    g = torch.Generator(device="cuda").manual_seed(1)
    for dtype in (B.DTYPE_BF16, B.DTYPE_F32):
        q, k, v = (torch.randn((r, H * 64), generator=g, device="cuda").to(B.torch_dtype(dtype)) for r in (M, N, N))
        outs = [torch.empty_like(q) for _ in copies]
        for lib, out in zip(copies, outs):
            assert lib.ovggt_k_attention(p(q), p(k), p(v), M, N, H, dtype, p(out), p(scratch), p(status), stream) == 0
        assert torch.equal(outs[0], outs[1]) and torch.equal(outs[0], B.k_attention(q, k, v, H))
    a, w = (torch.randn((128, 128), generator=g, device="cuda").bfloat16() for _ in range(2))
    outs = [torch.empty_like(a) for _ in copies]
    for lib, out in zip(copies, outs):
        assert lib.ovggt_k_gemm_bf16(p(a), p(w), 128, 128, 128, p(out), p(status), stream) == 0
    assert torch.equal(outs[0], outs[1])
    assert int(status[0]) == 0
