"""Max-plus GEMM of general strides: every tile form on sizes around tile edges.

Each output is the maximum of single-rounded sums, which no order changes, so all forms
equal the plain torch result bit for bit.
"""
import pytest
import torch

from paper_2008_06888_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile", ["1 2", "1 8", "2 8", None])
@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (16, 17, 15), (63, 65, 16), (64, 64, 33), (65, 129, 17),
                                   (127, 128, 1), (129, 63, 48), (257, 191, 31)])
@pytest.mark.parametrize("ta,tb", [(0, 0), (1, 0), (0, 1), (1, 1)])
def test_tiles_equal_torch(tile, M, N, K, ta, tb, monkeypatch):
    if tile:
        monkeypatch.setenv("TN_GEMM_TILE", tile)
    g = torch.Generator(device="cuda").manual_seed(M * N + K)
    for dtype in (torch.float32, torch.int32):
        A = torch.randint(-99, 100, (3, K, M) if ta else (3, M, K), generator=g, device="cuda")
        Bm = torch.randint(-99, 100, (3, N, K) if tb else (3, K, N), generator=g, device="cuda")
        A, Bm = A.to(dtype), Bm.to(dtype)
        if dtype == torch.float32:
            A, Bm = A * 0.37, Bm * 0.73
        C = torch.empty((3, M, N), dtype=dtype, device="cuda")
        B.tn_maxplus_gemm(A, Bm, C, transA=bool(ta), transB=bool(tb),
                          stream_handle=torch.cuda.current_stream().cuda_stream)
        a = A.transpose(1, 2) if ta else A
        b = Bm.transpose(1, 2) if tb else Bm
        ref = (a[:, :, :, None] + b[:, None, :, :]).amax(2)
        assert torch.equal(C, ref)
