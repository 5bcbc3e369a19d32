"""The narrow tiles of the 16-byte max-plus GEMM (64, 32 and 16 columns): every output is
the max of single-rounding sums, so results are bit-identical to the definition; ragged
neighbours of the sizes take the other kernels."""
import numpy as np
import pytest

from oracle import semiring as S
from paper_2008_06888_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2008_06888_gb300 import build
    build.build()


@pytest.mark.parametrize("dtype", ["float32", "int32"])
@pytest.mark.parametrize("shape", [(1, 128, 16, 16), (3, 256, 16, 80), (2, 128, 32, 32),
                                   (1, 384, 96, 16), (2, 128, 64, 48), (1, 256, 192, 32),
                                   (5, 2048, 256, 16), (2, 128, 24, 16), (2, 128, 32, 20)])
@pytest.mark.parametrize("offset", [0, 1], ids=["aligned", "C off by one word"])
def test_narrow_tiles_match_definition(dtype, shape, offset):
    import torch
    bt, M, N, K = shape
    rng = np.random.default_rng(M + N + K)
    A = rng.standard_normal((bt, M, K)) * 20
    Bm = rng.standard_normal((bt, K, N)) * 20
    A, Bm = A.astype(dtype), Bm.astype(dtype)
    ref = np.stack([S.maxplus_matmul(A[i], Bm[i]) for i in range(bt)]).astype(dtype)
    Ad, Bd = torch.tensor(A, device="cuda"), torch.tensor(Bm, device="cuda")
    buf = torch.empty(bt * M * N + 4, dtype=Ad.dtype, device="cuda")
    Cd = buf[offset:offset + bt * M * N].view(bt, M, N)
    B.tn_maxplus_gemm(Ad, Bd, Cd)
    torch.cuda.synchronize()
    assert np.array_equal(Cd.cpu().numpy(), ref)
