"""Products with few tiles and a long inner dimension, which several thread blocks share."""
import numpy as np
import pytest
import torch

from oracle import mrem_oracle as O
from paper_2109_15082_b200 import binding as B

pytestmark = pytest.mark.gpu
DEV = "cuda"


# one row, full and just beyond a tile; one, two and three 32-column chunks, many tiles; the fewest 128-byte deep blocks that
# are shared (8), an odd number of them with a ragged last one, and many
@pytest.mark.parametrize("M", [1, 128, 129, 216])
@pytest.mark.parametrize("N", [32, 96, 768])
@pytest.mark.parametrize("blocks,ragged", [(8, 0), (11, 3), (33, 1), (48, 0)])
def test_shared_products_are_exact(M, N, blocks, ragged):
    """Whole numbers small enough that every partial sum is exact (|sum| <= 3072 * 16 < 2^24): equal in any order, bit for bit."""
    rng = np.random.default_rng(M + N + blocks)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    stream = torch.cuda.current_stream().cuda_stream
    K = 64 * blocks - 16 * ragged
    a, b = rng.integers(-4, 5, (M, K)), rng.integers(-4, 5, (N, K))
    ref = O.int_matmul(a, b)
    for a_mn, b_mn in ((0, 0), (0, 1), (1, 1)):
        if a_mn and M % 8:
            continue                                       # the strides of an operand are multiples of 16 bytes
        ad = torch.from_numpy(np.ascontiguousarray(a.T if a_mn else a)).to(DEV).to(torch.bfloat16)
        bd = torch.from_numpy(np.ascontiguousarray(b.T if b_mn else b)).to(DEV).to(torch.bfloat16)
        out = torch.full((M, N), 0.5, device=DEV)
        B.mrem_gemm(B.BF16, ad, a_mn, M if a_mn else K, 0, bd, b_mn, N if b_mn else K, 0, M, N, K, 1, 1.0, out, N, 0, 0, status, stream)
        assert np.array_equal(out.cpu().numpy().astype(np.int64), ref), (a_mn, b_mn)
    K *= 2
    a, b = rng.integers(-127, 128, (M, K)), rng.integers(-127, 128, (N, K))
    acc = torch.full((M, N), -1, dtype=torch.int32, device=DEV)
    B.mrem_gemm_i8(torch.from_numpy(a.astype(np.int8)).to(DEV), 0, torch.from_numpy(b.astype(np.int8)).to(DEV), M, N, K, acc, 0, status, stream)
    assert np.array_equal(acc.cpu().numpy().astype(np.int64), O.int_matmul(a, b))
    assert int(status[0]) == 0
