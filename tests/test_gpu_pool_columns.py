"""The 3x3 / stride 1 max-pool, one or two output columns per thread by the number of threads, against the oracle: odd and even widths down to one column, strips
around their lengths, with and without padding, and nothing written past the output."""
import numpy as np
import pytest
import torch

from oracle import ref

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,H,W,C,pad", [(1, 1, 1, 16, 1), (2, 3, 2, 32, 1), (1, 3, 3, 16, 0), (3, 17, 5, 48, 1), (2, 16, 14, 64, 1), (1, 33, 27, 16, 1),
                                         (40, 9, 28, 112, 1), (1, 5, 4, 16, 0), (2, 4, 35, 16, 2),
                                         # enough threads for two columns each
                                         (700, 3, 3, 128, 1), (400, 5, 4, 256, 0), (60, 4, 35, 64, 2), (2, 9, 131, 512, 1), (20, 17, 5, 384, 1),
                                         (350, 33, 2, 32, 1), (1400, 4, 1, 64, 1), (48, 19, 23, 48, 1)])
def test_columns_per_thread_match_the_oracle(N, H, W, C, pad):
    from paper_1805_07941_b200 import binding
    x = np.random.default_rng(N + H + W).integers(-128, 128, (N, H, W, C), dtype=np.int8)
    want = ref.maxpool_i8(x, 3, 3, 1, pad)
    flat = torch.full((want.size + 64,), 77, dtype=torch.int8, device="cuda")
    y = flat[:want.size].view(want.shape)
    binding.qmaxpool_i8(torch.from_numpy(x).cuda(), 3, 3, 1, pad, out=y)
    assert (y.cpu().numpy() == want).all() and (flat[want.size:] == 77).all()
