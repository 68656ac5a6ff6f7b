"""Two-digit floating-point operands whose sums are recombined and converted in 32 bits, against the oracle: every output type's
conversion at the ties and beside them, shifts at the edge of the rule that takes the 32-bit form (and one below it, where the
64-bit form serves), the largest sums, and both forms on the same layer."""
import numpy as np
import pytest

from oracle import fpconv_ref
from paper_1805_07941_b200 import binding

pytestmark = pytest.mark.gpu


def run(w, bias, shift, x, fo, relu, R, hints=None):
    import torch
    N, H, W, C = x.shape
    with binding.plan_hints(**(hints or {})):
        conv = binding.QConvNP(w, bias, shift, N=N, H=H, W=W, C=C, K=w.shape[0], R=R, S=R, pad_h=R // 2, pad_w=R // 2, n_in=8, p_in=4, n_w=8,
                               p_w=4, n_out=fo[0], p_out=fo[1], relu=relu)
    y = torch.empty((N, conv.P, conv.Q, w.shape[0]), dtype=torch.uint8, device="cuda")
    conv.run(torch.from_numpy(x).cuda(), y)
    assert conv.status() == 0
    out, desc = y.cpu().numpy(), conv.describe()
    conv.destroy()
    return out, desc


@pytest.mark.parametrize("fo", [(8, 4), (8, 7), (8, 3), (6, 2), (5, 0), (4, 1), (2, 1)])
@pytest.mark.parametrize("C,R,K", [(16, 1, 40), (144, 3, 33), (64, 3, 128)])
def test_narrow_sums_match_the_oracle(fo, C, R, K):
    rng = np.random.default_rng(C + R + fo[1])
    x, w = (rng.integers(0, 256, s).astype(np.uint8) for s in ((2, 9, 8, C), (K, R, R, C)))
    for a in (x, w):
        a[(a & 0x7F) == 0] = 0
    x[0, 0, 0], w[0] = 0x7F, 0x7F                            # the largest values of both types
    w[1] = 0xFF
    largest = R * R * C * 1984**2
    bias = rng.integers(-2**20, 2**20, K).astype(np.int32)
    low = 7                                                  # the rule: |v| < 2^(22 + low) and low <= shift - 1
    while (largest + int(np.abs(bias.astype(np.int64)).max())) >> low >= (1 << 22) - 1:
        low += 1
    for least, narrow in ((low + 1, True), (low, False)):
        shift = (least + rng.integers(0, 9, K)).astype(np.int32)
        shift[0] = least
        # sums on the ties of the coarsest shift's grid and one beside them, by way of the bias
        acc = fpconv_ref.wide_value(x, w, bias, (8, 4), (8, 4), R=R, S=R, pad=(R // 2, R // 2))
        for k in range(2, K):
            v, half = int(acc[0, 3, 4, k]), 1 << (int(shift[k]) - 1)
            bias[k] += (half - v) % (2 * half) + (k % 3 - 1)
        for relu in (0, 1):
            want = fpconv_ref.qconv_np(x, w, bias, shift, (8, 4), (8, 4), fo, R=R, S=R, pad=(R // 2, R // 2), relu=relu)
            got, desc = run(w, bias, shift, x, fo, relu, R)
            assert ("sums=32" in desc) == narrow and (got == want).all(), desc
            if narrow:
                got, desc = run(w, bias, shift, x, fo, relu, R, dict(float_rounding=0))
                assert "sums=32" not in desc and (got == want).all(), desc


def test_what_the_narrow_sums_cannot_hold_keeps_the_wide_ones():
    rng = np.random.default_rng(0)
    x, w = (rng.integers(0, 128, s).astype(np.uint8) for s in ((1, 3, 3, 16), (16, 1, 1, 16)))
    for bias, narrow in ((2**30 - 1, True), (2**30, False), (-2**31 + 1, False)):
        b, shift = np.full(16, bias, np.int32), np.full(16, 24, np.int32)
        got, desc = run(w, b, shift, x, (8, 4), 0, 1)
        assert ("sums=32" in desc) == narrow
        assert (got == fpconv_ref.qconv_np(x, w, b, shift, (8, 4), (8, 4), (8, 4), R=1, S=1)).all()
