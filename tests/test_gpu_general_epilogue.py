"""The tensor-core kernel's general epilogue (any rounding mode, width, alignment; int32 / float output) against the
oracle, bit for bit, at every alignment of its row copies: K and the output window's pitch and offset decide how many
bytes a lane moves, K's remainder which columns a warp owns, the pixel count which rows of the last tile exist."""
import numpy as np
import pytest

from tests.helpers import gpu_conv, oracle_conv, rand_layer

pytestmark = pytest.mark.gpu

# K, out_c_offset, out_c_pitch (0: K): output pieces aligned to 1, 2, 4, 8 and 16 bytes; one and several channel tiles
WINDOWS = [(1, 0, 0), (7, 3, 21), (17, 0, 0), (18, 2, 22), (20, 4, 28), (24, 8, 40), (48, 16, 80), (63, 0, 64), (64, 0, 0),
           (129, 0, 0), (200, 0, 0), (250, 6, 262), (256, 16, 288)]


@pytest.mark.parametrize("K,off,pitch", WINDOWS)
@pytest.mark.parametrize("with_res", [0, 1])
def test_rows_at_every_alignment(K, off, pitch, with_res):
    rng = np.random.default_rng(100 * K + off + with_res)
    for i, (N, H, W, C, R, pad) in enumerate([(2, 9, 7, 32, 3, (1, 1)), (1, 11, 12, 16, 1, (0, 0))]):
        x, w, bias, shift, res, t = rand_layer(rng, N, H, W, C, K, R, R, with_res=bool(with_res), pad=pad)
        for rounding in (1, 2, 3, 0):
            kw = dict(R=R, S=R, pad=pad, relu=(rounding + i) & 1, rounding=rounding, n_out=8 if rounding else 7,
                      out_c_offset=off, out_c_pitch=pitch, symmetric=rounding & 1)
            got, desc = gpu_conv(x, w, bias, shift, res, t, **kw)
            want = oracle_conv(x, w, bias, shift, res, t, **kw)
            assert "fast=0" in desc and (got == want).all(), (desc, rounding)
        for out_mode in (1, 2):
            acc_exp = rng.integers(-20, -8, K).astype(np.int32)
            kw = dict(R=R, S=R, pad=pad, relu=i, out_mode=out_mode, out_c_offset=off, out_c_pitch=pitch)
            got, desc = gpu_conv(x, w, bias, None, res, t, acc_exp, **kw)
            want = oracle_conv(x, w, bias, None, res, t, acc_exp, **kw)
            assert (got == want).all(), (desc, out_mode)


@pytest.mark.parametrize("rounding", [0, 1, 2, 3])
@pytest.mark.parametrize("shift", [0, 1, 30, 31])
def test_shifts_at_the_ends_of_their_range(rounding, shift):
    """s = 0 leaves the value, s = 31 leaves no room for the single-pass rounding: the exact two-step form."""
    rng = np.random.default_rng(shift)
    x, w, bias, _, _, _ = rand_layer(rng, 1, 6, 5, 16, 24, 1, 1)
    bias = rng.integers(-2**30, 2**30, 24).astype(np.int32)
    bias[:4] = [-2**30, 2**30, 0, -1]
    s = np.full(24, shift, np.int32)
    kw = dict(R=1, S=1, rounding=rounding, n_out=5)
    got, desc = gpu_conv(x, w, bias, s, **kw)
    assert (got == oracle_conv(x, w, bias, s, **kw)).all(), desc


MAX_CASES = [  # N, H, W, C, K, R, groups, stride, n_run: every kernel that can run a float-out layer
    (3, 9, 7, 32, 40, 3, 1, 1, 3), (3, 9, 7, 32, 40, 3, 1, 1, 2), (2, 14, 14, 64, 64, 3, 1, 1, 2), (5, 6, 5, 16, 17, 1, 1, 1, 5),
    (2, 17, 15, 3, 24, 3, 1, 2, 2), (2, 12, 12, 32, 32, 3, 32, 1, 2), (2, 13, 11, 24, 24, 3, 24, 2, 1), (2, 8, 8, 20, 12, 3, 2, 1, 2)]


@pytest.mark.parametrize("case", MAX_CASES)
@pytest.mark.parametrize("with_res", [0, 1])
def test_maximum_of_the_float_output_without_the_output(case, with_res):
    import torch
    from oracle import ref
    from paper_1805_07941_b200 import binding
    N, H, W, C, K, R, groups, stride, n_run = case
    rng = np.random.default_rng(sum(case))
    x, w, bias, _, res, t = rand_layer(rng, N, H, W, C, K, R, R, groups=groups, with_res=bool(with_res), stride=(stride, stride),
                                       pad=(R // 2, R // 2))
    acc_exp = rng.integers(-20, -8, K).astype(np.int32)
    for relu in (0, 1):
        want = ref.qconv(x, w, bias, None, res, t, acc_exp, R=R, S=R, stride=(stride, stride), pad=(R // 2, R // 2), groups=groups,
                         relu=relu, out_mode=2)
        conv = binding.QConv(w, bias, None, t, acc_exp, N=N, H=H, W=W, C=C, K=K, R=R, S=R, stride_h=stride, stride_w=stride,
                             pad_h=R // 2, pad_w=R // 2, groups=groups, relu=relu, out_mode=2, has_residual=with_res)
        rd = torch.from_numpy(res).cuda() if with_res else None
        for _ in range(2):                                 # the word is cleared by every call
            assert conv.run_maxabs(torch.from_numpy(x).cuda(), rd, n_run=n_run) == np.abs(want[:n_run]).max(), conv.describe()
        conv.destroy()
    with pytest.raises(binding.QconvError):
        binding.QConv(w, bias, None, t, None, N=N, H=H, W=W, C=C, K=K, R=R, S=R, stride_h=stride, stride_w=stride, pad_h=R // 2,
                      pad_w=R // 2, groups=groups, has_residual=with_res).run_maxabs(torch.from_numpy(x).cuda(), rd)
