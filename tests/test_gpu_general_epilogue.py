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
