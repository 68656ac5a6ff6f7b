"""The general int8 epilogue in both arithmetics (float rounding where the weights bound the sum, integers elsewhere) against
the oracle: every rounding mode with and without ReLU and residual, shifts of 0, narrow output types, rows that start at any
address (whole units, heads and tails of 1 to 7 bytes, rows shorter than two units)."""
import numpy as np
import pytest

from tests.helpers import gpu_conv, oracle_conv, rand_layer

pytestmark = pytest.mark.gpu

SHAPES = [  # N, H, W, C, K, filter, offset, pitch
    (2, 9, 7, 32, 77, 1, 0, 0), (1, 13, 11, 48, 130, 3, 0, 0), (3, 5, 30, 16, 21, 1, 3, 29), (1, 12, 12, 64, 12, 3, 1, 15),
    (2, 20, 9, 16, 208, 1, 0, 0), (1, 33, 5, 32, 68, 1, 4, 76), (1, 6, 6, 256, 131, 3, 0, 0), (40, 14, 14, 32, 150, 1, 0, 0)]


@pytest.mark.parametrize("rounding", [0, 1, 2, 3])
@pytest.mark.parametrize("shape", SHAPES)
def test_every_rounding_mode(shape, rounding):
    N, H, W, C, K, R, off, pitch = shape
    rng = np.random.default_rng(sum(shape) + rounding)
    for small in (0, 1):
        x, w, bias, shift, res, t = rand_layer(rng, N, H, W, C, K, R, R, with_res=True, pad=(R // 2, R // 2))
        t = np.minimum(t, 5).astype(np.int32)
        if small:                                            # the float-rounding form
            w, bias, shift = (w // 16).astype(np.int8), bias // 8, np.maximum(shift - 4, 0).astype(np.int32)
        for relu in (0, 1):
            for n_out in (8, 5):
                kw = dict(R=R, S=R, pad=(R // 2, R // 2), relu=relu, rounding=rounding, n_out=n_out, out_c_offset=off, out_c_pitch=pitch)
                for r, tt in ((None, None), (res, t)):
                    got, desc = gpu_conv(x, w, bias, shift, r, tt, **kw)
                    assert (got == oracle_conv(x, w, bias, shift, r, tt, **kw)).all(), (desc, small, relu, n_out, r is None)


@pytest.mark.parametrize("rounding", [0, 1, 2, 3])
def test_shifts_of_zero_and_ties(rounding):
    rng = np.random.default_rng(rounding)
    x = rng.integers(-3, 4, size=(1, 16, 16, 16), dtype=np.int8)
    w = rng.integers(-2, 3, size=(40, 1, 1, 16), dtype=np.int8)
    bias = rng.integers(-9, 10, size=40, dtype=np.int32)
    shift = np.resize(np.array([0, 1, 2, 3, 5], np.int32), 40)
    for sh in (shift, np.maximum(shift, 1)):
        for relu in (0, 1):
            kw = dict(R=1, S=1, relu=relu, rounding=rounding)
            got, desc = gpu_conv(x, w, bias, sh, **kw)
            assert (got == oracle_conv(x, w, bias, sh, **kw)).all(), (desc, relu)
