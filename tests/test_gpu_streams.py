"""The streaming kernels (conversions, codec, statistics) against the oracle at the counts where their loops change:
below one vector, around one pass of the unrolled loop over the whole grid, and on misaligned tensors."""
import numpy as np
import pytest

from oracle import dynfloat, ref
from paper_1805_07941_b200 import binding

pytestmark = pytest.mark.gpu

LAP = 148 * 6 * 256 * 4                                    # values one grid takes per load
COUNTS = [1, 3, 4, 5, 255, 1023, 4 * 1024 + 1, LAP - 1, 4 * LAP, 4 * LAP + 4 * 1024 + 3]


def _values(n, seed):
    rng = np.random.default_rng(seed)
    x = (rng.standard_normal(n) * 3).astype(np.float32)
    x[:: max(1, n // 7)] = np.resize(np.array([np.nan, np.inf, -np.inf, 0.0, -0.0, 1e-40, -3e38], np.float32), x[:: max(1, n // 7)].shape)
    return x


@pytest.mark.parametrize("count", COUNTS)
@pytest.mark.parametrize("floats", [0, 1])
def test_conversions_and_statistics_at_loop_boundaries(count, floats):
    import torch
    x = _values(count, count)
    buf = torch.zeros(count + 4, dtype=torch.float32, device="cuda")
    xd = buf[floats:floats + count]
    xd.copy_(torch.from_numpy(x))
    assert (binding.qquantize_f32(xd, -4).cpu().numpy() == ref.quantize_f32(x, -4)).all()
    for nbins, hi in ((2048, 0.0), (7, 2.5)):
        got, want = binding.qcalib_collect(xd, nbins, hi), ref.calib_stats(x, nbins, hi)
        assert got["maxabs"] == want["maxabs"] and (got["hist"] == want["hist"]).all()
        assert (got["count"], got["nonfinite"]) == (want["count"], want["nonfinite"])
        # fp64 sums of float32 values in another order: at most count * 2^-53 relative to the sum of magnitudes
        mags = float(np.abs(x[np.isfinite(x)].astype(np.float64)).sum())
        assert abs(got["sum"] - want["sum"]) <= 2 * count * 2.0**-53 * mags
        assert abs(got["sumsq"] - want["sumsq"]) <= 2 * count * 2.0**-53 * want["sumsq"]
    part = x[: min(count, 3000)] if count > 3000 else x      # (the codec's oracle works value by value)
    tail = x[-1500:]
    for n, p in ((8, 4), (8, 0), (8, 7), (5, 2)):
        codes = binding.qquantize_f32_np(xd, -6, n, p)
        back = binding.qdequantize_np(codes, -6, n, p).cpu().numpy()
        codes = codes.cpu().numpy()
        for got, src in ((codes[: part.size], part), (codes[-tail.size:], tail)):
            assert (got == dynfloat.quantize_np(src, -6, n, p)).all(), (n, p)
        lut = dynfloat.dequantize_np(np.arange(1 << n, dtype=np.uint8), -6, n, p)
        assert (back.view(np.uint32) == np.asarray(lut, np.float32)[codes].view(np.uint32)).all(), (n, p)


@pytest.mark.parametrize("e", [-126, -40, 0, 40, 126])
def test_codec_over_the_exponent_range(e):
    """Scales at the ends of their range, values around the smallest and largest representable ones and their midpoints."""
    import torch
    for n, p in ((8, 4), (8, 3), (8, 1), (8, 0), (8, 7), (4, 1)):
        lut = np.asarray(dynfloat.dequantize_np(np.arange(1 << (n - 1), dtype=np.uint8), e, n, p), np.float32)
        lut = lut[np.isfinite(lut)].astype(np.float64)
        with np.errstate(over="ignore", under="ignore"):
            mid = ((lut[1:] + lut[:-1]) / 2).astype(np.float32)
            pts = np.concatenate([lut.astype(np.float32), mid, np.nextafter(mid, np.float32(0)), np.nextafter(mid, np.float32(np.inf))])
        pts = pts[np.isfinite(pts)]
        x = np.concatenate([pts, -pts]).astype(np.float32)
        codes = binding.qquantize_f32_np(torch.from_numpy(x).cuda(), e, n, p)
        assert (codes.cpu().numpy() == dynfloat.quantize_np(x, e, n, p)).all(), (n, p)
        want = np.asarray(dynfloat.dequantize_np(codes.cpu().numpy(), e, n, p), np.float32)
        assert (binding.qdequantize_np(codes, e, n, p).cpu().numpy().view(np.uint32) == want.view(np.uint32)).all(), (n, p)
