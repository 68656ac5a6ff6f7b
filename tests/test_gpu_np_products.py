"""The digit products of the floating-point layers against the oracle at the sizes where their plan changes: one to six
products (operands of one to three digits, mixed), one and two accumulator buffers, channel counts below / at / above a
ring-stage chunk, partial batches, output rows at every alignment, and every input pattern of a type."""
import numpy as np
import pytest

from oracle import fpconv_ref
from paper_1805_07941_b200 import binding

pytestmark = pytest.mark.gpu

FMT = {1: (8, 7), 2: (8, 4), 3: (8, 3)}                    # types whose betas have that many base-128 digits
PRODUCTS = {(1, 1): 1, (1, 2): 2, (2, 1): 2, (1, 3): 3, (3, 1): 3, (2, 2): 3, (2, 3): 5, (3, 2): 5, (3, 3): 6}
CASES = [  # N, n_run, H, W, C, K, R, stride
    (2, 2, 9, 7, 16, 17, 3, 1), (3, 2, 6, 5, 48, 80, 1, 1), (1, 1, 14, 14, 128, 100, 3, 1), (2, 2, 13, 11, 144, 33, 3, 2),
    (9, 9, 8, 8, 64, 256, 1, 2)]


@pytest.mark.parametrize("digits", sorted(PRODUCTS))
@pytest.mark.parametrize("case", CASES)
def test_products_match_the_oracle(digits, case):
    import torch
    N, n_run, H, W, C, K, R, stride = case
    fi, fw, fo = FMT[digits[0]], FMT[digits[1]], FMT[2 if digits[0] != 2 else 3]
    rng = np.random.default_rng(sum(case) + 10 * digits[0] + digits[1])
    x = rng.integers(0, 256, (N, H, W, C)).astype(np.uint8)           # every pattern, the largest magnitudes included
    x.reshape(-1)[:256] = np.arange(256, dtype=np.uint8)
    x[(x & 0x7F) == 0] = 0                                            # (patterns have no negative zero)
    w = rng.integers(0, 256, (K, R, R, C)).astype(np.uint8)
    w[(w & 0x7F) == 0] = 0
    bias = rng.integers(-2**31 + 1, 2**31 - 1, K).astype(np.int32)
    pad, st = (R // 2, R // 2), (stride, stride)
    acc = fpconv_ref.wide_value(x[:1], w, bias, fi, fw, R=R, S=R, stride=st, pad=pad)
    base = np.log2(max(1.0, float(np.abs(acc).mean()) * 3 / fpconv_ref.magnitudes(*fo)[-1]))
    shift = (int(base) + rng.integers(-2, 3, K)).clip(0, 40).astype(np.int32)
    for relu in (0, 1):
        want = fpconv_ref.qconv_np(x[:n_run], w, bias, shift, fi, fw, fo, R=R, S=R, stride=st, pad=pad, relu=relu)
        conv = binding.QConvNP(w, bias, shift, N=N, H=H, W=W, C=C, K=K, R=R, S=R, stride_h=stride, stride_w=stride, pad_h=R // 2,
                               pad_w=R // 2, n_in=fi[0], p_in=fi[1], n_w=fw[0], p_w=fw[1], n_out=fo[0], p_out=fo[1], relu=relu)
        assert "products=%d " % PRODUCTS[digits] in conv.describe()
        flat = torch.full((N * conv.P * conv.Q * K + 1,), 0x55, dtype=torch.uint8, device="cuda")
        for offset in (0, 1):                                         # aligned rows, and rows one byte off
            y = flat[offset:offset + N * conv.P * conv.Q * K].view(N, conv.P, conv.Q, K)
            y.fill_(0x55)
            conv.run(torch.from_numpy(x[:n_run]).cuda(), y)
            assert conv.status() == 0
            got = y.cpu().numpy()
            assert (got[:n_run] == want).all() and (got[n_run:] == 0x55).all(), conv.describe()
        conv.destroy()


@pytest.mark.parametrize("digits", [(2, 3), (3, 3), (2, 2)])
@pytest.mark.parametrize("case", [(1, 1, 80, 80, 16, 512, 1, 1), (2, 2, 45, 43, 16, 1000, 1, 1), (1, 1, 131, 129, 16, 520, 1, 2)])
def test_constants_of_many_channels_tile_by_tile(digits, case):
    """More channels than shared memory holds constants for (512 of 16 bytes, padding included): every tile stages its own, and
    a CTA walks several tiles of different channels, with one accumulator buffer (five and six products) and with two.  Shifts
    and biases differ from channel to channel, so that a tile on another tile's constants is wrong."""
    import torch
    N, n_run, H, W, C, K, R, stride = case
    fi, fw, fo = FMT[digits[0]], FMT[digits[1]], FMT[2]
    rng = np.random.default_rng(sum(case) + 10 * digits[0] + digits[1])
    x, w = (rng.integers(0, 256, s).astype(np.uint8) for s in ((N, H, W, C), (K, R, R, C)))
    for a in (x, w):
        a[(a & 0x7F) == 0] = 0
    bias = rng.integers(-2**31 + 1, 2**31 - 1, K).astype(np.int32)
    acc = fpconv_ref.wide_value(x[:1, :16], w, bias, fi, fw, R=R, S=R, stride=(stride, stride), pad=(0, 0))
    base = np.log2(max(1.0, float(np.abs(acc).mean()) * 3 / fpconv_ref.magnitudes(*fo)[-1]))
    shift = (int(base) + rng.integers(-3, 4, K)).clip(0, 40).astype(np.int32)
    want = fpconv_ref.qconv_np(x, w, bias, shift, fi, fw, fo, R=R, S=R, stride=(stride, stride), pad=(0, 0))
    conv = binding.QConvNP(w, bias, shift, N=N, H=H, W=W, C=C, K=K, R=R, S=R, stride_h=stride, stride_w=stride, n_in=fi[0],
                           p_in=fi[1], n_w=fw[0], p_w=fw[1], n_out=fo[0], p_out=fo[1])
    plan = dict(f.split("=") for f in conv.describe().split() if f.count("=") == 1)
    m_tiles = -(-N * conv.P * conv.Q // 128)
    assert int(plan["BN"]) * int(plan["tiles_k"]) > 512 and m_tiles * int(plan["tiles_k"]) > 148, plan
    xd = torch.from_numpy(x).cuda()
    for _ in range(3):
        y = torch.full((N, conv.P, conv.Q, K), 0x55, dtype=torch.uint8, device="cuda")
        conv.run(xd, y)
        assert conv.status() == 0 and (y.cpu().numpy() == want).all(), conv.describe()
    conv.destroy()


def test_first_run_on_another_stream_finds_the_padding_cleared():
    """48 channels are padded to 64 in the digit planes (0.8 GB here), which creation clears; a run right behind it on a stream
    that does not wait for the default one must not have its planes cleared under it."""
    import torch
    N, H, W, C, K = 256, 128, 128, 48, 16
    rng = np.random.default_rng(1)
    w = rng.integers(1, 127, (K, 1, 1, C)).astype(np.uint8)
    shift = np.full(K, 14, np.int32)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(2)
    x = torch.randint(1, 127, (N, H, W, C), generator=gen, device="cuda", dtype=torch.uint8)
    y = torch.empty((N, H, W, K), dtype=torch.uint8, device="cuda")
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        conv = binding.QConvNP(w, None, shift, N=N, H=H, W=W, C=C, K=K, R=1, S=1, n_in=8, p_in=4, n_w=8, p_w=4, n_out=8, p_out=4)
        conv.run(x, y)
    assert conv.status() == 0
    first = y.clone()
    conv.run(x, y)
    assert conv.status() == 0 and torch.equal(first, y)
    for n in (0, N // 2, N - 1):
        want = fpconv_ref.qconv_np(x[n:n + 1].cpu().numpy(), w, None, shift, (8, 4), (8, 4), (8, 4), R=1, S=1)
        assert (first[n:n + 1].cpu().numpy() == want).all()
    conv.destroy()
