"""The depthwise layers on warp-level matrix instructions against the oracle: image widths around the groups of 8 pixels and the
16 of a warp, channel counts around its 32 and the staged 32 / 64 / 128, images that share a CTA, strips around the rows in
flight, both strides, windows of a wider tensor, partial batches, unpadded layers, little-aligned outputs, and a wait that
expires."""
import time

import numpy as np
import pytest
import torch

from tests.helpers import gpu_conv, oracle_conv, rand_layer

pytestmark = pytest.mark.gpu

CASES = [  # N, H, W, C, stride, pad
    (1, 1, 1, 16, 1, 1), (3, 2, 7, 32, 1, 1), (2, 3, 8, 48, 1, 1), (5, 4, 9, 64, 1, 1), (2, 5, 15, 80, 1, 1), (2, 6, 16, 96, 1, 1), (1, 7, 17, 128, 1, 1),
    (9, 7, 7, 160, 1, 1), (2, 40, 33, 32, 1, 1), (1, 9, 129, 32, 1, 1), (1, 5, 255, 16, 1, 1), (2, 11, 63, 64, 1, 1), (1, 64, 20, 1008, 1, 1),
    (1, 1, 1, 16, 2, 1), (3, 2, 7, 32, 2, 1), (5, 9, 17, 64, 2, 1), (2, 14, 33, 96, 2, 1), (1, 31, 130, 32, 2, 1), (1, 6, 257, 16, 2, 1), (9, 14, 14, 144, 2, 1),
    (2, 9, 12, 64, 1, 0), (2, 9, 12, 64, 2, 0), (2, 9, 12, 32, 1, 2), (300, 5, 6, 32, 1, 1)]


@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("uniform", [0, 1])
def test_depthwise_on_warp_instructions_matches_the_oracle(case, uniform):
    from paper_1805_07941_b200 import binding
    N, H, W, C, st, pad = case
    rng = np.random.default_rng(sum(case))
    x, w, bias, shift, _, _ = rand_layer(rng, N, H, W, C, C, 3, 3, groups=C, stride=(st, st), pad=(pad, pad), per_channel_shift=not uniform)
    shift = (shift - 1).clip(4, 31)
    for relu in (0, 1):
        kw = dict(R=3, S=3, stride=(st, st), pad=(pad, pad), groups=C, relu=relu, symmetric=uniform)
        win = dict(kw, out_c_offset=8, out_c_pitch=C + 24)
        got, desc = gpu_conv(x, w, bias, shift, **kw)
        assert "depthwise3x3/mma+tma" in desc and (got == oracle_conv(x, w, bias, shift, **kw)).all(), desc
        got, desc = gpu_conv(x, w, bias, shift, **win)
        assert "depthwise3x3/mma+tma" in desc and (got == oracle_conv(x, w, bias, shift, **win)).all(), desc
    # a partial batch, then the whole one, and an output that is 8-byte aligned only
    want = oracle_conv(x, w, bias, shift, R=3, S=3, stride=(st, st), pad=(pad, pad), groups=C)
    conv = binding.QConv(w, bias, shift, N=N, H=H, W=W, C=C, K=C, R=3, S=3, stride_h=st, stride_w=st, pad_h=pad, pad_w=pad, groups=C)
    xd = torch.from_numpy(x).cuda()
    for n, off in ((max(1, N - 1), 0), (N, 8), (N, 4)):      # (4: the dp4a kernels)
        flat = torch.full((N * conv.P * conv.Q * C + 64,), 77, dtype=torch.int8, device="cuda")
        y = flat[off:off + N * conv.P * conv.Q * C].view(N, conv.P, conv.Q, C)
        conv.run(xd, y, n_run=n)
        assert conv.status() == 0
        got = y.cpu().numpy()
        assert (got[:n] == want[:n]).all() and (got[n:] == 77).all() and (flat[:off] == 77).all() and (flat[off + got.size:] == 77).all()
    conv.destroy()


@pytest.mark.parametrize("C,stride", [(64, 1), (16, 1), (112, 1), (240, 2), (1008, 1)])
def test_an_expired_wait_is_reported_and_the_next_run_is_right(C, stride):
    """No polls granted: every warp leaves, the copies in flight land, the status says so.  (Also where 32 does not divide the
    channels and no other kernel for the layer has waits.)"""
    from paper_1805_07941_b200 import binding
    rng = np.random.default_rng(1)
    x, w, bias, shift, _, _ = rand_layer(rng, 2, 40, 30, C, C, 3, 3, groups=C, stride=(stride, stride), pad=(1, 1))
    shift = (shift - 1).clip(4, 31)
    conv = binding.QConv(w, bias, shift, N=2, H=40, W=30, C=C, K=C, R=3, S=3, stride_h=stride, stride_w=stride, pad_h=1, pad_w=1, groups=C)
    assert "depthwise3x3/mma+tma" in conv.describe()
    xd, y = torch.from_numpy(x).cuda(), torch.empty((2, conv.P, conv.Q, C), dtype=torch.int8, device="cuda")
    want = oracle_conv(x, w, bias, shift, R=3, S=3, stride=(stride, stride), pad=(1, 1), groups=C)
    for _ in range(2):
        conv.set_wait_limit(0)
        conv.run(xd, y)
        assert conv.status() == binding.ERR_TIMEOUT
        conv.set_wait_limit(1 << 22)
        conv.run(xd, y)
        assert conv.status() == 0 and (y.cpu().numpy() == want).all()


def test_a_tall_layers_call_costs_the_host_no_more_than_a_short_ones():
    """How a batch is cut into strips is found once, not on every call; each batch size has its own cut."""
    from paper_1805_07941_b200 import binding
    rng = np.random.default_rng(2)
    per_call = {}
    for H in (64, 32768):
        x, w, bias, shift, _, _ = rand_layer(rng, 3, H, 1, 16, 16, 3, 3, groups=16, pad=(1, 1))
        shift = (shift - 1).clip(4, 31)
        conv = binding.QConv(w, bias, shift, N=3, H=H, W=1, C=16, K=16, R=3, S=3, pad_h=1, pad_w=1, groups=16)
        xd = torch.from_numpy(x).cuda()
        want = oracle_conv(x, w, bias, shift, R=3, S=3, pad=(1, 1), groups=16)
        for n in (1, 3, 2, 3):
            y = torch.full((3, H, 1, 16), 77, dtype=torch.int8, device="cuda")
            conv.run(xd, y, n_run=n)
            assert conv.status() == 0
            got = y.cpu().numpy()
            assert (got[:n] == want[:n]).all() and (got[n:] == 77).all()
        trials = []
        for _ in range(5):
            start = time.perf_counter()
            for _ in range(200):                             # (queued behind one another: the host's time alone)
                conv.run(xd, y)
            trials.append((time.perf_counter() - start) / 200)
            torch.cuda.synchronize()
        per_call[H] = min(trials)
    # the search took about 50 us at this height
    assert per_call[32768] < 2 * per_call[64] + 20e-6, per_call
